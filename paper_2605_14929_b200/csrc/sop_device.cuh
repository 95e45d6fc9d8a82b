// Device-side building blocks of libsop (sm_100a).  Everything here is compiled with -fmad=false:
// a fused multiply-add happens only where __fmaf_rn / __ffma2_rn is written, so every fp32 result
// is one IEEE-754 operation rounded to nearest even and reproducible bit for bit.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/sop.h"

#define SOP_MAX_TABLES 8      // distinct LUT contents per call
#define SOP_MAX_CLASSES 8     // distinct (scope, tmax, quantiser) groups per call
#define SOP_HIST_BINS 320     // exponent histogram: ilogb(sigma) + 160, ilogb in [-149, 128]
#define SOP_HIST_OFF 160

namespace sop {

// ---- host-side error plumbing --------------------------------------------------------------
void set_cuda_error(cudaError_t e, const char* where);
#define SOP_CUDA_TRY(expr)                                 \
  do {                                                     \
    cudaError_t e__ = (expr);                              \
    if (e__ != cudaSuccess) {                              \
      ::sop::set_cuda_error(e__, #expr);                   \
      return SOP_ERR_CUDA;                                 \
    }                                                      \
  } while (0)

// What the library remembers about a device, per device ordinal (a process may drive several devices; a call works
// on the device that is current when it is made).  device_facts() returns the entry of the current device, or a
// scratch entry that is never marked as known when the ordinal is beyond the table.
struct DeviceFacts {
  int sms;                    // 0: not asked yet
  int coop_blocks_per_sm;     // resident CTAs of the persistent Lloyd kernel per SM; -1: not asked yet, 0: no cooperative launch
  bool search_attr_set;       // the dynamic shared-memory limits of the search kernels have been raised on this device
  bool lloyd_attr_set;        // the same for the pool cache kernels
};
DeviceFacts* device_facts();
int num_sms();

// Optional timing of one kernel family of a call (CUDA events on the launching stream): edge 0 before
// the first launch, edge 1 after the last.  No-op unless profiling is enabled.
int profile_mark(int which, int edge, cudaStream_t st);

// ---- launches ------------------------------------------------------------------------------
// Every kernel of the library but one is launched so that it may start while the one before it on the stream still runs (programmatic
// dependent launch); the Lloyd iterations, whose CTAs wait for one another, are launched cooperatively instead and start in their turn.  A pass is a chain of twenty short kernels, and the time from the end of one to the start of the next was a
// sixth of a small layer's pass.  Rules that each kernel keeps: pdl_trigger() first (its successor may then be scheduled as its CTAs
// leave), and pdl_wait() -- which returns when the kernels before it have completed and their writes are visible -- before the
// first access to global memory; only what depends on the parameters alone comes before the wait.  Global memory is read by plain
// loads: __ldg and const __restrict__ promise data that does not change while the kernel lives, and a kernel that starts before its
// predecessor ends lives while that one still writes what it will read.
template <typename... P, typename... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
// Zeros: a kernel of the chain instead of a memset, which would neither start early nor let its successor.
cudaError_t clear(void* words, size_t bytes, cudaStream_t st);      // whole 32-bit words

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- kernel parameter blocks ---------------------------------------------------------------
struct FmtDev {
  int y;                // mantissa bits
  int bias;
  int emin, emax;       // unbiased exponent range of normal values
  int code_max;         // largest finite magnitude code (E << y | M)
  int sign_bits;
};

struct AtomsDev {
  int n_atoms;
  unsigned dd_mask;         // atoms whose table comes from dd_lut at kernel time
  const float* dd_lut;      // device, SOP_MAX_ENTRIES floats (may be null)
  sop_atom atoms[SOP_MAX_ATOMS];
};

int validate_fmt(const sop_scale_fmt* f, FmtDev* out);
int validate_atoms(const sop_atom* atoms, int n_atoms, unsigned dd_mask, const float* dd_lut, AtomsDev* out);
int validate_layer(const void* W, long long M, long long K, long long ldw, const float* c, int g);

// ---- small device helpers ------------------------------------------------------------------
__device__ __forceinline__ float pow2f_int(int e) {  // 2^e for e in [-126, 127]
  return __uint_as_float((uint32_t)(e + 127) << 23);
}

__device__ __forceinline__ int ilogb_pos(float v) {  // floor(log2 v) for finite v > 0, subnormals included
  const uint32_t b = __float_as_uint(v);
  const int e = (int)(b >> 23);
  if (e != 0) return e - 127;
  return (31 - __clz((int)(b & 0x7FFFFFu))) - 149;
}

__device__ __forceinline__ float bf16lo(uint32_t packed) { return __uint_as_float(packed << 16); }
__device__ __forceinline__ float bf16hi(uint32_t packed) { return __uint_as_float(packed & 0xFFFF0000u); }

// value = mant * 2^ex rounded once (only when the result is below the fp32 normal range)
__device__ __forceinline__ float ldexp_once(uint32_t mant, int ex) {
  const int e1 = max(-100, min(100, ex));
  const int e2 = max(-120, min(120, ex - e1));
  return __fmul_rn(__fmul_rn((float)mant, pow2f_int(e1)), pow2f_int(e2));
}

struct QScale { float s_hat; uint32_t code; };  // code = (E << y) | M

// Scale quantisation: sigma * 2^k rounded to nearest even on a y-bit mantissa with gradual
// underflow at E = 0, saturating at code_max, never rounding a positive value to zero; decoded and
// multiplied back by 2^-k.  Pure integer work on the fp32 bit pattern.
__device__ __forceinline__ QScale scale_quantize(float sigma, int k, const FmtDev& f) {
  QScale r;
  r.s_hat = 0.0f;
  r.code = 0;
  if (!(sigma > 0.0f)) return r;
  const uint32_t b = __float_as_uint(sigma);
  int e = (int)(b >> 23);
  {
    // The usual case: the shifted value lies in the format's normal range below its top binade (so that a
    // carry out of the mantissa cannot pass the largest code) and the format keeps at least one mantissa
    // bit.  Rounding to nearest even on y bits is then one integer addition on the fp32 pattern; the shift
    // k moves only the exponent, so the decoded scale is the rounded value itself.
    const int ev0 = e - 127 + k;
    if (e != 0 && f.y >= 1 && ev0 >= f.emin && ev0 < f.emax) {
      const int sh0 = 23 - f.y;
      const uint32_t rb = (b + ((1u << (sh0 - 1)) - 1u) + ((b >> sh0) & 1u)) & ~((1u << sh0) - 1u);
      r.s_hat = __uint_as_float(rb);
      r.code = (uint32_t)(((int)(rb >> 23) - 127 + k + f.bias) << f.y) | ((rb >> sh0) & ((1u << f.y) - 1u));
      return r;
    }
  }
  uint32_t m = b & 0x7FFFFFu;
  if (e == 0) {
    const int sh = __clz((int)m) - 8;
    m <<= sh;
    e = 1 - sh;
  } else {
    m |= 0x800000u;
  }
  const int ev = e - 127 + k;                  // exponent of the shifted value, m in [2^23, 2^24)
  const int sh = 23 - f.y + max(f.emin - ev, 0);
  uint32_t n;
  if (sh > 24) {
    n = 0;
  } else {
    const uint32_t q = m >> sh;
    const uint32_t rem = m & ((1u << sh) - 1u);
    const uint32_t half = 1u << (sh - 1);
    n = q + ((rem > half || (rem == half && (q & 1u))) ? 1u : 0u);
  }
  int code = ev >= f.emin ? ((ev + f.bias) << f.y) + (int)n - (1 << f.y) : (int)n;
  code = min(code, f.code_max);
  code = max(code, 1);
  r.code = (uint32_t)code;
  const int E = code >> f.y;
  const uint32_t M = (uint32_t)code & ((1u << f.y) - 1u);
  const uint32_t mant = E ? ((1u << f.y) + M) : M;
  r.s_hat = ldexp_once(mant, (E ? E : 1) - f.bias - f.y - k);
  return r;
}

// 1 / s rounded to nearest for a normal s whose reciprocal is normal: a Newton step with a fused residual (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", 1990; compared with the correctly rounded reciprocal for every significand).
__device__ __forceinline__ float reciprocal_scale(float s) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(s));
  return __fmaf_rn(y, __fmaf_rn(-s, y, 1.0f), y);
}

// one power-of-two scale per layer: 2^ceil(log2(wmax / tmax))
__device__ __forceinline__ float layer_pot_scale(float wmax, float tmax) {
  if (!(wmax > 0.0f)) return 0.0f;
  const float sigma = __fdiv_rn(wmax, tmax);
  int e = ilogb_pos(sigma);
  const uint32_t b = __float_as_uint(sigma);
  const bool pow2 = (b >> 23) ? ((b & 0x7FFFFFu) == 0u) : (__popc(b) == 1);
  if (!pow2) e += 1;
  return ldexp_once(1u, e);
}

// FP element grids: round |u| to the nearest grid value (ties to even), saturating.
//   E2M3: min_eb = 127 (quantum 2^-3 below 2), vmax = 7.5;  E4M3: min_eb = 121, vmax = 448.
template <int KIND>
__device__ __forceinline__ float fp_quantize(float u) {
  constexpr int min_eb = KIND == SOP_KIND_FP_E2M3 ? 127 : 121;
  constexpr float vmax = KIND == SOP_KIND_FP_E2M3 ? 7.5f : 448.0f;
  const float au = fminf(fabsf(u), vmax);
  // 2^(exponent of au, at least the smallest normal one) * 2^20: adding and subtracting it rounds au to a
  // multiple of the binade's step (3 mantissa bits), ties to even
  const float magic = __uint_as_float(max(__float_as_uint(au) & 0x7F800000u, (uint32_t)min_eb << 23) + (20u << 23));
  const float q = __fsub_rn(__fadd_rn(au, magic), magic);
  return __uint_as_float(__float_as_uint(q) | (__float_as_uint(u) & 0x80000000u));
}

// The same for two values at once through the conversion instructions of the two formats (round to nearest even, saturating,
// sign of zero kept; every E2M3 and E4M3 value is an fp16 number): fp_quantize<KIND> and fp_code<KIND> of x and y, compared for
// every finite fp32 pattern.  The codes come back as bytes, x in the lower one.  A NaN would stay one in E4M3, where
// fp_quantize saturates it: saturate_zeros keeps the one there is away from it.
template <int KIND>
__device__ __forceinline__ float2 fp_quantize2(float x, float y, uint32_t& codes) {
  unsigned short c;
  uint32_t h;
  if (KIND == SOP_KIND_FP_E2M3) {
    asm("cvt.rn.satfinite.e2m3x2.f32 %0, %1, %2;" : "=h"(c) : "f"(y), "f"(x));
    asm("cvt.rn.f16x2.e2m3x2 %0, %1;" : "=r"(h) : "h"(c));
  } else {
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(c) : "f"(y), "f"(x));
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h) : "h"(c));
  }
  codes = c;
  return __half22float2(*reinterpret_cast<const __half2*>(&h));
}

// The weights of a block whose reciprocal scale is infinite (a scale of 2^-128 or below): a zero times it is no number, every other
// weight saturates.  The zeros become the smallest positive weight, which saturates as well, as fp_quantize has it; in the norms of
// such a block it is as good as zero (its square and that of its error underflow).
__device__ __forceinline__ void saturate_zeros(uint32_t (&wb)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const uint32_t zero = __vcmpeq2(wb[q] & 0x7FFF7FFFu, 0u);
    wb[q] = (wb[q] & ~zero) | (zero & 0x00010001u);
  }
}

// Element grid given by parameters (SOP_KIND_FP_GRID): min_eb = biased fp32 exponent of the smallest normal
// magnitude (127 + 1 - bias), sh = 23 - man_bits, saturation at vpos above zero and at vneg below.
struct GridDev { int min_eb, sh; float vpos, vneg; };

__device__ __forceinline__ float grid_quantize(float u, const GridDev g) {
  const float au = fminf(fabsf(u), u < 0.0f ? g.vneg : g.vpos);
  const float magic = __uint_as_float(max(__float_as_uint(au) & 0x7F800000u, (uint32_t)g.min_eb << 23) + ((uint32_t)g.sh << 23));
  const float q = __fsub_rn(__fadd_rn(au, magic), magic);     // nearest multiple of the binade's step, ties to even
  return __uint_as_float(__float_as_uint(q) | (__float_as_uint(u) & 0x80000000u));
}

// magnitude number E * 2^y + M of a value already on such a grid, the sign at bit sign_pos
__device__ __forceinline__ uint32_t grid_code(float q, const GridDev g, int sign_pos) {
  const uint32_t b = __float_as_uint(q);
  const int y = 23 - g.sh;
  const int eb = (int)((b >> 23) & 255u);
  uint32_t mag;
  if (eb < g.min_eb) mag = (uint32_t)__float2int_rn(__fmul_rn(fabsf(q), __uint_as_float((uint32_t)(127 + 127 - g.min_eb + y) << 23)));
  else mag = ((uint32_t)(eb - g.min_eb + 1) << y) | ((b >> g.sh) & ((1u << y) - 1u));
  return ((b >> 31) << sign_pos) | mag;
}

// bit pattern sign|E|M of a value already on the grid
template <int KIND>
__device__ __forceinline__ uint32_t fp_code(float q) {
  constexpr int xb = KIND == SOP_KIND_FP_E2M3 ? 2 : 4;
  constexpr int bias = KIND == SOP_KIND_FP_E2M3 ? 1 : 7;
  const uint32_t b = __float_as_uint(q);
  const uint32_t sign = b >> 31;
  const float a = fabsf(q);
  uint32_t mag;
  if (a < pow2f_int(1 - bias)) {
    mag = (uint32_t)__float2int_rn(__fmul_rn(a, pow2f_int(bias - 1 + 3)));   // subnormal: M = a / 2^(1-bias-3)
  } else {
    const int E = (int)((b >> 23) & 255u) - 127 + bias;
    mag = ((uint32_t)E << 3) | ((b >> 20) & 7u);
  }
  return (sign << (xb + 3)) | mag;
}

// Decision threshold of a table above entry j: the largest fp32 <= (lut[j] + lut[j + 1]) / 2, so that for every fp32 u
// "u > threshold" is exactly "u is strictly closer to lut[j + 1] than to lut[j]".  A repeated entry takes the threshold above
// it, so its upper copy is never chosen.  +inf from the last of ne entries on.
__device__ __forceinline__ float table_threshold(const float* lut, int j, int ne) {
  while (j < ne - 1 && lut[j] == lut[j + 1]) ++j;
  return j < ne - 1 ? __double2float_rd(0.5 * ((double)lut[j] + (double)lut[j + 1])) : __int_as_float(0x7F800000);
}

// number of thresholds strictly below u: branch-free binary search over 2^STEPS - 1 sorted entries (+inf
// padded to 31).  Five steps cover any table; four are enough for a table of at most 16 entries.
template <int STEPS = 5>
__device__ __forceinline__ int count_below(const float* tau, float u) {
  int pos = 0;
#pragma unroll
  for (int step = 1 << (STEPS - 1); step >= 1; step >>= 1)
    if (tau[pos + step - 1] < u) pos += step;
  return pos;
}

// 16-term fp32 sum in the fixed order: four quads of consecutive elements, sequential inside a
// quad, (Q0 + Q1) + (Q2 + Q3).
__device__ __forceinline__ float quad_tree(const float q[4]) {
  return __fadd_rn(__fadd_rn(q[0], q[1]), __fadd_rn(q[2], q[3]));
}

__device__ __forceinline__ float block_cosine(float nw, float nq, float dot) {
  if (nw == 0.0f && nq == 0.0f) return 1.0f;
  if (nw == 0.0f || nq == 0.0f) return 0.0f;
  return __fdiv_rn(dot, __fsqrt_rn(__fmul_rn(nw, nq)));
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Cosines of two candidates at once: RN(dot / RN(sqrt(RN(nw nq)))), the value of block_cosine.  Square root and quotient by
// Newton steps with exact fused residuals and a final correction (P. Markstein, "Computation of elementary functions on the
// IBM RISC System/6000 processor", 1990): from the reciprocal root y the pair g ~ sqrt(x), h ~ 1 / (2 sqrt(x)) is refined once
// and g corrected by its residual x - g^2; 2 h, refined once against the rounded root, is its rounded reciprocal, with which the
// quotient is corrected by its residual.  The signs are chosen so that no operand needs a negation: G = -g, S = -sqrt(x).
// Valid for x in [2^-80, 2^80] and |dot| >= 2^-60 (no intermediate result leaves the normal range) where the rounded root has a
// zero in its significand: the reciprocal of an all-ones significand is halfway between two numbers up to a term that the last
// refinement rounds away, and the quotient of a power of two by it then comes out one step low.  The caller checks both.
constexpr float COS_LO = 8.271806125530277e-25f, COS_HI = 1.2089258196146292e24f, COS_DOT = 8.673617379884035e-19f;
__device__ __forceinline__ float2 cosine_pair(const float2 nx, const float2 dot) {       // nx = -(nw nq)
  const float2 y = make_float2(rsqrt_approx(-nx.x), rsqrt_approx(-nx.y));
  const float2 half = make_float2(0.5f, 0.5f), one = make_float2(1.0f, 1.0f);
  float2 G = __fmul2_rn(nx, y), h = __fmul2_rn(y, half);
  const float2 r = __ffma2_rn(G, h, half);
  G = __ffma2_rn(G, r, G);
  h = __ffma2_rn(h, r, h);
  const float2 D = __ffma2_rn(G, G, nx);
  const float2 S = __ffma2_rn(D, h, G);
  float2 z = __fadd2_rn(h, h);
  const float2 e = __ffma2_rn(S, z, one);
  z = __ffma2_rn(z, e, z);
  const float2 q = __fmul2_rn(dot, z);
  const float2 m = __ffma2_rn(S, q, dot);
  return __ffma2_rn(m, z, q);
}

__device__ __forceinline__ float cosine_one(float nx, float dot) {      // the same steps for one candidate
  const float y = rsqrt_approx(-nx);
  float G = __fmul_rn(nx, y), h = __fmul_rn(y, 0.5f);
  const float r = __fmaf_rn(G, h, 0.5f);
  G = __fmaf_rn(G, r, G);
  h = __fmaf_rn(h, r, h);
  const float S = __fmaf_rn(__fmaf_rn(G, G, nx), h, G);
  float z = __fadd_rn(h, h);
  z = __fmaf_rn(z, __fmaf_rn(S, z, 1.0f), z);
  const float q = __fmul_rn(dot, z);
  return __fmaf_rn(__fmaf_rn(S, q, dot), z, q);
}

// Zero exactly where sqrt(x) rounds to an all-ones significand (the two largest numbers below a power of four, the sign aside).
__device__ __forceinline__ unsigned all_ones_root(float x) { return (__float_as_uint(x) ^ 0x007FFFFEu) & 0x00FFFFFEu; }

}  // namespace sop
