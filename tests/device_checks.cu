// Test kernels: device functions of the library compared over whole ranges of patterns with the instructions or the longer arithmetic
// they stand for.  Each counts its mismatches.
#include "../paper_2605_14929_b200/csrc/sop_device.cuh"

namespace {

// The quotient dot / sqrt(x) of the fast steps against square root and division rounded to nearest, for the patterns x0 .. x0 + n - 1
// and every dot given.  bad[0]: mismatches where the root is not all ones, bad[1]: where it is, bad[2]: such x, [3]: all_ones_root that
// disagrees with the root itself.
__global__ void cosine_kernel(unsigned x0, unsigned n, const float* dots, int n_dots, unsigned long long* bad) {
  unsigned long long b0 = 0, b1 = 0, ones = 0, wrong = 0;
  const unsigned long long total = (unsigned long long)n * (unsigned)n_dots, stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const unsigned at = (unsigned)(i / (unsigned)n_dots), d = (unsigned)(i - (unsigned long long)at * (unsigned)n_dots);
    const float x = __uint_as_float(x0 + at), dot = dots[d], root = __fsqrt_rn(x), want = __fdiv_rn(dot, root);
    const bool all = (__float_as_uint(root) & 0x7FFFFFu) == 0x7FFFFFu;
    if (d == 0) {
      ones += all ? 1 : 0;
      wrong += all != (sop::all_ones_root(x) == 0u) || all != (sop::all_ones_root(-x) == 0u) ? 1 : 0;
    }
    const float2 two = sop::cosine_pair(make_float2(-x, -x), make_float2(dot, -dot));
    const bool differs = __float_as_uint(want) != __float_as_uint(two.x) || __float_as_uint(-want) != __float_as_uint(two.y) ||
                         __float_as_uint(want) != __float_as_uint(sop::cosine_one(-x, dot));
    if (differs) { if (all) ++b1; else ++b0; }
  }
  if (b0) atomicAdd(&bad[0], b0);
  if (b1) atomicAdd(&bad[1], b1);
  if (ones) atomicAdd(&bad[2], ones);
  if (wrong) atomicAdd(&bad[3], wrong);
}

// reciprocal_scale against the reciprocal rounded to nearest, for every significand at one exponent field.
__global__ void reciprocal_kernel(unsigned exponent, unsigned long long* bad) {
  unsigned long long b = 0;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << 23); i += gridDim.x * blockDim.x) {
    const float s = __uint_as_float((exponent << 23) | i);
    if (__float_as_uint(sop::reciprocal_scale(s)) != __float_as_uint(__frcp_rn(s))) ++b;
  }
  if (b) atomicAdd(&bad[0], b);
}

// fp_quantize2 against fp_quantize and fp_code, for every finite pattern in both places; bad[0]: values, bad[1]: codes.
template <int KIND>
__global__ void quantize_kernel(unsigned long long* bad) {
  unsigned long long b0 = 0, b1 = 0;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < (1ull << 32); i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned p = (unsigned)i, r = p * 2654435761u + 12345u;          // another pattern in the other place
    const float x = __uint_as_float(p), y = __uint_as_float((r & 0x7F800000u) == 0x7F800000u ? r & 0xBFFFFFFFu : r);
    if (((p >> 23) & 255u) == 255u) continue;
    const float qx = sop::fp_quantize<KIND>(x), qy = sop::fp_quantize<KIND>(y);
    uint32_t c1, c2;
    const float2 a = sop::fp_quantize2<KIND>(x, y, c1), b = sop::fp_quantize2<KIND>(y, x, c2);
    if (__float_as_uint(a.x) != __float_as_uint(qx) || __float_as_uint(a.y) != __float_as_uint(qy) || __float_as_uint(b.x) != __float_as_uint(qy) ||
        __float_as_uint(b.y) != __float_as_uint(qx)) ++b0;
    const uint32_t cx = sop::fp_code<KIND>(qx), cy = sop::fp_code<KIND>(qy);
    if (c1 != (cx | (cy << 8)) || c2 != (cy | (cx << 8))) ++b1;
  }
  if (b0) atomicAdd(&bad[0], b0);
  if (b1) atomicAdd(&bad[1], b1);
}

}  // namespace

extern "C" int check_reciprocal(unsigned exponent, unsigned long long* bad) {
  reciprocal_kernel<<<1184, 256>>>(exponent, bad);
  return (int)cudaDeviceSynchronize();
}

extern "C" int check_quantize(int kind, unsigned long long* bad) {
  if (kind == SOP_KIND_FP_E2M3) quantize_kernel<SOP_KIND_FP_E2M3><<<1184, 256>>>(bad);
  else quantize_kernel<SOP_KIND_FP_E4M3><<<1184, 256>>>(bad);
  return (int)cudaDeviceSynchronize();
}

extern "C" int check_cosine(unsigned x0, unsigned n, const float* dots, int n_dots, unsigned long long* bad) {
  cosine_kernel<<<1184, 256>>>(x0, n, dots, n_dots, bad);
  return (int)cudaDeviceSynchronize();
}
