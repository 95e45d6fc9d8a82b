// sop_pair_search: the per-layer candidate sweep.
//
//   prepass_kernel   reads W once: per-block absmax -> exponent histogram of sigma = absmax / tmax
//                    for every scale class that needs an F_layer search, and max|W|   (HBM-bound);
//                    the CTA that finishes last derives the F_layer shift k* per class from the
//                    histogram and the layer power-of-two scale for "^0" candidates.
//   kselect_kernel   that last step alone: the shifts of another scale format from the histogram a prepass of the
//                    same layer left in the workspace (SOP_SEARCH_REUSE_PREPASS).
//   sweep_kernel     persistent, one thread per 16-element block: evaluates every candidate of the call.  Table candidates of
//                    one class are evaluated together (up to eight: a "group"): their decision points are merged, an element
//                    looks up the interval it lies in once and reads all eight reconstruction values as one row of shared
//                    memory; packed f32x2 multiply-adds form the block metric in the fixed quad-tree order.  Element formats
//                    go through the conversion instructions.  Writes the per-block cosine and squared error of each candidate
//                    as one column.                                          (bound by register operands and issue)
//   reduce_kernel    reads the columns of every candidate present in the call (those just written
//                    and those an earlier call wrote) tile by tile into shared memory by bulk copies and forms
//                    the table entries: a warp owns a bundle of entries among up to six columns and keeps their
//                    sums in registers (fp32 over eight blocks, then FP64).
//                    The CTA that finishes last adds the per-CTA partials in a fixed order
//                    (deterministic), writes the tables and picks the best pair / best single.
#include <math.h>
#include <string.h>

#include "sop_device.cuh"

namespace sop {

constexpr int TB = 512;             // threads per CTA of the sweep kernel (one CTA per SM; two where it has no table candidates)
constexpr int MAX_SLOTS = 192;      // pair slots per call: 16 singles + 120 pairs + 36 signed < 192
constexpr int MAX_GRID = 1056;
constexpr float MAGIC = 12582912.0f;  // 1.5 * 2^23: adding it rounds to an integer in the low mantissa bits

struct CandDev { unsigned char cls, kind, neg, pad; };
struct ClassDev {
  float tmax;
  int scope, kind;   // kind of the quantiser: LUT, E2M3, E4M3
  int auto_k;        // 1: k* from the histogram
  int n_cand;                            // candidates evaluated in this call
  unsigned char cand[SOP_MAX_ATOMS];
  int n_mem;                             // candidates present in this call (evaluated or loaded)
  unsigned char mem[SOP_MAX_ATOMS];
  int k_src;                             // candidate whose shift an earlier result holds (k from result), or -1
  GridDev grid;                          // kind SOP_KIND_FP_GRID: the grid's parameters
};
// Up to eight table candidates of one class that the sweep evaluates together (see build_group): their joint rows and the
// cell grid that finds the row of a scaled value.
constexpr int GROUP_CAND = 8;
struct GroupDev {
  unsigned char cls, n, np, pad;             // n candidates in np pairs (an odd one is paired with itself)
  unsigned char cand[GROUP_CAND];
  unsigned row_off, cell_off, plane_bytes;   // shared-memory offsets; bytes of the rows of two pairs of candidates
  int n_cells;                               // cells 0 .. n_cells
  float inv_range;                           // cell = rint(n_cells * saturate(u * inv_range + 1/2))
};
struct SlotDev { unsigned char type, i0, i1, pad; };  // type 0: pair (i0, i1) (i0 == i1: single); 1: signed (i0, i0+1, i1, i1+1)

// One unit of work of the reduction (see reduce_run): up to six columns and the entries among them that a warp forms.
// shape 0: a[0..3], their singles and pairs (0,1) (0,2) (0,3) (1,2) (1,3) (2,3); 1: the same of a[0..1]; 2: entry 4 j + i pairs
// a[i] (first candidate) with b[j]; 3: the same with b[0] alone; 4: as 2 with a[i] as the second candidate.  slot: the table slot
// of every entry (255: none).  sgn = 1: the columns stand for base atoms (neg: the column of the negation).
constexpr int RTB = 512;                           // threads per CTA of the reduction (one CTA per SM): fifteen warps form
constexpr int RED_WARPS = 15;                      // entries, one issues the copies
constexpr int BUNDLE_ENT = 10, MAX_BUNDLES = RED_WARPS;
struct BundleDev {
  unsigned char shape, sgn, first_warp, n_warps;
  unsigned char a[4], b[2], neg[6];
  unsigned char slot[BUNDLE_ENT];
};
// One launch of the reduction: its bundles, the bundle of every warp, the candidates whose columns it fetches.
struct BundlesDev {
  int n_bundles, n_cols, n_warps;
  unsigned char warp_bundle[RED_WARPS], cols[SOP_MAX_ATOMS];
  BundleDev bundle[MAX_BUNDLES];
};
struct RedPlan {                            // what the reduction knows of the call
  int n_atoms, n_classes, n_slots, k_from_result, keep_loaded;
  unsigned eval_mask, load_mask, lut_mask;
  unsigned char cls_of[SOP_MAX_ATOMS];
  signed char k_src[SOP_MAX_CLASSES];
  SlotDev slots[MAX_SLOTS];
};

struct Plan {
  int n_atoms, n_classes, n_groups;
  int k_mode;
  unsigned eval_mask, load_mask;   // candidates evaluated here / read from the per-block arrays of an earlier call
  int k_from_result;               // 1: shifts and max|W| come from the result block of an earlier call, no prepass
  CandDev cand[SOP_MAX_ATOMS];
  ClassDev cls[SOP_MAX_CLASSES];
  GroupDev groups[SOP_MAX_CLASSES];
};

struct WsHeader {
  unsigned wmax_bits;
  int cls_k[SOP_MAX_CLASSES];
  float cls_pot[SOP_MAX_CLASSES];
  unsigned done_prepass, done_reduce;  // CTAs that have finished (the last one does the serial tail)
  unsigned reduce_error;               // a wait of the reduction gave up
  int pad[4];
};
// Sums of one entry over a CTA's blocks: gap and error, blocks of the second candidate and of a negated winner (31 bits each).
// Kept as two arrays [CTA][slot] so that the reads of the closing reduction are contiguous.
struct PartialSums { double2* sums; uint2* counts; };

static size_t ws_hist_off() { return 256; }
// after the histograms: max|W| as the prepass found it (the header is cleared by every call, the histograms and this
// word stay until the next prepass)
static size_t ws_wmax_off() { return 256 + sizeof(unsigned) * SOP_MAX_CLASSES * SOP_HIST_BINS; }
static size_t ws_part_off() { return ws_wmax_off() + 256; }
static size_t ws_total() { return ((ws_part_off() + (sizeof(double2) + sizeof(uint2)) * (size_t)MAX_GRID * MAX_SLOTS) + 255) & ~(size_t)255; }

struct LayerArgs {
  const uint16_t* W;
  const float* c;
  long long M, K, ldw;
  long long nbk;      // K / 16
  long long NB;       // M * nbk
};

// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void load_block_bits(const uint16_t* p, uint32_t (&v)[8]) {
  const uint4 a = *reinterpret_cast<const uint4*>(p);
  const uint4 b = *(reinterpret_cast<const uint4*>(p) + 1);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ float absmax_bits(const uint32_t (&v)[8]) {
  // bf16 magnitudes order like their bit patterns: the maximum of the sixteen 15-bit patterns, two per word at a time
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) m = __vmaxu2(m, v[i] & 0x7FFF7FFFu);
  m = max(m & 0xFFFFu, m >> 16);
  return __uint_as_float(m << 16);
}

__device__ void kselect_body(const Plan& P, const FmtDev& F, const unsigned* hist, WsHeader* hdr);

// exponent of sigma = a / tmax (the division rounded as the sweep rounds it), for a > 0; below every bin when sigma is zero
__device__ __forceinline__ int sigma_exponent(float a, float tmax) {
  const float sigma = tmax == 1.0f ? a : __fdiv_rn(a, tmax);
  return sigma > 0.0f ? ilogb_pos(sigma) : -1000;
}

// The exponent of a block's sigma in a class depends on the seven mantissa bits of the block maximum only through one cut
// point: from some mantissa on the quotient reaches the next power of two.  So a block is counted once, by its exponent
// and by the region between the classes' cut points that its mantissa lies in; the CTA's counts are spread to the classes
// at the end.  Where a quotient may leave the normal range the classes are counted one by one.
// A thread stays in its block column and steps down the rows (`rows` whole rows are covered by the grid's threads), four
// blocks in flight.
// What bounds it: DRAM on a large layer (28672 x 8192: 73 us, 470 MB; 106 us with a block per thread in storage order, a division and a
// shared-memory addition per class and block, and max|W| added up by every warp), latency on a small one.
constexpr int PPB = 256;                 // threads per CTA
constexpr int PP_FLY = 4;                // blocks in flight per thread
__global__ void __launch_bounds__(PPB) prepass_kernel(LayerArgs L, Plan P, FmtDev F, unsigned* hist, WsHeader* hdr, unsigned rows) {
  pdl_trigger();
  __shared__ unsigned s_cnt[(SOP_MAX_CLASSES + 1) * 256];      // [region][exponent]
  __shared__ unsigned s_mark[4];                               // mantissas that are a cut point
  __shared__ int s_cut[SOP_MAX_CLASSES], s_e0[SOP_MAX_CLASSES];
  __shared__ unsigned short s_reg[128];                        // 256 x region of a mantissa
  __shared__ unsigned s_wmax;
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < (SOP_MAX_CLASSES + 1) * 256; i += PPB) s_cnt[i] = 0;
  if (tid < SOP_MAX_CLASSES) s_cut[tid] = 128;
  if (tid == 0) s_wmax = 0;
  __syncthreads();
  bool cut = false;
  int e_lo = 1, e_hi = 254;              // exponent fields for which every quotient is a normal number
  for (int cl = 0; cl < P.n_classes; ++cl) {
    if (!P.cls[cl].auto_k) continue;
    const float tmax = P.cls[cl].tmax;
    const int e0 = sigma_exponent(1.0f, tmax);
    e_lo = max(e_lo, 1 - e0);
    e_hi = tmax >= 1e-30f && tmax <= 1e30f ? min(e_hi, 253 - e0) : 0;
    if (tid < 128 && tmax != 1.0f) {
      const int here = sigma_exponent(__uint_as_float((127u << 23) | ((unsigned)tid << 16)), tmax);
      const int below = tid ? sigma_exponent(__uint_as_float((127u << 23) | ((unsigned)(tid - 1) << 16)), tmax) : e0;
      if (here != below) { s_cut[cl] = tid; cut = true; }
    }
    if (tid == 0) s_e0[cl] = e0;
  }
  const unsigned marks = __ballot_sync(0xFFFFFFFFu, cut);
  if (warp < 4 && lane == 0) s_mark[warp] = marks;
  __syncthreads();
  int n_cuts = 0;
#pragma unroll
  for (int w = 0; w < 4; ++w) n_cuts += __popc(s_mark[w]);
  if (tid < 128) {
    int r = __popc(s_mark[warp] & (0xFFFFFFFFu >> (31 - lane)));
    for (int w = 0; w < warp; ++w) r += __popc(s_mark[w]);
    s_reg[tid] = (unsigned short)(256 * r);
  }
  __syncthreads();
  pdl_wait();
  const unsigned nbk = (unsigned)L.nbk, S = rows * nbk, t = blockIdx.x * PPB + tid;
  unsigned wmax = 0;                     // 15-bit patterns
  if (t < S) {
    const unsigned m0 = t / nbk, j = t - m0 * nbk;
    const uint16_t* p = L.W + (long long)m0 * L.ldw + (long long)j * SOP_G;
    const long long step = (long long)rows * L.ldw;
    unsigned left = ((unsigned)L.M - m0 + rows - 1) / rows;      // blocks of this thread
    while (left) {
      uint4 v[PP_FLY][2];
#pragma unroll
      for (int q = 0; q < PP_FLY; ++q) {           // (past the last one the first again: the loads go out together)
        const uint4* w = reinterpret_cast<const uint4*>(q < (int)left ? p + q * step : p);
        v[q][0] = w[0]; v[q][1] = w[1];
      }
      const int n = (int)min(left, (unsigned)PP_FLY);
      p += PP_FLY * step;
      left -= (unsigned)n;
#pragma unroll
      for (int q = 0; q < PP_FLY; ++q) {
        const uint32_t wb[8] = {v[q][0].x, v[q][0].y, v[q][0].z, v[q][0].w, v[q][1].x, v[q][1].y, v[q][1].z, v[q][1].w};
        const unsigned pat = q < n ? __float_as_uint(absmax_bits(wb)) >> 16 : 0u;
        wmax = max(wmax, pat);
        if (pat) {
          const int e = (int)(pat >> 7);
          if (e >= e_lo && e <= e_hi) {
            atomicAdd(&s_cnt[(n_cuts ? s_reg[pat & 127u] : 0) + e], 1u);
          } else {
            for (int cl = 0; cl < P.n_classes; ++cl) {
              if (!P.cls[cl].auto_k) continue;
              const int x = sigma_exponent(__uint_as_float(pat << 16), P.cls[cl].tmax);
              if (x > -1000) atomicAdd(&hist[cl * SOP_HIST_BINS + x + SOP_HIST_OFF], 1u);
            }
          }
        }
      }
    }
  }
  wmax = __reduce_max_sync(0xFFFFFFFFu, wmax);
  if (lane == 0 && wmax) atomicMax(&s_wmax, wmax);
  __syncthreads();
  for (int i = tid; i < (n_cuts + 1) * 256; i += PPB) {
    const unsigned n = s_cnt[i];
    if (!n) continue;
    int first = 0;                       // first mantissa of the region: all of a region's mantissas compare alike with every cut
    for (int r = i >> 8, w = 0; r; ++w) {
      unsigned mk = s_mark[w];
      while (mk && r) { first = 32 * w + __ffs((int)mk) - 1; mk &= mk - 1u; --r; }
    }
    for (int cl = 0; cl < P.n_classes; ++cl)
      if (P.cls[cl].auto_k) atomicAdd(&hist[cl * SOP_HIST_BINS + (i & 255) - 127 + s_e0[cl] + (first >= s_cut[cl] ? 1 : 0) + SOP_HIST_OFF], n);
  }
  if (tid == 0 && s_wmax) atomicMax(&hdr->wmax_bits, s_wmax << 16);
  // the CTA that arrives last turns the histogram into shifts; nobody waits for anybody
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&hdr->done_prepass, 1u) == gridDim.x - 1 ? 1 : 0;
  __syncthreads();
  if (s_last) {
    __threadfence();
    if (tid == 0) hist[SOP_MAX_CLASSES * SOP_HIST_BINS] = __ldcg(&hdr->wmax_bits);    // kept for later calls on this layer
    kselect_body(P, F, hist, hdr);
  }
}

// The shifts of another scale format from the histograms that an earlier prepass of the same layer left in the workspace.
__global__ void __launch_bounds__(256) kselect_kernel(Plan P, FmtDev F, const unsigned* hist, WsHeader* hdr) {
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x == 0) hdr->wmax_bits = hist[SOP_MAX_CLASSES * SOP_HIST_BINS];
  __threadfence();
  __syncthreads();
  kselect_body(P, F, hist, hdr);
}

// One CTA of 256 threads, a warp per class.  Reads the global histogram and max|W| through the L2 (they were written by
// other CTAs' atomics).  Prefix sums of the 320 bins, the count of every shift k in [-64, 64] as a difference of two
// prefix values, then the largest count with ties to the smallest |k| and then to k > 0 (preference order 0, +1, -1,
// +2, -2, ...).  (One class after the other with the whole CTA took 1.5 us per class.)
__device__ void kselect_body(const Plan& P, const FmtDev& F, const unsigned* hist, WsHeader* hdr) {
  static_assert(SOP_MAX_CLASSES <= 8, "a warp per class");
  constexpr int PER = SOP_HIST_BINS / 32;
  static_assert(SOP_HIST_BINS % 32 == 0, "whole bins per lane");
  __shared__ unsigned pre[SOP_MAX_CLASSES][SOP_HIST_BINS + 1];      // (at most one count per block: 31 bits)
  const int lane = threadIdx.x & 31, cl = threadIdx.x >> 5;
  if (cl >= P.n_classes) return;
  int kstar = P.k_mode == SOP_K_AUTO ? 0 : P.k_mode;
  if (P.cls[cl].scope == 0) kstar = 0;
  if (P.cls[cl].auto_k) {
    unsigned v[PER], local = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) v[i] = __ldcg(&hist[cl * SOP_HIST_BINS + PER * lane + i]);
#pragma unroll
    for (int i = 0; i < PER; ++i) local += v[i];
    unsigned incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    unsigned run = incl - local;
#pragma unroll
    for (int i = 0; i < PER; ++i) { pre[cl][PER * lane + i] = run; run += v[i]; }
    if (lane == 31) pre[cl][SOP_HIST_BINS] = run;
    __syncwarp();
    // shift k keeps the exponents e with emin <= e + k <= emax; bin of e is e + SOP_HIST_OFF
    unsigned best = 0;
    int order = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const int o = 32 * i + lane;                           // preference order of the shift
      if (o >= 129) break;
      const int k = (o & 1) ? (o + 1) / 2 : -(o / 2);
      const int lo = max(F.emin - k + SOP_HIST_OFF, 0), hi = min(F.emax - k + SOP_HIST_OFF, SOP_HIST_BINS - 1);
      const unsigned c = hi >= lo ? pre[cl][hi + 1] - pre[cl][lo] : 0u;
      if (i == 0 || c > best) { best = c; order = o; }
    }
    const unsigned top = __reduce_max_sync(0xFFFFFFFFu, best);
    order = (int)__reduce_min_sync(0xFFFFFFFFu, best == top ? (unsigned)order : 0xFFFFu);
    kstar = (order & 1) ? (order + 1) / 2 : -(order / 2);
  }
  if (lane == 0) {
    const float wmax = __uint_as_float(__ldcg(&hdr->wmax_bits));
    hdr->cls_k[cl] = kstar;
    hdr->cls_pot[cl] = P.cls[cl].scope == 0 ? layer_pot_scale(wmax, P.cls[cl].tmax) : 0.0f;
  }
}

// ---------------------------------------------------------------------------------------------
// Evaluators of the sweep.
//
// Table candidates.  The candidates of one class see the same scaled value u of an element, so the decision points of up to
// eight of them (a "group") are merged into one ascending list: between two neighbouring points every candidate's nearest
// entry is fixed, and the eight values of that interval form one row.  Finding the row (a cell of a uniform grid on u, then
// at most three comparisons) and loading it is then paid once per element instead of once per element and candidate, and no
// candidate needs a comparison, a selection or an unpacking of its own: what remains per candidate are the five products and
// sums of its metric, as packed f32x2 operations whose two lanes are two candidates.
// What bounds it: the packed operations read six registers each, and the register file, not the FMA units, limits them (3.2
// cycles each where the units would take 2); the metric of eight candidates alone takes 900 of the 1640 cycles that a warp
// spends on 32 blocks.  More resident warps do not help (256, 384 and 512 threads per SM take the same time).  8192 x 8192 at
// E5M6, eight candidates: 188 us (310 us with a lookup, a comparison and a selection per element and candidate); two
// candidates: 85 us (127 us).
// ---------------------------------------------------------------------------------------------
constexpr int SLOW_STEPS = 8;                        // a binary search over at most 255 decision points

// Shared-memory scratch: while the tables are built, the candidates' values and decision points; for the sweep the merged
// decision points (for a group that is searched).
struct __align__(16) ColumnPtr { float *cos, *sse; };      // a candidate's columns
struct GroupScratch {
  ColumnPtr col[SOP_MAX_CLASSES][GROUP_CAND];
  float vals[GROUP_CAND][32];          // the values of a candidate, in ascending order of u
  float breaks[GROUP_CAND][32];        // the value index of u is the number of these below u (+inf padded)
  float u[SOP_MAX_CLASSES][256];       // merged decision points per group, without repeats (+inf padded)
  unsigned short cell[256];            // their cells
  float sorted[256];                   // the points before repeats are dropped, and which of them is the first of its value
  unsigned char first[256];
  unsigned warp_count[8];
  int n_breaks[SOP_MAX_CLASSES];       // distinct merged decision points
  int per_cell[SOP_MAX_CLASSES];       // the most of them that a cell holds (4: more than three)
};

__device__ __forceinline__ unsigned group_cell(float u, float inv_range, float n_cells) {
  return __float_as_uint(__fmaf_rn(__saturatef(__fmaf_rn(u, inv_range, 0.5f)), n_cells, MAGIC));     // cell number + bits of MAGIC
}

__device__ __forceinline__ int count_not_above(const float* breaks, float u) {      // entries <= u of 31 sorted ones
  int pos = 0;
#pragma unroll
  for (int step = 16; step >= 1; step >>= 1)
    if (breaks[pos + step - 1] <= u) pos += step;
  return pos;
}

// Builds the rows and cells of one group (the whole CTA; at least 256 threads).
//   A candidate is brought into ascending order of u: value index = number of its points below u.  For a negated candidate
//   (the table run on -u) the values are -lut in reverse; its points are the thresholds' negatives, where a tie goes to the
//   upper value (the lower table index), so each moves down by one fp32 step.
//   Row r holds the candidates' values for u in (point r - 1, point r], those of every two pairs in a plane of their own; it is
//   stored in 8 copies of 16 bytes (16 of 8 bytes for a single pair) so that the lanes that load together never meet in a bank.
//   A cell entry is {up to three points of the cell, byte offset of this copy of the row below the first of them}, in as many copies.
__device__ void build_group(const Plan& P, const AtomsDev& A, int g, unsigned char* smem, GroupScratch& S) {
  const GroupDev& G = P.groups[g];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
  for (int i = tid; i < GROUP_CAND * 32; i += nt) {
    const int q = i >> 5, j = i & 31, a = G.cand[q], ne = A.atoms[a].n_entries;
    const bool neg = A.atoms[a].negated != 0;
    const float* lut = ((A.dd_mask >> a) & 1u) ? A.dd_lut : A.atoms[a].lut;
    const int jj = min(j, ne - 1);
    const float v = lut[neg ? ne - 1 - jj : jj];
    S.vals[q][j] = neg ? -v : v;
    float x = __int_as_float(0x7F800000);
    if (j < ne - 1) {
      x = table_threshold(lut, neg ? ne - 2 - j : j, ne);
      if (neg) {
        const float y = -x;
        const unsigned b = __float_as_uint(y);
        x = (b << 1) == 0u ? __uint_as_float(0x80000001u)                      // below zero: the smallest negative number
            : b == 0xFF800000u ? y                                              // -inf: below every u
            : __uint_as_float((b >> 31) ? b + 1u : b - 1u);
      }
    }
    S.breaks[q][j] = x;
  }
  if (tid < 256) S.u[g][tid] = __int_as_float(0x7F800000);
  if (tid == 0) S.per_cell[g] = 0;
  __syncthreads();
  // merge: thread (q, j) finds the place of its point among all, equal points in the order of (q, j); repeats are dropped
  float mine = __int_as_float(0x7F800000);
  int place = 0;
  bool first = false;
  if (tid < GROUP_CAND * 32 && (tid >> 5) < G.n) {
    const int q = tid >> 5, j = tid & 31;
    mine = S.breaks[q][j];
    if (mine < __int_as_float(0x7F800000)) {
      first = j == 0 || S.breaks[q][j - 1] != mine;
#pragma unroll
      for (int b = 0; b < GROUP_CAND; ++b) {
        if (b >= G.n) break;
        const int lt = count_below<5>(S.breaks[b], mine), le = count_not_above(S.breaks[b], mine);
        place += b < q ? le : lt;
        if (b < q && le != lt) first = false;
      }
      place += j - count_below<5>(S.breaks[q], mine);
    }
  }
  if (tid < 256) S.first[tid] = 0;
  __syncthreads();
  if (mine < __int_as_float(0x7F800000)) { S.sorted[place] = mine; S.first[place] = first ? 1 : 0; }
  __syncthreads();
  if (tid < 256) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, S.first[tid] != 0);
    if (lane == 0) S.warp_count[warp] = (unsigned)__popc(m);
  }
  __syncthreads();
  if (tid < 256) {
    const unsigned m = __ballot_sync(0xFFFFFFFFu, S.first[tid] != 0);
    unsigned at = (unsigned)__popc(m & ((1u << lane) - 1u)), total = 0;
    for (int w = 0; w < 8; ++w) { if (w < warp) at += S.warp_count[w]; total += S.warp_count[w]; }
    if (S.first[tid]) {
      S.u[g][at] = S.sorted[tid];
      S.cell[at] = (unsigned short)(group_cell(S.sorted[tid], G.inv_range, (float)G.n_cells) - __float_as_uint(MAGIC));
    }
    if (tid == 0) S.n_breaks[g] = (int)total;
  }
  __syncthreads();
  const int R = S.n_breaks[g];
  for (int i = tid; i < (R + 1) * GROUP_CAND; i += nt) {
    const int r = i >> 3, q = i & 7;
    if (q >= 2 * G.np) continue;
    const float v = S.vals[q][count_below<5>(S.breaks[q], r < R ? S.u[g][r] : __int_as_float(0x7F800000))];
    unsigned char* row = smem + G.row_off + (q >> 2) * G.plane_bytes + r * 128;
    if (G.np == 1) {
      for (int c = 0; c < 16; ++c) *reinterpret_cast<float*>(row + 8 * ((c + r) & 15) + 4 * q) = v;      // (neighbouring threads in different banks)
    } else {
      for (int c = 0; c < 8; ++c) *reinterpret_cast<float*>(row + 16 * ((c + (i >> 2)) & 7) + 4 * (q & 3)) = v;
    }
  }
  for (int k = tid; k <= G.n_cells; k += nt) {
    int lo = 0;                                    // points in lower cells
#pragma unroll
    for (int step = 128; step >= 1; step >>= 1)
      if (lo + step <= R && (int)S.cell[lo + step - 1] < k) lo += step;
    float t[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) t[x] = lo + x < R && (int)S.cell[lo + x] == k ? S.u[g][lo + x] : __int_as_float(0x7F800000);
    int most = 0;
#pragma unroll
    for (int x = 0; x < 4; ++x) most += lo + x < R && (int)S.cell[lo + x] == k ? 1 : 0;
    if (most > 1) atomicMax(&S.per_cell[g], most);
    const int copies = G.np == 1 ? 16 : 8;
    float4* dst = reinterpret_cast<float4*>(smem + G.cell_off) + (size_t)k * copies;
    for (int x = 0; x < copies; ++x) {
      const int c = (x + k) & (copies - 1);
      dst[c] = make_float4(t[0], t[1], t[2], __uint_as_float((unsigned)lo * 128u + (unsigned)c * (128u / copies)));
    }
  }
  __syncthreads();
}

__device__ __forceinline__ float4 lds_f4(unsigned addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __noinline__ float block_cosine_any(float nw, float nq, float dot) { return block_cosine(nw, nq, dot); }

// Rounding of a scale in its usual range, with what does not change from block to block worked out beforehand: the pattern of
// sigma, rounded to nearest even on y mantissa bits by one integer addition (see scale_quantize).
struct ScaleFast {
  unsigned lo, span;          // patterns lo .. lo + span - 1 take the fast path
  unsigned half, mask;        // half a step less one, the bits that are dropped
  int sh;
  __device__ __forceinline__ void init(const FmtDev& F, int k) {
    const int e0 = max(F.emin + 127 - k, 4), e1 = min(F.emax + 127 - k, 250);      // normal, below the top binade, reciprocal normal
    const bool ok = F.y >= 1 && e1 > e0;
    lo = ok ? (unsigned)e0 << 23 : 0u;
    span = ok ? (unsigned)(e1 - e0) << 23 : 0u;
    sh = 23 - F.y;
    half = (1u << (sh - 1)) - 1u;
    mask = (1u << sh) - 1u;
  }
};

// What the block loops of one class share: the class's scale rule and the thread's walk over the rows of its column block.
struct SweepCtx {
  const unsigned char* smem;
  unsigned c_addr;                 // shared-memory address of the thread's channel norms: four, then TB * 16 bytes on the next four
  // scale
  float tmax, pot;
  bool block_scope;
  int k;
  ScaleFast fast;
  // blocks
  const uint16_t* w0;
  long long w_step;
  unsigned n_rows, blk0, blk_step; // this thread's blocks, the number of the first, the step (31 bits: widened where a column is indexed)
  unsigned n_iter;                 // blocks of the thread that has the most

  __device__ __forceinline__ void scale(float amax, const FmtDev& F, float& s_hat, float& rcp) const {
    const float sigma = tmax == 1.0f ? amax : __fdiv_rn(amax, tmax);
    const unsigned b = __float_as_uint(sigma);
    if (block_scope && b - fast.lo < fast.span) {
      s_hat = __uint_as_float((b + fast.half + ((b >> fast.sh) & 1u)) & ~fast.mask);
      rcp = reciprocal_scale(s_hat);
    } else {
      s_hat = !block_scope ? (amax > 0.0f ? pot : 0.0f) : scale_quantize(sigma, k, F).s_hat;
      rcp = s_hat > 0.0f ? __frcp_rn(s_hat) : 0.0f;
    }
  }
};

constexpr unsigned C_STEP = TB * 16u;

// The metrics of NP pairs of candidates on one block: row offsets of its elements in `off` (elements 8 p + i and 8 p + 4 + i
// in the halves of word 4 p + i), their rows at `plane`.  The sums run in the order of the quad tree: four quads of consecutive
// elements, sequential inside a quad, (Q0 + Q1) + (Q2 + Q3).
template <int NP>
__device__ __forceinline__ void sweep_pass(const unsigned char* plane, const uint32_t (&wb)[8], const uint32_t (&off)[8],
                                           unsigned c_addr, float s_hat, float2 (&nq)[NP], float2 (&dot)[NP], float2 (&sse)[NP]) {
  const float2 ns = make_float2(-s_hat, -s_hat);
  float2 n2[NP], d2[NP], s2[NP];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float2 n[NP], d[NP], s[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) n[p] = d[p] = s[p] = make_float2(0.0f, 0.0f);
    const float4 cc = lds_f4(c_addr + (unsigned)h * C_STEP);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = 4 * h + r;
      const float c = r == 0 ? cc.x : r == 1 ? cc.y : r == 2 ? cc.z : cc.w;
      const float w = (i & 1) ? bf16hi(wb[i >> 1]) : bf16lo(wb[i >> 1]);
      const uint32_t o = off[4 * (h >> 1) + r];
      const unsigned char* row = plane + ((h & 1) ? o >> 16 : o & 0xFFFFu);
      float2 q[NP];
      if (NP == 1) {
        q[0] = *reinterpret_cast<const float2*>(row);
      } else {
        const float4 a = *reinterpret_cast<const float4*>(row);
        q[0] = make_float2(a.x, a.y);
        q[NP - 1] = make_float2(a.z, a.w);
      }
      const float2 w2 = make_float2(w, w), c2 = make_float2(c, c);
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const float2 cq = __fmul2_rn(c2, q[p]);
        n[p] = __ffma2_rn(cq, q[p], n[p]);
        d[p] = __ffma2_rn(cq, w2, d[p]);
        const float2 e = __ffma2_rn(ns, q[p], w2);
        s[p] = __ffma2_rn(e, e, s[p]);
      }
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      if (h == 0) { nq[p] = n[p]; dot[p] = d[p]; sse[p] = s[p]; }
      if (h == 1) { nq[p] = __fadd2_rn(nq[p], n[p]); dot[p] = __fadd2_rn(dot[p], d[p]); sse[p] = __fadd2_rn(sse[p], s[p]); }
      if (h == 2) { n2[p] = n[p]; d2[p] = d[p]; s2[p] = s[p]; }
      if (h == 3) {
        nq[p] = __fadd2_rn(nq[p], __fadd2_rn(n2[p], n[p]));
        dot[p] = __fadd2_rn(dot[p], __fadd2_rn(d2[p], d[p]));
        sse[p] = __fadd2_rn(sse[p], __fadd2_rn(s2[p], s[p]));
      }
    }
  }
}

// The cosines of NP pairs from their sums, then both per-block values into the columns.
template <int NP>
__device__ __forceinline__ void sweep_emit(float nw, float2 (&nq)[NP], float2 (&dot)[NP], float2 (&sse)[NP], const ColumnPtr* cols,
                                           unsigned at, bool on) {
  float2 nx[NP];
  unsigned lo = 0xFFFFFFFFu, hi = 0u, ones = 0xFFFFFFFFu;
  float dl = 3.0e38f;
  const float2 nnw = make_float2(-nw, -nw);
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    nx[p] = __fmul2_rn(nnw, nq[p]);
    // compared as patterns: a product that is no number (a sum that overflowed times one that underflowed) lies outside too
    lo = min(lo, min(__float_as_uint(nx[p].x), __float_as_uint(nx[p].y)));
    hi = max(hi, max(__float_as_uint(nx[p].x), __float_as_uint(nx[p].y)));
    ones = min(ones, min(all_ones_root(nx[p].x), all_ones_root(nx[p].y)));
    dl = fminf(dl, fminf(fabsf(dot[p].x), fabsf(dot[p].y)));
  }
  if (lo >= __float_as_uint(-COS_LO) && hi <= __float_as_uint(-COS_HI) && ones && dl >= COS_DOT) {
#pragma unroll
    for (int p = 0; p < NP; ++p) dot[p] = cosine_pair(nx[p], dot[p]);
  } else {
#pragma unroll
    for (int p = 0; p < NP; ++p) dot[p] = make_float2(block_cosine_any(nw, nq[p].x, dot[p].x), block_cosine_any(nw, nq[p].y, dot[p].y));
  }
  if (on) {
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const ColumnPtr a = cols[2 * p], b = cols[2 * p + 1];          // (the last candidate again where their number is odd)
      a.cos[at] = dot[p].x;
      a.sse[at] = sse[p].x;
      b.cos[at] = dot[p].y;
      b.sse[at] = sse[p].y;
    }
  }
}

// The candidates of one group on every block of the thread: first the rows of its sixteen elements (kept as 16-bit offsets),
// then the metrics of two pairs of candidates at a time -- the sums of all eight at once do not fit the 128 registers that a thread
// of 512 has.
//   KT: decision points per cell that are compared (0: the group is searched).
template <int NP, int KT>
__device__ __forceinline__ void sweep_group(const SweepCtx& X, const FmtDev& F, const GroupDev& G, const float* merged, const ColumnPtr* cols) {
  const int lane = threadIdx.x & 31;
  const unsigned copy = NP == 1 ? (unsigned)(lane & 15) * 8u : (unsigned)(lane & 7) * 16u;
  constexpr unsigned CELL = NP == 1 ? 256u : 128u;
  const unsigned cells = G.cell_off + (NP == 1 ? 2u : 1u) * copy - __float_as_uint(MAGIC) * CELL;      // modulo 2^32
  const unsigned char* plane = X.smem + G.row_off;
  const unsigned plane_bytes = G.plane_bytes;
  const float inv_range = G.inv_range, n_cells = (float)G.n_cells;
  const uint16_t* wp = X.w0;
  unsigned at = X.blk0;
  uint32_t wn[8];
  load_block_bits(wp, wn);
#pragma unroll 1
  for (unsigned it = 0; it < X.n_iter; ++it) {
    uint32_t wb[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) wb[q] = wn[q];
    // the next row's block, one iteration ahead; a thread past its last row keeps the block and stores nothing more
    if (it + 1 < X.n_rows) wp += X.w_step;
    load_block_bits(wp, wn);
    float s_hat, rcp;
    X.scale(absmax_bits(wb), F, s_hat, rcp);
    uint32_t off[8];
    float nw4[4];
    const float2 r2 = make_float2(rcp, rcp);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const float4 ca = lds_f4(X.c_addr + (unsigned)(2 * p) * C_STEP), cb = lds_f4(X.c_addr + (unsigned)(2 * p + 1) * C_STEP);
      const float a4[4] = {ca.x, ca.y, ca.z, ca.w}, b4[4] = {cb.x, cb.y, cb.z, cb.w};
      nw4[2 * p] = nw4[2 * p + 1] = 0.0f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int ix = 8 * p + i, iy = ix + 4;
        const float2 w = make_float2((ix & 1) ? bf16hi(wb[ix >> 1]) : bf16lo(wb[ix >> 1]), (iy & 1) ? bf16hi(wb[iy >> 1]) : bf16lo(wb[iy >> 1]));
        const float2 u2 = __fmul2_rn(w, r2);
        nw4[2 * p] = __fmaf_rn(__fmul_rn(a4[i], w.x), w.x, nw4[2 * p]);
        nw4[2 * p + 1] = __fmaf_rn(__fmul_rn(b4[i], w.y), w.y, nw4[2 * p + 1]);
        unsigned o[2];
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const float u = y ? u2.y : u2.x;
          if (KT == 0) {
            unsigned pos = 0;
#pragma unroll
            for (int step = 1 << (SLOW_STEPS - 1); step >= 1; step >>= 1)
              if (merged[pos + step - 1] < u) pos += step;
            o[y] = pos * 128u + copy;
          } else {
            const float4 e = *reinterpret_cast<const float4*>(X.smem + (cells + group_cell(u, inv_range, n_cells) * CELL));
            o[y] = __float_as_uint(e.w);
            if (u > e.x) o[y] += 128u;
            if (u > e.y) o[y] += 128u;
            if (KT > 2 && u > e.z) o[y] += 128u;
          }
        }
        off[4 * p + i] = o[0] + (o[1] << 16);
      }
    }
    const float nw = quad_tree(nw4);
#pragma unroll
    for (int b = 0; b < NP; b += 2) {
      constexpr int LAST = NP % 2 ? 1 : 2;
      if (b + 2 <= NP) {
        float2 nq[2], dot[2], sse[2];
        sweep_pass<2>(plane + (b / 2) * plane_bytes, wb, off, X.c_addr, s_hat, nq, dot, sse);
        sweep_emit<2>(nw, nq, dot, sse, cols + 2 * b, at, it < X.n_rows);
      } else {
        float2 nq[LAST], dot[LAST], sse[LAST];
        sweep_pass<LAST>(plane + (b / 2) * plane_bytes, wb, off, X.c_addr, s_hat, nq, dot, sse);
        sweep_emit<LAST>(nw, nq, dot, sse, cols + 2 * b, at, it < X.n_rows);
      }
    }
    at += X.blk_step;
  }
}

// Element-format candidates (no table): element layout as float2 over elements i of quads 2p (x) and 2p + 1 (y), so that the
// two lanes of a packed operation are two independent sequential chains.
//   MODE: E2M3, E4M3 or a grid given by parameters.  PAIRED: the channel norms lie in shared memory in that layout too.
__device__ __forceinline__ float fold(const float2 a, const float2 b) {
  return __fadd_rn(__fadd_rn(a.x, a.y), __fadd_rn(b.x, b.y));
}

template <int MODE, bool PAIRED>
__device__ __forceinline__ void sweep_format(const SweepCtx& X, const FmtDev& F, const ClassDev& K, size_t NB, float* block_cos,
                                             float* block_sse) {
  const uint16_t* wp = X.w0;
  unsigned at = X.blk0;
  const int n_cand = K.n_cand;
  const GridDev grid = K.grid;
  float *cos0 = block_cos + (size_t)K.cand[0] * NB, *sse0 = block_sse + (size_t)K.cand[0] * NB;
  uint32_t wn[8];
  load_block_bits(wp, wn);
#pragma unroll 1
  for (unsigned it = 0; it < X.n_iter; ++it) {
    uint32_t wb[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) wb[q] = wn[q];
    if (it + 1 < X.n_rows) wp += X.w_step;
    // (the rows after that on their way into L2, there are no registers to hold them: 14336 x 4096, two formats, a pass 178.7 us; 2 us more without)
    if (it + 3 < X.n_rows) asm volatile("prefetch.global.L2 [%0];" ::"l"(wp + 2 * X.w_step));
    load_block_bits(wp, wn);
    float s_hat, rcp;
    X.scale(absmax_bits(wb), F, s_hat, rcp);
    if (MODE == SOP_KIND_FP_E4M3 && isinf(rcp)) saturate_zeros(wb);
    float cc[16];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const float4 v = lds_f4(X.c_addr + (unsigned)h * C_STEP);
      if (PAIRED) { const int i = 8 * (h >> 1) + 2 * (h & 1); cc[i] = v.x; cc[i + 4] = v.y; cc[i + 1] = v.z; cc[i + 5] = v.w; }
      else { cc[4 * h] = v.x; cc[4 * h + 1] = v.y; cc[4 * h + 2] = v.z; cc[4 * h + 3] = v.w; }
    }
    float2 nw2[2], nq[2], dot[2], sse[2];
    nw2[0] = nw2[1] = nq[0] = nq[1] = dot[0] = dot[1] = sse[0] = sse[1] = make_float2(0.0f, 0.0f);
    const float2 ns = make_float2(-s_hat, -s_hat), r2 = make_float2(rcp, rcp);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int ix = 8 * p + i, iy = ix + 4;
        const float2 w = make_float2((ix & 1) ? bf16hi(wb[ix >> 1]) : bf16lo(wb[ix >> 1]), (iy & 1) ? bf16hi(wb[iy >> 1]) : bf16lo(wb[iy >> 1]));
        const float2 c = make_float2(cc[ix], cc[iy]);
        const float2 u = __fmul2_rn(w, r2);
        float2 q;
        if constexpr (MODE == SOP_KIND_FP_GRID) { q.x = grid_quantize(u.x, grid); q.y = grid_quantize(u.y, grid); }
        else { uint32_t codes; q = fp_quantize2<MODE>(u.x, u.y, codes); }
        nw2[p] = __ffma2_rn(__fmul2_rn(c, w), w, nw2[p]);
        const float2 cq = __fmul2_rn(c, q);
        nq[p] = __ffma2_rn(cq, q, nq[p]);
        dot[p] = __ffma2_rn(cq, w, dot[p]);
        const float2 e = __ffma2_rn(ns, q, w);
        sse[p] = __ffma2_rn(e, e, sse[p]);
      }
    }
    const float nw = fold(nw2[0], nw2[1]), nqs = fold(nq[0], nq[1]), dots = fold(dot[0], dot[1]), err = fold(sse[0], sse[1]);
    const float x = __fmul_rn(nw, nqs);
    const float cosv = x >= COS_LO && x <= COS_HI && all_ones_root(x) && fabsf(dots) >= COS_DOT ? cosine_one(-x, dots) : block_cosine_any(nw, nqs, dots);
    if (it < X.n_rows) {
      cos0[at] = cosv;
      sse0[at] = err;
      for (int ci = 1; ci < n_cand; ++ci) {      // (candidates of one format and scale have the same values)
        const size_t col = (size_t)K.cand[ci] * NB + at;
        block_cos[col] = cosv;
        block_sse[col] = err;
      }
    }
    at += X.blk_step;
  }
}

// Evaluates the candidates of eval_mask on every block and writes their columns of block_cos / block_sse: group by group, then
// format by format (W is read again for each: it is a tenth of the time of one).
template <int MAX_NP>
__global__ void __launch_bounds__(TB, MAX_NP == 0 ? 2 : 1) sweep_kernel(LayerArgs L, Plan P, AtomsDev A, FmtDev F, WsHeader* hdr,
                                                      float* block_cos, float* block_sse,
                                                      const sop_search_result* prev, unsigned c_off, unsigned tba) {
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smem[];
  GroupScratch& S = *reinterpret_cast<GroupScratch*>(smem);
  __shared__ int cls_k[SOP_MAX_CLASSES];
  __shared__ float cls_pot[SOP_MAX_CLASSES];

  const int tid = threadIdx.x;
  // the tables of fixed candidates come from the parameters: they are built while the kernel before this one ends
  const bool early = (A.dd_mask & P.eval_mask) == 0u;
  if (early)
    for (int g = 0; g < P.n_groups; ++g) build_group(P, A, g, smem, S);
  pdl_wait();
  if (blockIdx.x == 0 && tid == 0) { hdr->done_reduce = 0u; hdr->reduce_error = 0u; }      // for the reduction that follows
  // thread -> fixed column block j, rows m = r0, r0 + R, ...; its sixteen channel norms stay in shared memory.  Control flow is
  // uniform: a thread with fewer rows evaluates its last block once more and stores nothing.
  const unsigned nbk = (unsigned)L.nbk, M = (unsigned)L.M;       // the block count fits 31 bits
  const unsigned R = gridDim.x * tba / nbk;                      // rows in flight (host guarantees R >= 1)
  const unsigned gt = blockIdx.x * tba + min((unsigned)tid, tba - 1u);
  const unsigned r0 = gt / nbk, j = gt - r0 * nbk;
  SweepCtx X;
  X.smem = smem;
  X.c_addr = smem_u32(smem) + c_off + (unsigned)tid * 16u;
  X.n_iter = (M + R - 1) / R;
  X.n_rows = r0 < R && r0 < M ? (M - r0 + R - 1) / R : 0u;
  X.w0 = L.W + (size_t)j * SOP_G + (long long)min(r0, M - 1) * L.ldw;
  X.w_step = (long long)R * L.ldw;
  X.blk0 = r0 * nbk + j;
  X.blk_step = R * nbk;
  for (int i = tid; i < P.n_groups * GROUP_CAND; i += TB) {
    const size_t at = (size_t)P.groups[i / GROUP_CAND].cand[i % GROUP_CAND] * (size_t)L.NB;
    S.col[i / GROUP_CAND][i % GROUP_CAND] = {block_cos + at, block_sse + at};
  }
  {
    const float4* cp = reinterpret_cast<const float4*>(L.c + (size_t)j * SOP_G);
    float4* dst = reinterpret_cast<float4*>(smem + c_off);
    const float4 v0 = *cp, v1 = cp[1], v2 = cp[2], v3 = cp[3];
    asm volatile("prefetch.global.L2 [%0];" ::"l"(X.w0));          // the first block arrives while the tables are built
    if (MAX_NP == 0) {
      dst[tid] = make_float4(v0.x, v1.x, v0.y, v1.y);
      dst[TB + tid] = make_float4(v0.z, v1.z, v0.w, v1.w);
      dst[2 * TB + tid] = make_float4(v2.x, v3.x, v2.y, v3.y);
      dst[3 * TB + tid] = make_float4(v2.z, v3.z, v2.w, v3.w);
    } else {
      dst[tid] = v0; dst[TB + tid] = v1; dst[2 * TB + tid] = v2; dst[3 * TB + tid] = v3;
    }
  }
  if (tid < SOP_MAX_CLASSES) {
    if (P.k_from_result) {
      const bool live = tid < P.n_classes;
      cls_k[tid] = live && P.cls[tid].k_src >= 0 ? prev->k[P.cls[tid].k_src] : 0;
      cls_pot[tid] = live && P.cls[tid].scope == 0 ? layer_pot_scale(prev->layer_absmax, P.cls[tid].tmax) : 0.0f;
    } else {
      cls_k[tid] = hdr->cls_k[tid];
      cls_pot[tid] = hdr->cls_pot[tid];
    }
  }

  if (!early)
    for (int g = 0; g < P.n_groups; ++g) build_group(P, A, g, smem, S);
  __syncthreads();
  if ((unsigned)tid >= tba) return;                              // (whole warps: they only helped with the tables)

#pragma unroll 1
  for (int x = 0; x < P.n_groups + P.n_classes; ++x) {
    const int cl = x < P.n_groups ? P.groups[x].cls : x - P.n_groups;
    const ClassDev& K = P.cls[cl];
    if (x >= P.n_groups && (K.kind == SOP_KIND_LUT || K.n_cand == 0)) continue;
    X.tmax = K.tmax; X.pot = cls_pot[cl]; X.block_scope = K.scope != 0; X.k = cls_k[cl];
    X.fast.init(F, X.k);
    if (x < P.n_groups) {
      const GroupDev& G = P.groups[x];
      const float* merged = S.u[x];
      const int per_cell = S.per_cell[x];
#define SOP_RUN_GROUP(NP)                                                    \
  if constexpr (NP <= MAX_NP) {                                              \
    if (G.np == NP) {                                                        \
      if (per_cell <= 2) sweep_group<NP, 2>(X, F, G, merged, S.col[x]);            \
      else if (per_cell == 3) sweep_group<NP, 3>(X, F, G, merged, S.col[x]);       \
      else sweep_group<NP, 0>(X, F, G, merged, S.col[x]);                          \
    }                                                                        \
  }
      SOP_RUN_GROUP(1) SOP_RUN_GROUP(2) SOP_RUN_GROUP(3) SOP_RUN_GROUP(4)
#undef SOP_RUN_GROUP
    } else if (K.kind == SOP_KIND_FP_E2M3) sweep_format<SOP_KIND_FP_E2M3, MAX_NP == 0>(X, F, K, (size_t)L.NB, block_cos, block_sse);
    else if (K.kind == SOP_KIND_FP_GRID) sweep_format<SOP_KIND_FP_GRID, MAX_NP == 0>(X, F, K, (size_t)L.NB, block_cos, block_sse);
    else sweep_format<SOP_KIND_FP_E4M3, MAX_NP == 0>(X, F, K, (size_t)L.NB, block_cos, block_sse);
  }
}

// ---------------------------------------------------------------------------------------------
// The reduction of the per-block columns into table entries.
//   A CTA takes tiles of 768 blocks (256 in a small layer).  The columns (cosines and errors of every candidate that the launch
//   needs) of a tile are brought into a ring of up to four shared-memory buffers by bulk copies, one per row, that one thread
//   issues; per buffer an mbarrier says that it has landed and another that its readers are done.
//   The entries are grouped into "bundles": a few columns and the entries among them that a warp forms with everything in
//   registers -- four columns with their singles and six pairs, or four first candidates against two second ones.  A bundle
//   belongs to one or more warps (dealt by its cost), which take every n-th run of 128 blocks, four blocks per lane.
//   An entry costs one comparison and five predicated additions per block (no selections: both outcomes are additions under
//   opposite predicates, so that only the comparison runs on the ALU); its gap 1 - cos and error are summed in fp32 over eight
//   blocks (gaps exactly, for cosines in [0.5, 1]) and then go to FP64 registers of the lane.
//   At the end the lanes' sums are added by a fixed shuffle tree, a bundle's warps in order: the result depends on the launch
//   shape only.
//   A signed four-way entry {i, -i, j, -j} is the two-way entry of "the better of i and -i" and "the better of j and -j"
//   (ties to the atom), formed on the fly from the two columns of each base atom.
//   A block beyond the end of the layer reads as (cos 1, error 0): it adds nothing.
// What bounds it: at an unsigned format the copies (28672 x 8192, both calls of a pass: 2.1 GB of columns in 407 us, 325 us at the
// measured copy rate; 523 us with tasks whose sums lived in shared memory), at a signed format issue (8192 x 8192: 92 + 80 us, 148 +
// 125 us before).  A lane of the copying warp per row matters: one thread issuing twenty copies a tile took 30 % longer; so does the
// tail of the last CTA (see finalize_body): 256 x 1024 takes 11 us, 16 us with the serial tail.
// ---------------------------------------------------------------------------------------------
constexpr int RUNIT = 128;            // blocks of a run: four per lane
constexpr int RED_UNITS = 6;          // runs of a tile, at most
// A lane counts its blocks in 12 bits until they are folded away: after every 128 tiles, of which it sees at most 24 blocks each.
constexpr unsigned COUNT_TILES = 128;
static_assert(COUNT_TILES * RED_UNITS * (RUNIT / 32) < 4096, "a lane's counts fit 12 bits");
constexpr int MAX_STAGE = 4;          // tile buffers of the ring

__device__ void finalize_body(const LayerArgs& L, const RedPlan& P, int grid, PartialSums partials, unsigned char* smem, sop_pair_stat* pair_table,
                              sop_pair_stat* signed_table, sop_search_result* res, const sop_search_result* prev, WsHeader* hdr);

// Sums over the 32 lanes of N values each: in every step a lane hands half of its values to its partner and adds the partner's share
// of the other half, so that N values take about N + 5 exchanges.  Afterwards the lane whose return value is q >= 0 holds the sum of
// value q in v[0] (lanes in pairs hold the same one); -1: the lane holds none.
template <int N, int O>
__device__ __forceinline__ void lane_sums_step(double* v, int lane, int& idx, int& cnt) {
  if constexpr (O > 0) {
    constexpr int H = (N + 1) / 2;
    const bool up = (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const double hi = i + H < N ? v[i + H] : 0.0;
      const double got = __shfl_xor_sync(0xFFFFFFFFu, N > 1 ? (up ? v[i] : hi) : v[i], O);
      v[i] = (N > 1 && up ? hi : v[i]) + got;
    }
    if (N > 1) { idx += up ? H : 0; cnt = up ? cnt - H : min(cnt, H); }
    lane_sums_step<H, O / 2>(v, lane, idx, cnt);
  }
}
template <int N>
__device__ __forceinline__ int lane_sums(double (&v)[N], int lane) {
  int idx = 0, cnt = N;
  lane_sums_step<N, 16>(v, lane, idx, cnt);
  return cnt > 0 ? idx : -1;
}

// One entry on one block: the second candidate takes the block when it is strictly better.  v1 / v0: what the count gains
// when the second / first candidate wins (unsigned entries: 1 and nothing).
template <bool SEL_ERR, bool SGN>
__device__ __forceinline__ void entry_add(float& g, float& e, float& n, float c0, float c1, float g0, float g1, float e0, float e1, float v0, float v1) {
  const float x = SEL_ERR ? e0 : c1, y = SEL_ERR ? e1 : c0;            // strictly better: x > y
  if (SGN)
    asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %3, %4;\n\t@p add.rn.f32 %0, %0, %6;\n\t@!p add.rn.f32 %0, %0, %5;\n\t@p add.rn.f32 %1, %1, %8;\n\t"
        "@!p add.rn.f32 %1, %1, %7;\n\t@p add.rn.f32 %2, %2, %10;\n\t@!p add.rn.f32 %2, %2, %9;\n\t}"
        : "+f"(g), "+f"(e), "+f"(n) : "f"(x), "f"(y), "f"(g0), "f"(g1), "f"(e0), "f"(e1), "f"(v0), "f"(v1));
  else
    asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %3, %4;\n\t@p add.rn.f32 %0, %0, %6;\n\t@!p add.rn.f32 %0, %0, %5;\n\t@p add.rn.f32 %1, %1, %8;\n\t"
        "@!p add.rn.f32 %1, %1, %7;\n\t@p add.rn.f32 %2, %2, 0f3F800000;\n\t}"
        : "+f"(g), "+f"(e), "+f"(n) : "f"(x), "f"(y), "f"(g0), "f"(g1), "f"(e0), "f"(e1));
}

struct ReduceCtx {
  long long NB;
  unsigned n_tiles;                    // tiles of this CTA: blockIdx.x, blockIdx.x + gridDim.x, ...
  int n_cols, units, n_stage;
  int row_len;                         // floats from one row of a tile buffer to the next
  const float* ring;                   // [stage][column][cosines, errors][row_len]
  unsigned full, empty;                // shared-memory addresses of the stages' barriers (8 bytes each)
  const int* row_off;                  // first float of every row in a tile buffer
  WsHeader* hdr;
};

// Waits for the phase of an mbarrier that completes with the given parity.  Bounded: a warp that gives up raises the error flag and
// goes on without waiting; the tables of the call are then marked undefined.
__device__ __forceinline__ void mbar_wait(unsigned bar, unsigned parity, WsHeader* hdr) {
  for (unsigned tries = 0;; ++tries) {
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return;
    if (tries > (1u << 20) || ((tries & 1023u) == 1023u && *(volatile unsigned*)&hdr->reduce_error)) {
      atomicExch(&hdr->reduce_error, 1u);
      return;
    }
  }
}

// The copies of this CTA's tiles by one warp, a lane per row (column, array; at most 32): one bulk copy per row and tile, started at
// the 16-byte boundary at or below its first float and rounded up to whole 16 bytes (the neighbouring floats belong to the same
// 16-byte granule of the array's allocation; what lies beyond the layer is masked by its readers).
__device__ __forceinline__ void reduce_produce(const ReduceCtx& X, unsigned long long row_src) {
  const int tile_len = X.units * RUNIT, rows = 2 * X.n_cols, lane = threadIdx.x & 31;
  const unsigned row_bytes = 4u * (unsigned)X.row_len, dst0 = smem_u32(X.ring) + (unsigned)lane * row_bytes;
  const unsigned skew = (unsigned)(row_src & 15u);       // (tiles are multiples of four blocks)
  int stage = 0;
  unsigned parity = 1;                                   // a fresh barrier passes a wait for the phase before its first
  for (unsigned t = 0; t < X.n_tiles; ++t) {
    const long long blk0 = ((long long)blockIdx.x + (long long)t * gridDim.x) * tile_len;
    const unsigned len = 4u * (unsigned)min((long long)tile_len, X.NB - blk0);
    const unsigned bytes = lane < rows ? (skew + len + 15u) & ~15u : 0u;
    const unsigned total = __reduce_add_sync(0xFFFFFFFFu, bytes);
    const unsigned bar = X.full + 8u * stage;
    mbar_wait(X.empty + 8u * stage, parity, X.hdr);
    if (lane == 0) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(total) : "memory");
    __syncwarp();
    if (lane < rows)
      asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(dst0 + (unsigned)(stage * rows) * row_bytes), "l"(row_src - skew + 4ull * (unsigned long long)blk0), "r"(bytes), "r"(bar) : "memory");
    if (++stage == X.n_stage) { stage = 0; parity ^= 1u; }
  }
}

struct BundleSums {              // what a warp hands to the CTA: the sums of its bundle's entries
  double2 sums[BUNDLE_ENT];
  uint2 counts[BUNDLE_ENT];
  int n_warps;                   // of the bundle, this one the first (the only one with slots)
  unsigned char slot[BUNDLE_ENT + 2];
};

// The loop of one warp (k-th of nk of its bundle) over its runs, SHAPE 0: four columns, their singles and pairs; 1: the same of
// two; 2: four first candidates against two second ones; 3: against one; 4: four second candidates against two first ones.
// The runs of all tiles are dealt in one sequence (run k, k + nk, ...): a warp that has little of one tile has more of the next,
// and the ring lets the warps drift apart by its length.
//   VEC: rows start at 16-byte boundaries, a lane owns four consecutive blocks of a run; else every 32nd.
template <int SHAPE, bool SGN, bool SEL_ERR, bool VEC>
__device__ __forceinline__ void reduce_run(const ReduceCtx& X, const BundleDev& B, int k, int nk, BundleSums* part) {
  constexpr int NA = SHAPE == 1 ? 2 : 4, NBC = SHAPE == 2 || SHAPE == 4 ? 2 : SHAPE == 3 ? 1 : 0, NC = NA + NBC;
  constexpr int NE = SHAPE == 0 ? 10 : SHAPE == 1 ? 3 : SHAPE == 3 ? 4 : 8;
  constexpr int BL = SGN ? 2 : 4;                   // blocks per lane and step: the registers of a signed bundle hold two
  constexpr float NEG = 4096.0f;                    // a count gains 1 for the second candidate, 4096 for a negated winner
  const int lane = threadIdx.x & 31, row_len = X.row_len, lane0 = VEC ? BL * lane : lane;
  int col[SGN ? 2 * NC : NC];                       // VEC: first float of the columns in a tile buffer; else their first row
#pragma unroll
  for (int i = 0; i < NC; ++i) {
    const int c = 2 * (i < NA ? B.a[i] : B.b[i - NA]);
    col[SGN ? 2 * i : i] = VEC ? c * row_len + lane0 : c;
    if (SGN) col[2 * i + 1] = VEC ? 2 * B.neg[i] * row_len + lane0 : 2 * B.neg[i];
  }
  double dg[NE], de[NE];
  float g[NE], e[NE], n[NE];
#pragma unroll
  for (int q = 0; q < NE; ++q) { dg[q] = de[q] = 0.0; g[q] = e[q] = n[q] = 0.0f; }
  auto load = [&](const float* bu, int cc, int arr, float (&v)[BL]) {
    if constexpr (VEC) {
      const float* p = bu + cc + arr * row_len;
      if constexpr (BL == 4) { const float4 t = *reinterpret_cast<const float4*>(p); v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w; }
      else { const float2 t = *reinterpret_cast<const float2*>(p); v[0] = t.x; v[1] = t.y; }
    } else {
      const float* p = bu + X.row_off[cc + arr] + lane0;
#pragma unroll
      for (int r = 0; r < BL; ++r) v[r] = p[32 * r];
    }
  };
  auto fold_sums = [&]() {
#pragma unroll
    for (int q = 0; q < NE; ++q) { dg[q] += (double)g[q]; de[q] += (double)e[q]; g[q] = e[q] = 0.0f; }
  };
  if (lane < BUNDLE_ENT) part->counts[lane] = make_uint2(0u, 0u);
  int stage = 0, run = k, half = 0;                 // run: of this tile, counted from its first
  unsigned parity = 0;
  const unsigned last_full = (unsigned)(X.NB / (X.units * RUNIT));      // tiles below this one are whole
#pragma unroll 1
  for (unsigned t = 0; t < X.n_tiles;) {
    const unsigned t_end = min(t + COUNT_TILES, X.n_tiles);
#pragma unroll 1
    for (; t < t_end; ++t) {
      mbar_wait(X.full + 8u * stage, parity, X.hdr);
      const float* buf = X.ring + (size_t)stage * (2 * X.n_cols) * row_len;
      const long long tile = (long long)blockIdx.x + (long long)t * gridDim.x;
      const int live = tile < last_full ? 1 << 30 : (int)(X.NB - tile * (X.units * RUNIT));       // blocks of this tile
#pragma unroll 1
      for (; run < X.units; run += nk) {
#pragma unroll 1
        for (int h = 0; h < 4 / BL; ++h) {
          const int at = run * RUNIT + h * (32 * BL);
          const float* bu = buf + at;
          float c[NC][BL], er[NC][BL], va[NC][BL];
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            load(bu, col[SGN ? 2 * i : i], 0, c[i]);
            load(bu, col[SGN ? 2 * i : i], 1, er[i]);
            if constexpr (SGN) {
              float mc[BL], me[BL];
              load(bu, col[2 * i + 1], 0, mc);
              load(bu, col[2 * i + 1], 1, me);
#pragma unroll
              for (int r = 0; r < BL; ++r) {
                const bool neg = SEL_ERR ? me[r] < er[i][r] : mc[r] > c[i][r];                    // ties to the atom
                c[i][r] = neg ? mc[r] : c[i][r]; er[i][r] = neg ? me[r] : er[i][r]; va[i][r] = neg ? NEG : 0.0f;
              }
            } else {
#pragma unroll
              for (int r = 0; r < BL; ++r) va[i][r] = 0.0f;
            }
          }
          if (at + 32 * BL > live) {                   // blocks beyond the layer: cosine 1, error 0
#pragma unroll
            for (int i = 0; i < NC; ++i)
#pragma unroll
              for (int r = 0; r < BL; ++r)
                if (at + lane0 + (VEC ? r : 32 * r) >= live) { c[i][r] = 1.0f; er[i][r] = va[i][r] = 0.0f; }
          }
#pragma unroll
          for (int r = 0; r < BL; ++r) {
            float gp[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) gp[i] = __fsub_rn(1.0f, c[i][r]);
            int q = 0;
            if (SHAPE < 2) {
#pragma unroll
              for (int i = 0; i < NA; ++i, ++q) {
                g[q] = __fadd_rn(g[q], gp[i]); e[q] = __fadd_rn(e[q], er[i][r]);
                if (SGN) n[q] = __fadd_rn(n[q], va[i][r]);
              }
#pragma unroll
              for (int i = 0; i < NA; ++i)
#pragma unroll
                for (int j = i + 1; j < NA; ++j, ++q)
                  entry_add<SEL_ERR, SGN>(g[q], e[q], n[q], c[i][r], c[j][r], gp[i], gp[j], er[i][r], er[j][r], va[i][r], SGN ? __fadd_rn(va[j][r], 1.0f) : 1.0f);
            } else {
#pragma unroll
              for (int j = NA; j < NC; ++j)
#pragma unroll
                for (int i = 0; i < NA; ++i, ++q) {
                  const int x = SHAPE == 4 ? j : i, y = SHAPE == 4 ? i : j;        // first and second candidate
                  entry_add<SEL_ERR, SGN>(g[q], e[q], n[q], c[x][r], c[y][r], gp[x], gp[y], er[x][r], er[y][r], va[x][r], SGN ? __fadd_rn(va[y][r], 1.0f) : 1.0f);
                }
            }
          }
        }
        half ^= 1;
        if (!half) fold_sums();                        // eight blocks per lane
      }
      run -= X.units;
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(X.empty + 8u * stage) : "memory");
      if (++stage == X.n_stage) { stage = 0; parity ^= 1u; }
    }
    // the lanes' counts go to the CTA's (lane q keeps those of entry q)
#pragma unroll
    for (int q = 0; q < NE; ++q) {
      const unsigned c = __float2uint_rn(n[q]);                // exact: below 2^24
      const unsigned a = __reduce_add_sync(0xFFFFFFFFu, SGN ? c & 4095u : c), b = SGN ? __reduce_add_sync(0xFFFFFFFFu, c >> 12) : 0u;
      if (lane == q) { part->counts[q].x += a; part->counts[q].y += b; }
      n[q] = 0.0f;
    }
  }
  fold_sums();
  if (lane < BUNDLE_ENT) part->slot[lane] = lane < NE && k == 0 ? B.slot[lane] : (unsigned char)255;
  if (lane == 0) part->n_warps = nk;
  const int q = lane_sums<NE>(dg, lane);
  lane_sums<NE>(de, lane);
  if (q >= 0) part->sums[q] = make_double2(dg[0], de[0]);
}

template <bool SEL_ERR, bool VEC>
__global__ void __launch_bounds__(RTB, 1) reduce_kernel(LayerArgs L, RedPlan P, BundlesDev Q, int units, int n_stage, int do_final,
                                                        WsHeader* hdr, PartialSums partials, const float* block_cos,
                                                        const float* block_sse, sop_pair_stat* pair_table, sop_pair_stat* signed_table,
                                                        sop_search_result* res, const sop_search_result* prev) {
  pdl_trigger();
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ BundleSums s_part[RED_WARPS];
  __shared__ unsigned long long s_row[2 * SOP_MAX_ATOMS];      // address of every fetched row: a column's cosines, its errors
  __shared__ int s_off[2 * SOP_MAX_ATOMS];
  __shared__ __align__(8) unsigned long long s_bar[2 * MAX_STAGE];
  __shared__ int s_last;
  const int tid = threadIdx.x, warp = tid >> 5;
  ReduceCtx X;
  X.NB = L.NB; X.n_cols = Q.n_cols; X.units = units; X.n_stage = n_stage;
  X.row_len = units * RUNIT + (VEC ? 0 : 4);
  const unsigned tiles = (unsigned)((L.NB + units * RUNIT - 1) / (units * RUNIT));
  // (no entry to form: no columns, no warp that would hand a buffer back, nothing to copy)
  X.n_tiles = Q.n_warps && blockIdx.x < tiles ? (tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0u;
  X.ring = reinterpret_cast<const float*>(smem);
  X.full = smem_u32(s_bar); X.empty = X.full + 8u * MAX_STAGE;
  X.row_off = s_off; X.hdr = hdr;
  if (tid < 2 * Q.n_cols) {
    const unsigned long long a = reinterpret_cast<unsigned long long>(((tid & 1) ? block_sse : block_cos) + (size_t)Q.cols[tid >> 1] * (size_t)L.NB);
    s_row[tid] = a;
    s_off[tid] = tid * X.row_len + (int)((a & 15u) >> 2);      // (tiles are multiples of four blocks)
  }
  if (tid == 0) {
    for (int i = 0; i < n_stage && Q.n_warps; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(X.full + 8u * i) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(X.empty + 8u * i), "r"(Q.n_warps) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  pdl_wait();
  __syncthreads();
  BundleSums* mine = s_part + (warp < RED_WARPS ? warp : 0);
  if (warp == RED_WARPS) {
    reduce_produce(X, s_row[tid & 31]);
  } else if (warp < Q.n_warps) {
    const BundleDev& B = Q.bundle[Q.warp_bundle[warp]];
    const int k = warp - B.first_warp, nk = B.n_warps;
    switch (2 * B.shape + B.sgn) {
      case 0: reduce_run<0, false, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 1: reduce_run<0, true, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 2: reduce_run<1, false, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 3: reduce_run<1, true, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 4: reduce_run<2, false, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 5: reduce_run<2, true, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 6: reduce_run<3, false, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 7: reduce_run<3, true, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      case 8: reduce_run<4, false, SEL_ERR, VEC>(X, B, k, nk, mine); break;
      default: reduce_run<4, true, SEL_ERR, VEC>(X, B, k, nk, mine); break;
    }
  }
  __syncthreads();                      // every copy has landed: the warps have waited for each
  // ---- per-CTA partials: a bundle's warps in order ----
  if (tid < Q.n_warps * BUNDLE_ENT) {
    const BundleSums* p = s_part + tid / BUNDLE_ENT;
    const int q = tid % BUNDLE_ENT;
    const unsigned slot = p->slot[q];
    if (slot != 255u) {
      double2 v = p->sums[q];
      uint2 c = p->counts[q];
      const int n = p->n_warps;
#pragma unroll 1
      for (int w = 1; w < n; ++w) { const double2 o = p[w].sums[q]; const uint2 oc = p[w].counts[q]; v.x += o.x; v.y += o.y; c.x += oc.x; c.y += oc.y; }
      partials.sums[(size_t)blockIdx.x * MAX_SLOTS + slot] = v;
      partials.counts[(size_t)blockIdx.x * MAX_SLOTS + slot] = c;
    }
  }
  if (!do_final) return;
  // the CTA that arrives last adds everybody's partials and writes the tables; nobody waits for anybody
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&hdr->done_reduce, 1u) == gridDim.x - 1 ? 1 : 0;
  __syncthreads();
  if (s_last) finalize_body(L, P, (int)gridDim.x, partials, smem, pair_table, signed_table, res, prev, hdr);
}

// One warp.  The defined entry of `tab` ([A x A]) with the largest acos, ties to the smallest index: among the entries above the
// diagonal (diag = 0) or among the diagonal entries of the candidates in lut_mask (diag = 1).  -1: none.
__device__ __noinline__ int warp_best(const sop_pair_stat* tab, int A, int diag, unsigned lut_mask) {
  const int lane = threadIdx.x & 31;
  const unsigned per = 65536u / (unsigned)A + 1u;             // i / A = i per >> 16 for i < 256
  int best = -1;
  double bv = 0.0;
#pragma unroll 1
  for (int i = lane; i < (diag ? A : A * A); i += 32) {
    const int a = diag ? i : (int)((unsigned)i * per >> 16), b = diag ? i : i - a * A;
    const bool in = diag ? ((lut_mask >> a) & 1u) != 0u : b > a;
    const int at = a * A + b;
    if (in && tab[at].n_sel1 >= 0 && (best < 0 || tab[at].acos > bv)) { best = at; bv = tab[at].acos; }
  }
#pragma unroll 1
  for (int o = 16; o; o >>= 1) {
    const double ov = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    if (oi >= 0 && (best < 0 || ov > bv || (ov == bv && oi < best))) { bv = ov; best = oi; }
  }
  return best;
}

// Run by one whole CTA of RTB threads, the last one to arrive: its time is added to every search, so what does not depend on one
// another is loaded together and the three selections run in warps of their own (the serial form took 12 to 20 us of a launch).
// Thread (slot, chunk) adds the partials of CTAs chunk, chunk + C, ... in that order (C = min(RTB / n_slots, ceil(grid / 4)) chunks,
// loads coalesced over the slots and issued eight at a time), the chunks are then added in chunk order: the result depends only on
// the grid size, not on scheduling.
struct FinalSmem {
  sop_pair_stat pair[SOP_MAX_ATOMS * SOP_MAX_ATOMS], sig[SOP_MAX_ATOMS * SOP_MAX_ATOMS];
  double2 sums[RTB];
  uint2 counts[RTB];
};
__device__ void finalize_body(const LayerArgs& L, const RedPlan& P, int grid, PartialSums partials, unsigned char* smem, sop_pair_stat* pair_table,
                              sop_pair_stat* signed_table, sop_search_result* res, const sop_search_result* prev, WsHeader* hdr) {
  __threadfence();
  FinalSmem& S = *reinterpret_cast<FinalSmem*>(smem);
  const int A = P.n_atoms, tid = threadIdx.x, n_slots = P.n_slots;
  const bool failed = *(volatile unsigned*)&hdr->reduce_error != 0u;
  const int n_chunks = max(1, min(RTB / max(n_slots, 1), (grid + 3) / 4));
  const int chunk = tid / max(n_slots, 1), slot = tid - chunk * n_slots;
  if (chunk < n_chunks && n_slots > 0) {
    double2 t = make_double2(0.0, 0.0);
    uint2 c = make_uint2(0u, 0u);
#pragma unroll 1
    for (int g0 = chunk; g0 < grid; g0 += 8 * n_chunks) {
      double2 a[8];
      uint2 b[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const size_t at = (size_t)(g0 + u * n_chunks) * MAX_SLOTS + slot;
        const bool in = g0 + u * n_chunks < grid;
        a[u] = in ? __ldcg(partials.sums + at) : make_double2(0.0, 0.0);
        b[u] = in ? __ldcg(partials.counts + at) : make_uint2(0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) { t.x += a[u].x; t.y += a[u].y; c.x += b[u].x; c.y += b[u].y; }
    }
    S.sums[tid] = t;
    S.counts[tid] = c;
  }
  for (int i = tid; i < 2 * SOP_MAX_ATOMS * SOP_MAX_ATOMS; i += RTB) {
    // entries among candidates that an earlier call evaluated stay as that call left them in the tables
    const int w = i / (SOP_MAX_ATOMS * SOP_MAX_ATOMS), e = i - w * (SOP_MAX_ATOMS * SOP_MAX_ATOMS);
    if (e >= A * A) continue;
    const int a = e / A, b = e - a * A;
    const sop_pair_stat* tab = w ? signed_table : pair_table;
    sop_pair_stat u; u.acos = 0.0; u.mse = 0.0; u.n_sel1 = -1; u.n_neg = -1;
    if (P.keep_loaded && tab && ((P.load_mask >> a) & 1u) && ((P.load_mask >> b) & 1u)) u = tab[e];
    (w ? S.sig : S.pair)[e] = u;
  }
  int k = 0;
  float wmax = 0.0f;
  if (tid >= RTB - 32) {
    const int i = tid - (RTB - 32);
    if (i < A && (((P.eval_mask | P.load_mask) >> i) & 1u)) {
      const int cl = P.cls_of[i];
      k = P.k_from_result ? (P.k_src[cl] >= 0 ? prev->k[P.k_src[cl]] : 0) : __ldcg(&hdr->cls_k[cl]);
    }
    wmax = P.k_from_result ? prev->layer_absmax : __uint_as_float(__ldcg(&hdr->wmax_bits));
  }
  SlotDev sd = {0, 0, 0, 0};
  if (tid < n_slots) sd = P.slots[tid];
  __syncthreads();
  if (tid < n_slots && !failed) {      // (a wait that gave up: every entry formed here stays undefined)
    double2 t = S.sums[tid];
    uint2 c = S.counts[tid];
#pragma unroll 4
    for (int q = 1; q < n_chunks; ++q) {
      const double2 o = S.sums[q * n_slots + tid];
      const uint2 oc = S.counts[q * n_slots + tid];
      t.x += o.x; t.y += o.y; c.x += oc.x; c.y += oc.y;
    }
    sop_pair_stat st;
    st.acos = ((double)L.NB - t.x) / (double)L.NB;
    st.mse = t.y / ((double)L.M * (double)L.K);
    st.n_sel1 = (long long)c.x;
    st.n_neg = sd.type ? (long long)c.y : 0;
    (sd.type ? S.sig : S.pair)[sd.i0 * A + sd.i1] = st;
  }
  __syncthreads();
  // best two-codebook pair, best single LUT candidate, best signed pair: largest ACos, ties to the smallest (a, b)
  if (tid < 96) {
    const int w = tid >> 5;
    const int best = w == 2 && !signed_table ? -1 : warp_best(w == 2 ? S.sig : S.pair, A, w == 1, P.lut_mask);
    if ((tid & 31) == 0) {
      const int a = best >= 0 ? best / A : -1, b = best >= 0 ? best - a * A : -1;
      if (w == 0) { res->best_a = a; res->best_b = b; }
      else if (w == 1) res->best_single = a;
      else { res->best_sa = a; res->best_sb = b; }
    }
  } else if (tid >= RTB - 32) {
    const int i = tid - (RTB - 32);
    if (i < SOP_MAX_ATOMS) res->k[i] = k;
    if (i == 0) { res->layer_absmax = wmax; res->reserved[0] = res->reserved[1] = 0; }
  } else {
    for (int i = tid - 96; i < A * A; i += RTB - 128) {
      pair_table[i] = S.pair[i];
      if (signed_table) signed_table[i] = S.sig[i];
    }
  }
}

// ---------------------------------------------------------------------------------------------
// host: plan construction
// ---------------------------------------------------------------------------------------------
static bool same_table(const sop_atom& a, const sop_atom& b) {
  return a.n_entries == b.n_entries && memcmp(a.lut, b.lut, sizeof(float) * a.n_entries) == 0;
}

int build_plan(const AtomsDev& A, const FmtDev& F, int k_mode, unsigned eval_mask, unsigned load_mask, int singles_only, int keep_loaded, Plan* P, RedPlan* Rp) {
  memset(P, 0, sizeof(*P));
  memset(Rp, 0, sizeof(*Rp));
  const int n = A.n_atoms;
  P->n_atoms = n;
  P->k_mode = k_mode;
  P->eval_mask = eval_mask;
  P->load_mask = load_mask;
  const unsigned present = eval_mask | load_mask;
  int n_tables = 0, table_atom[SOP_MAX_TABLES], table_signs[SOP_MAX_TABLES];
  // classes
  for (int i = 0; i < n; ++i) {
    const sop_atom& a = A.atoms[i];
    P->cand[i].kind = (unsigned char)a.kind;
    P->cand[i].neg = (unsigned char)a.negated;
    if (!((present >> i) & 1u)) continue;
    int cl = -1;
    for (int c = 0; c < P->n_classes; ++c)
      if (P->cls[c].scope == a.scope && P->cls[c].tmax == a.tmax && P->cls[c].kind == a.kind &&
          (a.kind != SOP_KIND_FP_GRID || (P->cls[c].grid.min_eb == 128 - a.grid_bias && P->cls[c].grid.sh == 23 - a.grid_man_bits &&
                                          P->cls[c].grid.vneg == a.grid_neg_max))) cl = c;
    if (cl < 0) {
      if (P->n_classes == SOP_MAX_CLASSES) return SOP_ERR_ALPHABET;
      cl = P->n_classes++;
      P->cls[cl].scope = a.scope; P->cls[cl].tmax = a.tmax; P->cls[cl].kind = a.kind;
      P->cls[cl].auto_k = (k_mode == SOP_K_AUTO && a.scope != 0) ? 1 : 0;
      P->cls[cl].grid.min_eb = 128 - a.grid_bias; P->cls[cl].grid.sh = 23 - a.grid_man_bits;
      P->cls[cl].grid.vpos = a.tmax; P->cls[cl].grid.vneg = a.grid_neg_max;
    }
    ClassDev& C = P->cls[cl];
    C.mem[C.n_mem++] = (unsigned char)i;
    P->cand[i].cls = (unsigned char)cl;
    if (!((eval_mask >> i) & 1u)) continue;
    C.cand[C.n_cand++] = (unsigned char)i;
    if (a.kind != SOP_KIND_LUT) continue;
    // distinct tables of the call (an atom and its negation share one)
    const bool dd = (A.dd_mask >> i) & 1u;
    int t = -1;
    for (int q = 0; q < n_tables; ++q) {
      const int o = table_atom[q];
      if (P->cand[o].cls != cl || (((A.dd_mask >> o) & 1u) != 0) != dd || ((table_signs[q] >> a.negated) & 1)) continue;
      if (dd ? (A.atoms[o].n_entries == a.n_entries) : same_table(A.atoms[o], a)) t = q;
    }
    if (t < 0) {
      if (n_tables == SOP_MAX_TABLES) return SOP_ERR_ALPHABET;
      t = n_tables++;
      table_atom[t] = i;
      table_signs[t] = 0;
    }
    table_signs[t] |= 1 << a.negated;
  }
  // groups of up to eight table candidates of one class (never more groups than distinct tables: eight candidates that differ
  // have at least four)
  for (int c = 0; c < P->n_classes; ++c) {
    if (P->cls[c].kind != SOP_KIND_LUT) continue;
    for (int i = 0; i < P->cls[c].n_cand; i += GROUP_CAND) {
      if (P->n_groups == SOP_MAX_CLASSES) return SOP_ERR_ALPHABET;
      GroupDev& G = P->groups[P->n_groups++];
      G.cls = (unsigned char)c;
      G.n = (unsigned char)(P->cls[c].n_cand - i < GROUP_CAND ? P->cls[c].n_cand - i : GROUP_CAND);
      G.np = (unsigned char)((G.n + 1) / 2);
      for (int q = 0; q < GROUP_CAND; ++q) G.cand[q] = P->cls[c].cand[i + (q < G.n ? q : G.n - 1)];
      G.inv_range = (float)(1.0 / (2.5 * (double)P->cls[c].tmax));       // the cells cover |u| <= 1.25 tmax, the end cells everything beyond
    }
  }
  // slots: pair-type first (singles as (a, a)), then signed.  With keep_loaded an entry whose candidates were all
  // evaluated by an earlier call is not formed again: the tables hold it.
  Rp->keep_loaded = keep_loaded;
  int ns = 0;
  auto has = [present](int i) { return ((present >> i) & 1u) != 0; };
  auto old = [keep_loaded, load_mask](int i) { return keep_loaded && ((load_mask >> i) & 1u) != 0; };
  for (int a = 0; a < n; ++a) {
    if (!has(a) || old(a)) continue;
    Rp->slots[ns].type = 0; Rp->slots[ns].i0 = Rp->slots[ns].i1 = (unsigned char)a; ++ns;
  }
  for (int a = 0; a < n && !singles_only; ++a)
    for (int b = a + 1; b < n; ++b) {
      if (!has(a) || !has(b) || (old(a) && old(b))) continue;
      if (A.atoms[a].kind != SOP_KIND_LUT || A.atoms[b].kind != SOP_KIND_LUT || A.atoms[a].n_bits != A.atoms[b].n_bits) continue;
      Rp->slots[ns].type = 0; Rp->slots[ns].i0 = (unsigned char)a; Rp->slots[ns].i1 = (unsigned char)b; ++ns;
    }
  if (F.sign_bits && !singles_only) {
    bool base[SOP_MAX_ATOMS];
    for (int i = 0; i < n; ++i) {
      base[i] = false;
      if (i + 1 >= n || !has(i) || !has(i + 1)) continue;
      const sop_atom &a = A.atoms[i], &b = A.atoms[i + 1];
      if (a.kind != SOP_KIND_LUT || b.kind != SOP_KIND_LUT || a.negated || !b.negated || a.tmax != b.tmax) continue;
      const bool da = (A.dd_mask >> i) & 1u, db = (A.dd_mask >> (i + 1)) & 1u;
      base[i] = (da && db && a.n_entries == b.n_entries) || (!da && !db && same_table(a, b));
    }
    for (int i = 0; i < n; ++i)
      for (int j = i; j < n; ++j) {
        if (!base[i] || !base[j] || A.atoms[i].n_bits != A.atoms[j].n_bits) continue;
        if (old(i) && old(i + 1) && old(j) && old(j + 1)) continue;
        Rp->slots[ns].type = 1; Rp->slots[ns].i0 = (unsigned char)i; Rp->slots[ns].i1 = (unsigned char)j; ++ns;   // base atoms
      }
  }
  if (ns > MAX_SLOTS) return SOP_ERR_ALPHABET;
  Rp->n_slots = ns;
  Rp->n_atoms = n; Rp->n_classes = P->n_classes; Rp->eval_mask = eval_mask; Rp->load_mask = load_mask;
  for (int i = 0; i < n; ++i) {
    Rp->cls_of[i] = P->cand[i].cls;
    if (A.atoms[i].kind == SOP_KIND_LUT) Rp->lut_mask |= 1u << i;
  }
  return SOP_OK;
}

// The bundles that form the slots of a plan.  Per kind of entry (two-way, signed): first the candidates with a single entry in
// fours (twos for a rest of two) with the pairs among them, then the remaining pairs as rectangles -- the second candidate with
// the most pairs left and the one that shares the most first candidates with it, against up to four of those; where one first
// candidate meets many second ones the rectangle is taken the other way round.
struct BundleList { int n; BundleDev b[MAX_SLOTS]; };      // (every bundle forms at least one entry)
static void build_bundles(const RedPlan& P, BundleList* out) {
  out->n = 0;
  for (int ty = 0; ty < 2; ++ty) {
    int slot_of[SOP_MAX_ATOMS][SOP_MAX_ATOMS];
    for (int i = 0; i < SOP_MAX_ATOMS; ++i)
      for (int j = 0; j < SOP_MAX_ATOMS; ++j) slot_of[i][j] = 255;
    int single[SOP_MAX_ATOMS], n_single = 0;
    for (int s = 0; s < P.n_slots; ++s)
      if (P.slots[s].type == ty) slot_of[P.slots[s].i0][P.slots[s].i1] = s;
    for (int i = 0; i < SOP_MAX_ATOMS; ++i)
      if (slot_of[i][i] != 255) single[n_single++] = i;
    auto make = [&](int shape) {
      BundleDev B;
      memset(&B, 0, sizeof(B));
      memset(B.slot, 255, sizeof(B.slot));
      B.shape = (unsigned char)shape; B.sgn = (unsigned char)ty;
      return B;
    };
    for (int at = 0; at < n_single;) {
      const int take = n_single - at < 4 ? n_single - at : 4;
      const int na = take <= 2 ? 2 : 4;
      BundleDev B = make(take <= 2 ? 1 : 0);
      for (int i = 0; i < na; ++i) B.a[i] = (unsigned char)single[at + (i < take ? i : take - 1)];
      int q = 0;
      for (int i = 0; i < na; ++i, ++q)
        if (i < take) { B.slot[q] = (unsigned char)slot_of[B.a[i]][B.a[i]]; slot_of[B.a[i]][B.a[i]] = 255; }
      for (int i = 0; i < na; ++i)
        for (int j = i + 1; j < na; ++j, ++q)
          if (j < take) { B.slot[q] = (unsigned char)slot_of[B.a[i]][B.a[j]]; slot_of[B.a[i]][B.a[j]] = 255; }
      out->b[out->n++] = B;
      at += take;
    }
    for (;;) {
      // rev = 0: x is the second candidate of its pairs (column of the matrix), rev = 1: the first (row)
      auto left = [&](int rev, int x, int y) { return (rev ? slot_of[x][y] : slot_of[y][x]) != 255; };
      int best = 0, brev = 0, bx = 0;
      for (int rev = 0; rev < 2; ++rev)
        for (int x = 0; x < SOP_MAX_ATOMS; ++x) {
          int c = 0;
          for (int y = 0; y < SOP_MAX_ATOMS; ++y) c += left(rev, x, y) ? 1 : 0;
          if ((c < 4 ? c : 4) > best) { best = c < 4 ? c : 4; brev = rev; bx = x; }
        }
      if (!best) break;
      int b2 = -1, shared = 0;
      for (int x = 0; x < SOP_MAX_ATOMS; ++x) {
        if (x == bx) continue;
        int c = 0;
        for (int y = 0; y < SOP_MAX_ATOMS; ++y) c += left(brev, bx, y) && left(brev, x, y) ? 1 : 0;
        if ((c < 4 ? c : 4) > shared) { shared = c < 4 ? c : 4; b2 = x; }
      }
      if (2 * shared < best) b2 = -1;                 // hardly anything in common: one at a time
      BundleDev B = make(brev ? 4 : b2 < 0 ? 3 : 2);
      B.b[0] = (unsigned char)bx; B.b[1] = (unsigned char)(b2 < 0 ? bx : b2);
      int n = 0;
      for (int pass = 0; pass < 2 && n < 4; ++pass)    // what both share first
        for (int y = 0; y < SOP_MAX_ATOMS && n < 4; ++y) {
          const bool both = b2 >= 0 && left(brev, bx, y) && left(brev, b2, y);
          if (left(brev, bx, y) && (pass == 0 ? both || b2 < 0 : !both && b2 >= 0)) B.a[n++] = (unsigned char)y;
        }
      for (int i = n; i < 4; ++i) B.a[i] = B.a[n - 1];
      for (int j = 0; j < (b2 < 0 ? 1 : 2); ++j)
        for (int i = 0; i < n; ++i) {
          int& s = brev ? slot_of[B.b[j]][B.a[i]] : slot_of[B.a[i]][B.b[j]];
          B.slot[4 * j + i] = (unsigned char)s;
          s = 255;
        }
      out->b[out->n++] = B;
    }
  }
}

// One launch of up to fifteen bundles: the columns it fetches, the columns' places in the bundles, and the warps dealt to them,
// always to the bundle whose warps have the most to do (instructions per run).
static void deal_bundles(const BundleDev* b, int n, BundlesDev* Q) {
  memset(Q, 0, sizeof(*Q));
  Q->n_bundles = n;
  unsigned cand = 0;
  auto cols_of = [](const BundleDev& B) { return B.shape == 0 ? 4 : B.shape == 1 ? 2 : B.shape == 3 ? 5 : 6; };
  auto col = [](const BundleDev& B, int i) { const int na = B.shape == 1 ? 2 : 4; return i < na ? (int)B.a[i] : (int)B.b[i - na]; };
  for (int i = 0; i < n; ++i)
    for (int c = 0; c < cols_of(b[i]); ++c) cand |= (b[i].sgn ? 3u : 1u) << col(b[i], c);
  int place[SOP_MAX_ATOMS + 1] = {0};
  for (int a = 0; a < SOP_MAX_ATOMS; ++a)
    if ((cand >> a) & 1u) { place[a] = Q->n_cols; Q->cols[Q->n_cols++] = (unsigned char)a; }
  int cost[MAX_BUNDLES], nw[MAX_BUNDLES];
  for (int i = 0; i < n; ++i) {
    BundleDev B = b[i];
    const int nc = cols_of(B), ne = B.shape == 0 ? 10 : B.shape == 1 ? 3 : B.shape == 3 ? 4 : 8;
    cost[i] = B.sgn ? 15 * ne + 24 * nc : 13 * ne + 6 * nc;
    nw[i] = 1;
    const int na = B.shape == 1 ? 2 : 4;
    for (int c = 0; c < nc; ++c) {
      const int a = col(b[i], c);
      (c < na ? B.a[c] : B.b[c - na]) = (unsigned char)place[a];
      if (B.sgn) B.neg[c] = (unsigned char)place[a + 1];
    }
    Q->bundle[i] = B;
  }
  for (int w = n; w < RED_WARPS && n; ++w) {
    int pick = 0;
    for (int i = 1; i < n; ++i)
      if (cost[i] * nw[pick] > cost[pick] * nw[i]) pick = i;
    ++nw[pick];
  }
  int at = 0;
  for (int i = 0; i < n; ++i) {
    Q->bundle[i].first_warp = (unsigned char)at; Q->bundle[i].n_warps = (unsigned char)nw[i];
    for (int w = 0; w < nw[i]; ++w) Q->warp_bundle[at++] = (unsigned char)i;
  }
  Q->n_warps = at;
}

// Tiles of 768 blocks, of 256 where those would leave SMs without one; at most one CTA per SM, and never more than the workspace has
// partials for.
static long long reduce_grid(long long NB, int sms, int* units) {
  *units = NB >= (long long)sms * RED_UNITS * RUNIT ? RED_UNITS : 2;
  const long long n_tiles = (NB + *units * RUNIT - 1) / (*units * RUNIT), most = sms < MAX_GRID ? sms : MAX_GRID;
  return n_tiles < most ? n_tiles : most;
}

// the ring of tile buffers; at least the room the closing reduction of the last CTA needs
static size_t reduce_smem_bytes(int n_cols, int units, int n_stage) {
  const size_t ring = (size_t)n_stage * n_cols * 2 * (units * RUNIT + 4) * sizeof(float);
  const size_t fin = sizeof(FinalSmem);
  return ((ring > fin ? ring : fin) + 127) & ~(size_t)127;
}

// Shared memory of the sweep: per group its rows (one more than its decision points) and its cells, 128 bytes per cell and
// 128 or 256 per row with the copies; every group gets the same number of cells, the largest of 640, 320, 160, ... that fits
// `limit` bytes in all (a cell then rarely holds more than three decision points; a group where one does is searched instead).
constexpr size_t SWEEP_C_BYTES = (size_t)TB * SOP_G * sizeof(float);
static size_t sweep_layout(const AtomsDev& A, Plan* P, size_t limit) {
  for (int cells = 640;; cells /= 2) {
    size_t b = (sizeof(GroupScratch) + 127) & ~(size_t)127;
    for (int g = 0; g < P->n_groups; ++g) {
      GroupDev& G = P->groups[g];
      int breaks = 0;
      for (int q = 0; q < G.n; ++q) breaks += A.atoms[G.cand[q]].n_entries - 1;
      G.row_off = (unsigned)b;
      G.plane_bytes = (unsigned)(breaks + 1) * 128u;
      b += (size_t)G.plane_bytes * (size_t)((G.np + 1) / 2);
      G.cell_off = (unsigned)b;
      G.n_cells = cells;
      b += (size_t)(cells + 1) * (G.np == 1 ? 256 : 128);
    }
    b += SWEEP_C_BYTES;                           // the threads' channel norms
    if (b <= limit || cells <= 20) return b;
  }
}

// sop_pair_search_tuning(0): a ring of two tile buffers instead of as many as fit, up to four (tests compare both: the results
// are the same bit for bit).
static bool g_reduce_ring = true;

}  // namespace sop

extern "C" {

int sop_pair_search_tuning(int reduce_tile_pairs) {
  if (reduce_tile_pairs != 0 && reduce_tile_pairs != 1) return SOP_ERR_RANGE;
  sop::g_reduce_ring = reduce_tile_pairs != 0;
  return SOP_OK;
}

int sop_pair_search_workspace(long long M, long long K, int n_atoms, size_t* bytes) {
  if (!bytes) return SOP_ERR_NULL;
  if (M < 1 || K < 1 || (K % SOP_G) != 0) return SOP_ERR_SHAPE;
  if (n_atoms < 1 || n_atoms > SOP_MAX_ATOMS) return SOP_ERR_ALPHABET;
  *bytes = sop::ws_total();
  return SOP_OK;
}

int sop_pair_search(const void* W_dev, long long M, long long K, long long ldw, const float* c_dev, int g,
                    const sop_scale_fmt* fmt, int k_mode, const sop_atom* atoms, int n_atoms,
                    const float* dd_lut_dev, unsigned dd_mask, unsigned eval_mask, unsigned load_mask, int flags,
                    const sop_search_result* prev_result_dev,
                    sop_pair_stat* pair_table_dev, sop_pair_stat* signed_table_dev,
                    sop_search_result* result_dev, float* block_cos_dev, float* block_sse_dev,
                    void* workspace_dev, size_t workspace_bytes, void* stream) {
  using namespace sop;
  int rc = validate_layer(W_dev, M, K, ldw, c_dev, g);
  if (rc) return rc;
  if (!pair_table_dev || !result_dev) return SOP_ERR_NULL;
  FmtDev F;
  if ((rc = validate_fmt(fmt, &F))) return rc;
  AtomsDev A;
  if ((rc = validate_atoms(atoms, n_atoms, dd_mask, dd_lut_dev, &A))) return rc;
  const bool k_from_result = k_mode == SOP_K_FROM_RESULT;
  if (k_mode != SOP_K_AUTO && !k_from_result && (k_mode < -64 || k_mode > 64)) return SOP_ERR_RANGE;
  if (k_from_result && (!prev_result_dev || prev_result_dev == result_dev)) return SOP_ERR_NULL;
  const long long NB = M * (K / SOP_G);
  // without the caller's per-block arrays the columns live behind the fixed part of the workspace
  const bool own_columns = !block_cos_dev || !block_sse_dev;
  const size_t col_bytes = (((size_t)n_atoms * (size_t)NB * sizeof(float)) + 255) & ~(size_t)255;
  const size_t need = ws_total() + (own_columns ? 2 * col_bytes : 0);
  if (!workspace_dev || ((uintptr_t)workspace_dev & 255u) || workspace_bytes < need) return SOP_ERR_WORKSPACE;
  const unsigned all = n_atoms >= 32 ? 0xFFFFFFFFu : ((1u << n_atoms) - 1u);
  eval_mask &= all;
  if ((load_mask & ~all) || (load_mask & eval_mask) || !(eval_mask | load_mask)) return SOP_ERR_ALPHABET;
  if (load_mask && own_columns) return SOP_ERR_NULL;
  if (flags & ~(SOP_SEARCH_SINGLES_ONLY | SOP_SEARCH_SELECT_MSE | SOP_SEARCH_KEEP_LOADED_ENTRIES | SOP_SEARCH_REUSE_PREPASS)) return SOP_ERR_RANGE;
  const bool reuse_prepass = (flags & SOP_SEARCH_REUSE_PREPASS) && !k_from_result;
  const int keep_loaded = (flags & SOP_SEARCH_KEEP_LOADED_ENTRIES) && load_mask ? 1 : 0;
  Plan P;
  RedPlan Rp;
  if ((rc = build_plan(A, F, k_from_result ? 0 : k_mode, eval_mask, load_mask, flags & SOP_SEARCH_SINGLES_ONLY, keep_loaded, &P, &Rp))) return rc;
  P.k_from_result = Rp.k_from_result = k_from_result ? 1 : 0;
  for (int c = 0; c < P.n_classes; ++c) {
    // the shift of a class is read from a candidate of that class that the earlier call had
    P.cls[c].k_src = -1;
    for (int i = 0; i < P.cls[c].n_mem; ++i)
      if ((load_mask >> P.cls[c].mem[i]) & 1u) { P.cls[c].k_src = P.cls[c].mem[i]; break; }
    Rp.k_src[c] = (signed char)P.cls[c].k_src;
    if (k_from_result && P.cls[c].scope != 0 && P.cls[c].k_src < 0) return SOP_ERR_RANGE;
  }

  LayerArgs L;
  L.W = (const uint16_t*)W_dev; L.c = c_dev; L.M = M; L.K = K; L.ldw = ldw; L.nbk = K / SOP_G; L.NB = NB;
  cudaStream_t st = (cudaStream_t)stream;
  unsigned char* ws = (unsigned char*)workspace_dev;
  WsHeader* hdr = (WsHeader*)ws;
  unsigned* hist = (unsigned*)(ws + ws_hist_off());
  PartialSums partials;
  partials.sums = (double2*)(ws + ws_part_off());
  partials.counts = (uint2*)(partials.sums + (size_t)MAX_GRID * MAX_SLOTS);
  float* cos_cols = own_columns ? (float*)(ws + ws_total()) : block_cos_dev;
  float* sse_cols = own_columns ? (float*)(ws + ws_total() + col_bytes) : block_sse_dev;

  // everything that can refuse the call is decided before the first enqueue
  constexpr size_t SMEM_MAX = 226 * 1024;   // 227 KB per CTA minus the kernels' few static bytes
  int max_np = 0;
  for (int g = 0; g < P.n_groups; ++g) max_np = P.groups[g].np > max_np ? P.groups[g].np : max_np;
  constexpr size_t RED_SMEM_MAX = 220 * 1024;
  const size_t smem = sweep_layout(A, &P, SMEM_MAX);
  if (smem > SMEM_MAX) return SOP_ERR_ALPHABET;
  const int sms = num_sms();
  // persistent grid: one CTA per SM, fewer when the layer is small; at least enough threads for one row
  // (a small layer is spread over all of them: its CTAs build the tables with all their threads and evaluate with tba)
  long long tba = ((L.NB + sms - 1) / sms + 31) / 32 * 32;
  if (tba > TB) tba = TB;
  long long grid = (L.NB + tba - 1) / tba;
  const long long resident = (long long)sms * (max_np == 0 ? 2 : 1);
  if (grid > resident) grid = resident;
  const long long min_grid = (L.nbk + tba - 1) / tba;
  if (grid < min_grid) grid = min_grid;
  if (grid > MAX_GRID) return SOP_ERR_SHAPE;
  // the reduction: up to fifteen bundles per launch; persistent grid over its tiles.  16-byte copies need 16-byte aligned column starts and runs: a block count that is a multiple of four.
  BundleList bundles;
  build_bundles(Rp, &bundles);
  const int n_launch = bundles.n ? (bundles.n + MAX_BUNDLES - 1) / MAX_BUNDLES : 1;
  const bool vec = (L.NB % 4) == 0 && (((uintptr_t)cos_cols | (uintptr_t)sse_cols) & 15u) == 0;
  int units = 0;
  const long long rgrid = reduce_grid(L.NB, sms, &units);

  // the prepass adds to its histograms; the reduction's counters are cleared by the sweep where there is one
  if (!k_from_result && !reuse_prepass) SOP_CUDA_TRY(clear(ws, ws_part_off(), st));
  else if (!eval_mask) SOP_CUDA_TRY(clear(ws, ws_hist_off(), st));
  if ((rc = profile_mark(SOP_PROFILE_PREPASS, 0, st))) return rc;
  if (reuse_prepass) {
    SOP_CUDA_TRY(launch(kselect_kernel, 1, 256, 0, st, P, F, hist, hdr));
    SOP_CUDA_TRY(cudaGetLastError());
  } else if (!k_from_result) {
    // one read of W: block scales' exponent histogram, max|W|, then the shifts (last CTA)
    // (as many whole rows as four CTAs per SM have threads for)
    const long long fit = (long long)sms * 4 * PPB / L.nbk;
    const unsigned prows = (unsigned)(fit < 1 ? 1 : fit < M ? fit : M);
    const int pgrid = (int)((prows * L.nbk + PPB - 1) / PPB);
    SOP_CUDA_TRY(launch(prepass_kernel, pgrid, PPB, 0, st, L, P, F, hist, hdr, prows));
    SOP_CUDA_TRY(cudaGetLastError());
  }
  if ((rc = profile_mark(SOP_PROFILE_PREPASS, 1, st))) return rc;
  DeviceFacts* facts = device_facts();
  if (!facts->search_attr_set) {
    SOP_CUDA_TRY(cudaFuncSetAttribute(sweep_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(sweep_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(sweep_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(sweep_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(sweep_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(reduce_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RED_SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(reduce_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RED_SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(reduce_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RED_SMEM_MAX));
    SOP_CUDA_TRY(cudaFuncSetAttribute(reduce_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RED_SMEM_MAX));
    facts->search_attr_set = true;
  }
  if ((rc = profile_mark(SOP_PROFILE_SWEEP, 0, st))) return rc;
  if (eval_mask) {
    const unsigned c_off = (unsigned)(smem - SWEEP_C_BYTES);
#define SOP_LAUNCH_SWEEP(NP) SOP_CUDA_TRY(launch(sweep_kernel<NP>, grid, TB, smem, st, L, P, A, F, hdr, cos_cols, sse_cols, prev_result_dev, c_off, (unsigned)tba))
    if (max_np == 0) SOP_LAUNCH_SWEEP(0);
    else if (max_np == 1) SOP_LAUNCH_SWEEP(1);
    else if (max_np == 2) SOP_LAUNCH_SWEEP(2);
    else if (max_np == 3) SOP_LAUNCH_SWEEP(3);
    else SOP_LAUNCH_SWEEP(4);
#undef SOP_LAUNCH_SWEEP
    SOP_CUDA_TRY(cudaGetLastError());
  }
  if ((rc = profile_mark(SOP_PROFILE_SWEEP, 1, st))) return rc;
  if ((rc = profile_mark(SOP_PROFILE_REDUCE, 0, st))) return rc;
  const bool sel_err = (flags & SOP_SEARCH_SELECT_MSE) != 0;
  for (int l = 0; l < n_launch; ++l) {
    const int b0 = l * MAX_BUNDLES, nb = bundles.n - b0 < MAX_BUNDLES ? bundles.n - b0 : MAX_BUNDLES;
    BundlesDev Q;
    deal_bundles(bundles.b + b0, nb, &Q);
    int n_stage = g_reduce_ring ? MAX_STAGE : 2;             // (sixteen columns: two buffers of 98 KB)
    while (n_stage > 2 && reduce_smem_bytes(Q.n_cols, units, n_stage) > RED_SMEM_MAX) --n_stage;
    const size_t rs = reduce_smem_bytes(Q.n_cols, units, n_stage);
    const int fin = l == n_launch - 1 ? 1 : 0;
#define SOP_LAUNCH_REDUCE(SE, VC)                                                                                                   \
  SOP_CUDA_TRY(launch(reduce_kernel<SE, VC>, rgrid, RTB, rs, st, L, Rp, Q, units, n_stage, fin, hdr, partials, cos_cols, sse_cols, pair_table_dev, \
                                                     signed_table_dev, result_dev, prev_result_dev))
    if (sel_err) { if (vec) SOP_LAUNCH_REDUCE(true, true); else SOP_LAUNCH_REDUCE(true, false); }
    else { if (vec) SOP_LAUNCH_REDUCE(false, true); else SOP_LAUNCH_REDUCE(false, false); }
#undef SOP_LAUNCH_REDUCE
    SOP_CUDA_TRY(cudaGetLastError());
  }
  if ((rc = profile_mark(SOP_PROFILE_REDUCE, 1, st))) return rc;
  return SOP_OK;
}

}  // extern "C"
