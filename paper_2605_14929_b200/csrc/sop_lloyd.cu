// sop_dd4_lloyd: per-layer data-derived codebook (DD-n) by Lloyd iteration on the pool of blocks
// that the primary codebook reconstructs worst.
//
//   lloyd_init_kernel     clears the header, max(c), the shift k, the initial table (FMTa, reversed and negated if
//                         FMTa is a negated atom) as the first iteration's descriptor.
//   select_kernel<PASS>   three-pass radix select (11 + 11 + 10 bits) of the pool_rank-th worst block by
//                         its ranking key (cosine ascending, or error descending); each pass finds the bin
//                         of the previous histogram with a CTA-wide scan.  Not run when the
//                         caller fixes the pool threshold.
//   pool_list_kernel      threshold key from the last histogram (or from the given threshold); compacts the indices of the pool
//                         blocks into a dense list; the per-channel weight table omega = c / max(c) (or 1).
//   pool_cache_kernel     the pool elements never change between iterations, only the table does:
//                         (u, omega) of every pool element is computed once (u = w / scale) and kept
//                         in tiles of 6144 elements, each counting-sorted by the cell of u on a
//                         uniform grid (641 cells of width 2^-8); the start of every cell inside
//                         every tile is kept too, and per cell, over the whole pool, the int64
//                         fixed-point sums of omega and omega u and the moments of omega
//                         about the cell's centre.
//   lloyd_iter_kernel     the iterations.  A cell that holds no decision threshold of
//                         the current table lies inside one entry's interval: its elements are
//                         accounted for by the cell's sums and moments, without touching them.  Only
//                         the cells that hold a threshold are walked element by element, exactly.
//                         Per-entry sums are int64 fixed point (exactly associative: the table is the
//                         same bit for bit as a sequential sum over all elements gives), distortion
//                         FP64.  All iterations run in one cooperative launch, with a bounded wait for
//                         everybody's sums between them, or one per launch where the grid cannot be
//                         resident at once.
#include <math.h>
#include <stddef.h>
#include <string.h>

#include "sop_device.cuh"

namespace sop {

constexpr int LTB = 256;
constexpr int INIT_TB = 1024;
constexpr int SOP_MAX_LLOYD_ITERS = 64;
constexpr int SORT_CHALF = 320;                 // lookup grid on u: cell width 2^-8, rows cover |u| <= 1.25,
constexpr int SORT_ROWS = 2 * SORT_CHALF + 1;   // the first and last row take everything beyond
constexpr float SORT_INVH = 256.0f;
constexpr float SORT_MAGIC = 12582912.0f;       // 1.5 * 2^23

struct CellEntry { float thr; unsigned codes; };   // codes: lo | hi << 8; 0xFFFF: more than one threshold in the cell

// Everything an iteration reads about the current table, contiguous so that a CTA fetches it with one
// load per thread: the table (padded with its last entry), the exact decision thresholds (+inf padded)
// and the lookup cell of every threshold (ascending, like the thresholds).
struct IterDesc {
  int n_entries;
  int pad[3];
  float lut[SOP_MAX_ENTRIES];
  float tau[SOP_MAX_ENTRIES];
  int thr_cell[SOP_MAX_ENTRIES];
};

struct LloydWs {
  // radix select state
  unsigned hist[3][2048];
  // iteration state
  // per entry: sum fix(omega); sum of the low words of the CTAs' sums fix(omega u); of their high words.  Each with the number of
  // CTAs that have added theirs in its top byte (persistent iterations)
  unsigned long long acc[SOP_MAX_LLOYD_ITERS + 1][3][SOP_MAX_ENTRIES];
  double accD[SOP_MAX_LLOYD_ITERS + 1];
  unsigned prefix[3];       // of the selected key after one, two passes
  unsigned pad3;
  long long rank[3];        // its rank inside that prefix
  unsigned arrive[SOP_MAX_LLOYD_ITERS + 1];      // CTAs that have added their sums of an iteration (persistent iterations: of all of them)
  unsigned error;        // a CTA gave up waiting for a flag
  unsigned list_count;   // blocks appended to the pool list
  // per cell, over the whole pool (filled once by pool_cache_kernel)
  unsigned long long cellN[SORT_ROWS];     // sum fix(omega)
  long long cellS[SORT_ROWS];              // sum fix(omega u)
  double cellA[3][SORT_ROWS];              // sum omega, sum omega d, sum omega d^2, d = 256 u - (number of the cell's centre)
  long long cellQ[SORT_ROWS];              // sum fix((omega u) u): the exact second moment the grid-constrained construction needs
  // from here on set by lloyd_init_kernel
  alignas(16) float cmax;
  int k;
  int fmta;
  // the current codebook, rewritten by whoever changes it (set-up, then each update)
  IterDesc desc;
  // neither: where the last run starts per (number of runs, last cell) of the dynamic programme
  short dp_cut[SOP_MAX_ENTRIES][SORT_ROWS];
};

struct LloydArgs {
  const uint16_t* W;
  const float* c;
  const float* cosrow_base;   // [n_atoms x NB]
  long long M, K, ldw, nbk, NB;
  long long pool_rank;
  int k_mode, fmta_index, n_atoms;
  int flags;                  // SOP_LLOYD_*
  float pool_threshold;       // with SOP_LLOYD_POOL_THRESHOLD
  float* omega;               // workspace: K floats, c / max(c)
  unsigned* pool_idx;         // workspace: NB words, indices of the pool blocks
  uint2* cache;               // workspace: pairs (u, omega) as bit patterns, tiles of TILE_ELEMS sorted by cell
  unsigned short* tile_start; // workspace: [tiles][TS_PITCH] first sorted position of every cell in every tile
};

static size_t lloyd_off_dp() { return (sizeof(LloydWs) + 255) & ~(size_t)255; }
static size_t lloyd_dp_bytes();
static size_t lloyd_off_omega() { return lloyd_off_dp() + lloyd_dp_bytes(); }
static size_t lloyd_off_idx(long long K) { return lloyd_off_omega() + (((size_t)K * 4 + 255) & ~(size_t)255); }
static size_t lloyd_off_cache(long long M, long long K) { return lloyd_off_idx(K) + ((((size_t)M * (size_t)(K / SOP_G)) * 4 + 255) & ~(size_t)255); }
constexpr int CTB = 384;                        // threads of a cache CTA = pool blocks of a cache tile
constexpr int TILE_ELEMS = CTB * SOP_G;         // pool elements per cache tile
constexpr int TS_PITCH = (SORT_ROWS + 1 + 7) / 8 * 8;     // cell starts of a tile, whole 16-byte groups
static size_t lloyd_off_tiles(long long M, long long K) {
  const size_t nb = (size_t)M * (size_t)(K / SOP_G);
  return lloyd_off_cache(M, K) + ((nb + CTB - 1) / CTB) * TILE_ELEMS * sizeof(uint2);   // whole tiles
}
static size_t lloyd_ws_bytes(long long M, long long K) {
  const size_t nb = (size_t)M * (size_t)(K / SOP_G);
  return lloyd_off_tiles(M, K) + ((((nb + CTB - 1) / CTB) * TS_PITCH * sizeof(unsigned short) + 255) & ~(size_t)255);
}

__device__ __forceinline__ unsigned cos_key(float x) {
  const unsigned b = __float_as_uint(__fadd_rn(x, 0.0f));   // -0 -> +0
  return b ^ ((b >> 31) ? 0xFFFFFFFFu : 0x80000000u);
}
// Ranking key of a block: ascending key = worst block first.  By cosine the worst is the smallest value,
// by error (SOP_LLOYD_POOL_BY_ERROR) the largest.
__device__ __forceinline__ unsigned pool_key(float x, int flags) {
  const unsigned k = cos_key(x);
  return (flags & SOP_LLOYD_POOL_BY_ERROR) ? ~k : k;
}

__device__ __forceinline__ int resolve_fmta(const LloydArgs& a, const sop_search_result* res) {
  int f = a.fmta_index == SOP_FMTA_FROM_RESULT ? res->best_single : a.fmta_index;
  return max(0, min(a.n_atoms - 1, f));
}

// CTA of LTB threads: the bin of `hist` (LTB PER bins) holding the element of 1-based rank `rank`; *before = elements in lower bins.
// Every CTA of the pass that follows does this before it can start, so a thread's bins are loaded together.
template <int PER>
__device__ void find_bin(const unsigned* hist, long long rank, int* bin, long long* before) {
  __shared__ unsigned s_warp[LTB / 32];
  __shared__ int s_bin;
  __shared__ unsigned s_before;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned h[PER], local = 0;                        // (at most 2^27 blocks)
#pragma unroll
  for (int i = 0; i < PER; i += 4) {
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(hist + tid * PER + i));
    h[i] = v.x; h[i + 1] = v.y; h[i + 2] = v.z; h[i + 3] = v.w;
  }
#pragma unroll
  for (int i = 0; i < PER; ++i) local += h[i];
  unsigned incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  unsigned run = incl - local;
#pragma unroll
  for (int w = 0; w < LTB / 32; ++w) run += w < warp ? s_warp[w] : 0u;
  const unsigned want = (unsigned)rank;
  if (run < want && want <= run + local) {
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      if (run < want && want <= run + h[i]) { s_bin = tid * PER + i; s_before = run; }
      run += h[i];
    }
  }
  __syncthreads();
  *bin = s_bin; *before = s_before;
  __syncthreads();
}

// Whole CTA, after `passes` >= 1 passes: the prefix of the selected key from the histogram of the last pass; the passes before it
// have left theirs in the workspace, and the first CTA leaves this one.
__device__ unsigned derive_prefix(LloydWs* ws, long long pool_rank, int passes) {
  const int p = passes - 1;
  const unsigned pre = p ? __ldcg(&ws->prefix[p - 1]) : 0u;
  const long long rank = p ? __ldcg(&ws->rank[p - 1]) : pool_rank;
  int bin;
  long long before;
  if (p < 2) find_bin<2048 / LTB>(ws->hist[p], rank, &bin, &before);
  else find_bin<1024 / LTB>(ws->hist[p], rank, &bin, &before);
  const unsigned out = (pre << (p < 2 ? 11 : 10)) | (unsigned)bin;
  if (blockIdx.x == 0 && threadIdx.x == 0) { ws->prefix[p] = out; ws->rank[p] = rank - before; }
  return out;
}

template <int PASS>
__global__ void __launch_bounds__(LTB) select_kernel(LloydArgs a, const sop_search_result* res, LloydWs* ws) {
  pdl_trigger();
  pdl_wait();
  __shared__ unsigned sh[2048];
  for (int i = threadIdx.x; i < 2048; i += LTB) sh[i] = 0;
  unsigned prefix = 0;
  if (PASS > 0) prefix = derive_prefix(ws, a.pool_rank, PASS);
  __syncthreads();
  const float* row = a.cosrow_base + (size_t)resolve_fmta(a, res) * a.NB;
  auto count = [&](float x) {
    const unsigned key = pool_key(x, a.flags);
    if (PASS == 0) atomicAdd(&sh[key >> 21], 1u);
    else if (PASS == 1) { if ((key >> 21) == prefix) atomicAdd(&sh[(key >> 10) & 2047u], 1u); }
    else { if ((key >> 10) == prefix) atomicAdd(&sh[key & 1023u], 1u); }
  };
  // sixteen keys per thread and round, their loads in flight together (the pass is bound by memory latency otherwise):
  // four 128-bit loads where the row is 16-byte aligned, else four rounds of four single loads
  const long long stride = (long long)gridDim.x * LTB;
  const long long nv = (reinterpret_cast<uintptr_t>(row) & 15u) == 0 ? a.NB / 4 : 0;      // whole float4 groups
  for (long long i = (long long)blockIdx.x * LTB + threadIdx.x; i < nv; i += 4 * stride) {
    float4 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = i + q * stride < nv ? *(reinterpret_cast<const float4*>(row) + i + q * stride) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (i + q * stride >= nv) break;
      count(v[q].x); count(v[q].y); count(v[q].z); count(v[q].w);
    }
  }
  for (long long i = 4 * nv + (long long)blockIdx.x * LTB + threadIdx.x; i < a.NB; i += 4 * stride) {
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = i + q * stride < a.NB ? row[i + q * stride] : 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (i + q * stride >= a.NB) break;
      count(v[q]);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2048; i += LTB)
    if (sh[i]) atomicAdd(&ws->hist[PASS][i], sh[i]);
}

__device__ __forceinline__ int sort_cell(float u) {
  const float t = fminf(fmaxf(__fmaf_rn(u, SORT_INVH, SORT_MAGIC + (float)SORT_CHALF), SORT_MAGIC), SORT_MAGIC + (float)(2 * SORT_CHALF));
  return (int)(__float_as_uint(t) - __float_as_uint(SORT_MAGIC));
}

__device__ void make_desc(IterDesc* d, const float* table, int ne);

// CTA 0: max(c) and what the first table needs; the others clear the header.
__global__ void __launch_bounds__(INIT_TB) lloyd_init_kernel(LloydArgs a, AtomsDev A, const sop_search_result* res,
                                                             LloydWs* ws, double* distortion, int iters) {
  __shared__ float red[INIT_TB / 32];
  __shared__ float s_lut[SOP_MAX_ENTRIES];
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x;
  if (blockIdx.x != 0) {
    // everything that kernels add to, up to the values that CTA 0 writes
    uint4* h = reinterpret_cast<uint4*>(ws);
    const int n = (int)(offsetof(LloydWs, cmax) / sizeof(uint4));
    for (int i = (int)(blockIdx.x - 1) * INIT_TB + tid; i < n; i += (int)(gridDim.x - 1) * INIT_TB) h[i] = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  float mx = 0.0f;
  for (long long i = tid; i < a.K; i += INIT_TB) mx = fmaxf(mx, a.c[i]);
  for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
  if ((tid & 31) == 0) red[tid >> 5] = mx;
  const int f = resolve_fmta(a, res), ne = A.atoms[f].n_entries;
  if (tid < SOP_MAX_ENTRIES) {
    const int j = min(tid, ne - 1), src = A.atoms[f].negated ? ne - 1 - j : j;       // padded with the last entry
    float v = ((A.dd_mask >> f) & 1u) ? A.dd_lut[src] : A.atoms[f].lut[src];
    if (A.atoms[f].negated) v = -v;
    s_lut[tid] = v;
  }
  __syncthreads();
  if (tid < 32) {
    float t = red[tid];
    for (int o = 16; o; o >>= 1) t = fmaxf(t, __shfl_xor_sync(0xFFFFFFFFu, t, o));
    make_desc(&ws->desc, s_lut, ne);
    if (tid == 0) {
      ws->cmax = t;
      ws->fmta = f;
      ws->k = a.k_mode == SOP_K_FROM_RESULT ? res->k[f] : a.k_mode;
      // "not finished": the closing iteration overwrites it with the final distortion (never negative)
      distortion[iters] = -1.0;
    }
  }
}

// Dense list of the pool blocks.  A warp takes 512 consecutive blocks per round (four 128-bit loads per lane in flight, each a
// contiguous half kilobyte of the row, where it is 16-byte aligned); the counts of a lane's four groups of four are scanned
// together as bytes of one word.  The CTA's count goes to the list's counter once per round; the indices are laid out in shared
// memory and leave in whole lines.  The order of the list depends on the scheduling of the CTAs; nothing downstream depends on it
// (integer sums, and FP64 sums compared with a tolerance).
constexpr int LIST_ROUND = (LTB / 32) * 512;
__global__ void __launch_bounds__(LTB) pool_list_kernel(LloydArgs a, LloydWs* ws) {
  __shared__ unsigned s_cnt[LTB / 32 + 1];
  __shared__ unsigned s_base;
  __shared__ unsigned s_idx[LIST_ROUND];
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned tau_key = (a.flags & SOP_LLOYD_POOL_THRESHOLD) ? pool_key(a.pool_threshold, a.flags)      // the caller fixes the threshold
                                                                : derive_prefix(ws, a.pool_rank, 3);
  {
    const float cmax = ws->cmax;
    for (long long i = (long long)blockIdx.x * LTB + tid; i < a.K; i += (long long)gridDim.x * LTB)
      a.omega[i] = (a.flags & SOP_LLOYD_UNIFORM_WEIGHTS) ? 1.0f : (cmax > 0.0f ? __fdiv_rn(a.c[i], cmax) : 0.0f);
  }
  const float* row = a.cosrow_base + (size_t)ws->fmta * a.NB;
  const bool vec = (reinterpret_cast<uintptr_t>(row) & 15u) == 0;
  for (long long base = (long long)blockIdx.x * LIST_ROUND; base < a.NB; base += (long long)gridDim.x * LIST_ROUND) {
    const long long i0 = base + warp * 512 + 4 * lane;
    unsigned in = 0;                     // bit 4 q + b: block i0 + 128 q + b
    if (vec && base + warp * 512 + 512 <= a.NB) {
      float4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = *reinterpret_cast<const float4*>(row + i0 + 128 * q);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        in |= (pool_key(v[q].x, a.flags) <= tau_key ? 1u : 0u) << (4 * q);
        in |= (pool_key(v[q].y, a.flags) <= tau_key ? 1u : 0u) << (4 * q + 1);
        in |= (pool_key(v[q].z, a.flags) <= tau_key ? 1u : 0u) << (4 * q + 2);
        in |= (pool_key(v[q].w, a.flags) <= tau_key ? 1u : 0u) << (4 * q + 3);
      }
    } else {
      float v[16];                       // (in flight together as well)
#pragma unroll
      for (int x = 0; x < 16; ++x) {
        const long long i = i0 + 128 * (x >> 2) + (x & 3);
        v[x] = i < a.NB ? row[i] : 0.0f;
      }
#pragma unroll
      for (int x = 0; x < 16; ++x)
        if (i0 + 128 * (x >> 2) + (x & 3) < a.NB && pool_key(v[x], a.flags) <= tau_key) in |= 1u << x;
    }
    unsigned mine = 0;                   // a lane's four counts, a byte each (a warp's sum is at most 128)
#pragma unroll
    for (int q = 0; q < 4; ++q) mine |= (unsigned)__popc((in >> (4 * q)) & 15u) << (8 * q);
    unsigned incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += v;
    }
    const unsigned tot = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - mine;
    if (lane == 0) s_cnt[warp] = (tot & 255u) + ((tot >> 8) & 255u) + ((tot >> 16) & 255u) + (tot >> 24);
    __syncthreads();
    unsigned at = 0, all = 0;
#pragma unroll
    for (int w = 0; w < LTB / 32; ++w) { const unsigned c = s_cnt[w]; at += w < warp ? c : 0u; all += c; }
    if (tid == 0) s_base = all ? atomicAdd(&ws->list_count, all) : 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      unsigned p = at + ((excl >> (8 * q)) & 255u);
      at += (tot >> (8 * q)) & 255u;
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if ((in >> (4 * q + b)) & 1u) s_idx[p++] = (unsigned)(i0 + 128 * q + b);
    }
    __syncthreads();
    const unsigned to = s_base;
    for (unsigned x = tid; x < all; x += LTB) a.pool_idx[to + x] = s_idx[x];
    __syncthreads();             // s_cnt, s_base and s_idx are rewritten in the next round
  }
}

// One tile = the CTB pool blocks (TILE_ELEMS elements) of one CTA pass.  The tile is counting-sorted by
// cell in shared memory.  Sorted position p is stored at slot (p & ~15) | ((p ^ (p >> 4)) & 15): the elements of a
// cell stay next to each other in memory (an iteration reads the split cells' runs, a few 32-byte sectors each,
// instead of one sector per element), and the thread that sums positions 16 t .. 16 t + 15 of the tile in shared
// memory meets no bank conflict (the slots of one step differ in their low four bits over a half-warp).  The
// exclusive-or keeps a group of four consecutive positions inside one 32-byte sector.
// A tile that the pool does not fill is padded with (u, omega) = (0, 0): such elements add nothing.
__device__ __forceinline__ unsigned tile_slot(unsigned p) { return (p & ~15u) | ((p ^ (p >> 4)) & 15u); }
__device__ __forceinline__ long long fix24(float v) {   // llrint(v * 2^24): exact scaling, one rounding to an integer
  const float s = __fmul_rn(v, 16777216.0f);
  return fabsf(s) < 2147483648.0f ? (long long)__float2int_rn(s) : __float2ll_rn(s);
}

constexpr int CELL_SPILL_TILES_MAX = 128;     // cache tiles a CTA sorts between two transfers of its per-cell sums to the global ones (any number is safe)
constexpr int TILES_PER_WARP_MAX = 4;         // range of a reserved tuning argument

// Launch-shape parameters of the pool cache and of the iteration grid; sop_dd4_lloyd_tuning lowers them (tests reach the
// mid-loop transfer and CTAs with many tiles on small layers that way).  Results do not depend on them.
struct LloydTune { int spill_tiles, cache_ctas, iter_ctas; };
static LloydTune g_tune = {CELL_SPILL_TILES_MAX, 0, 0};

// Sums of a run (at most 16 elements of one cell, |u| <= WIDE_U): fix(omega) below 2^29, fix(omega u) below 2^30 in magnitude, and
//   Lloyd: the moments sum omega, sum omega d, sum omega d^2 of the distance d = 256 u - (number of the cell's centre);
//   DP: fix(omega u u), exact, in the bits of m0.
// Kept as arrays: the runs that neighbouring threads store go to neighbouring cells.
template <int N> struct RunArrays { int2 ns[N]; double m0[N], m1[N], m2[N]; };
constexpr float WIDE_U = 2.0f;                   // blocks with a larger |u| (a scale that saturated) make their tile a wide one

struct CacheSmem {
  uint2 stage[TILE_ELEMS];
  unsigned hist[2][SORT_ROWS + 3];               // per cell: count, then first sorted position; of this tile and the next
  // runs: [0, CTB) the threads' first ones, then by cell a thread's other ones (no two threads have the same cell among them)
  RunArrays<CTB + SORT_ROWS> run;
  unsigned long long accN[SORT_ROWS];            // this CTA's per-cell sums
  long long accS[SORT_ROWS];
  double accA[3][SORT_ROWS];
  unsigned warp_tot[CTB / 32];
};

// Whole CTA, after a barrier: the CTA's sums are added to the per-cell sums of the pool and cleared.
template <bool DP>
__device__ void spill_cells(CacheSmem& S, LloydWs* ws) {
  for (int r = threadIdx.x; r < SORT_ROWS; r += CTB) {
    if (S.accN[r]) atomicAdd(&ws->cellN[r], S.accN[r]);
    if (S.accS[r]) atomicAdd(reinterpret_cast<unsigned long long*>(&ws->cellS[r]), (unsigned long long)S.accS[r]);
    S.accN[r] = 0; S.accS[r] = 0;
    if (DP) {
      const long long q = __double_as_longlong(S.accA[0][r]);
      if (q) atomicAdd(reinterpret_cast<unsigned long long*>(&ws->cellQ[r]), (unsigned long long)q);
      S.accA[0][r] = 0.0;
    } else {
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        if (S.accA[x][r] != 0.0) atomicAdd(&ws->cellA[x][r], S.accA[x][r]);
        S.accA[x][r] = 0.0;
      }
    }
  }
}

// What bounds it: shared-memory wavefronts (80 % busy): the sort's scattered accesses and the runs' sums.  A tile's weights are loaded
// while the tile before it is summed (the kernel waited for them for a third of its time), the sums run without divergence -- a run is
// stored when the next one begins, and the owner of a cell collects its runs afterwards -- and the sorted tile leaves by one
// asynchronous bulk copy.  8192 x 8192, half the blocks in the pool: 167 us (228 us with limb atomics per run, executed for one lane
// at a time); 28672 x 8192: 563 us (772 us).
template <bool DP>
__global__ void __launch_bounds__(CTB, 2) pool_cache_kernel(LloydArgs a, FmtDev F, LloydWs* ws, long long* pool_count_out,
                                                         unsigned spill_tiles) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(128) unsigned char cache_smem[];
  CacheSmem& S = *reinterpret_cast<CacheSmem*>(cache_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int r = tid; r < SORT_ROWS; r += CTB) { S.accN[r] = 0; S.accS[r] = 0; S.accA[0][r] = S.accA[1][r] = S.accA[2][r] = 0.0; }
  for (int i = tid; i < SORT_ROWS + 3; i += CTB) S.hist[0][i] = 0;
  const unsigned count = ws->list_count;
  const unsigned n_tiles = (count + CTB - 1) / CTB;
  const int k = ws->k;
  if (blockIdx.x == 0 && tid == 0) *pool_count_out = (long long)count;   // the list is complete: its length is the pool size
  const unsigned nbk = (unsigned)a.nbk;
  unsigned tiles_since_spill = 0;
  int cur = 0;
  // the weights of a tile are loaded one tile ahead, the list entries two
  uint4 wn0 = make_uint4(0u, 0u, 0u, 0u), wn1 = wn0;
  unsigned jn = 0, idx2 = 0;
  auto load_idx = [&](unsigned tile) { const unsigned i = tile * CTB + tid; return tile < n_tiles && i < count ? a.pool_idx[i] : 0xFFFFFFFFu; };
  auto load_w = [&](unsigned blk) {
    wn0 = wn1 = make_uint4(0u, 0u, 0u, 0u);
    jn = 0xFFFFFFFFu;
    if (blk != 0xFFFFFFFFu) {
      const unsigned m = blk / nbk;
      jn = blk - m * nbk;
      const uint4* p = reinterpret_cast<const uint4*>(a.W + (long long)m * a.ldw + (long long)jn * SOP_G);
      wn0 = *p; wn1 = p[1];
    }
  };
  load_w(load_idx(blockIdx.x));
  idx2 = load_idx(blockIdx.x + gridDim.x);
  __syncthreads();
  for (unsigned tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, cur ^= 1) {
    unsigned* hist = S.hist[cur];
    const uint32_t wb[8] = {wn0.x, wn0.y, wn0.z, wn0.w, wn1.x, wn1.y, wn1.z, wn1.w};
    float om[16];
    if (jn != 0xFFFFFFFFu) {
      const float4* op = reinterpret_cast<const float4*>(a.omega + (size_t)jn * SOP_G);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 o = op[q];
        om[4 * q] = o.x; om[4 * q + 1] = o.y; om[4 * q + 2] = o.z; om[4 * q + 3] = o.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 16; ++e) om[e] = 0.0f;
    }
    uint32_t mb = 0;       // the maximum of the sixteen 15-bit magnitude patterns, two per word at a time
#pragma unroll
    for (int q = 0; q < 8; ++q) mb = __vmaxu2(mb, wb[q] & 0x7FFF7FFFu);
    mb = max(mb & 0xFFFFu, mb >> 16);
    const float amax = __uint_as_float(mb << 16);
    const float s_hat = scale_quantize(amax, k, F).s_hat;    // a DD table declares tmax = 1
    const float rcp = s_hat > 0.0f ? __frcp_rn(s_hat) : 0.0f;
    unsigned where[16];   // cell << 16 | arrival number inside the cell
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float u = __fmul_rn((e & 1) ? bf16hi(wb[e >> 1]) : bf16lo(wb[e >> 1]), rcp);
      const unsigned c = (unsigned)sort_cell(u);
      where[e] = (c << 16) | atomicAdd(&hist[c], 1u);
    }
    const bool wide = __syncthreads_or(!(__fmul_rn(amax, rcp) <= WIDE_U)) != 0;
    // exclusive scan of the counts: two bins per thread
    {
      static_assert(2 * CTB >= SORT_ROWS + 1, "two bins per thread");
      const int b0 = 2 * tid;
      unsigned c0 = 0, c1 = 0;
      if (b0 < SORT_ROWS) { c0 = hist[b0]; c1 = hist[b0 + 1]; }        // (hist[SORT_ROWS] is zero)
      const unsigned local = c0 + c1;
      unsigned incl = local;
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane == 31) S.warp_tot[warp] = incl;
      if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");       // the tile before this one has left the stage
      __syncthreads();
      unsigned base = 0;
      for (int w = 0; w < warp; ++w) base += S.warp_tot[w];
      const unsigned excl = base + incl - local;
      if (b0 <= SORT_ROWS) { hist[b0] = excl; hist[b0 + 1] = excl + c0; }      // hist[SORT_ROWS] = TILE_ELEMS: the end of the last cell
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float u = __fmul_rn((e & 1) ? bf16hi(wb[e >> 1]) : bf16lo(wb[e >> 1]), rcp);
      const unsigned p = hist[where[e] >> 16] + (where[e] & 0xFFFFu);
      S.stage[tile_slot(p)] = make_uint2(__float_as_uint(u), __float_as_uint(om[e]));
    }
    load_w(idx2);
    idx2 = load_idx(tile + 2 * gridDim.x);
    if (!DP) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (!DP) {      // the dynamic programme reads the per-cell sums only: no iteration walks the elements again
      if (tid == 0) {
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                     ::"l"(a.cache + (size_t)tile * TILE_ELEMS), "r"((unsigned)__cvta_generic_to_shared(S.stage)), "r"((unsigned)(TILE_ELEMS * sizeof(uint2))) : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
      unsigned* ts = reinterpret_cast<unsigned*>(a.tile_start + (size_t)tile * TS_PITCH);
      if (2 * tid <= SORT_ROWS) ts[tid] = hist[2 * tid] | (hist[2 * tid + 1] << 16);
    }
    for (int i = tid; i < SORT_ROWS + 3; i += CTB) S.hist[cur ^ 1][i] = 0;
    if (!wide) {
      // thread t owns the sorted positions 16 t .. 16 t + 15 (ascending cells): run after run in registers
      int n = 0, s = 0, c_now = -1, q_sum = 0;
      double m0 = 0.0, m1 = 0.0, m2 = 0.0;
      int dst = tid;
      auto store = [&]() {
        S.run.ns[dst] = make_int2(n, s);
        if (DP) { S.run.m0[dst] = __longlong_as_double((long long)q_sum); }
        else { S.run.m0[dst] = m0; S.run.m1[dst] = m1; S.run.m2[dst] = m2; }
      };
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint2 v = S.stage[(unsigned)(16 * tid) + (unsigned)(i ^ (tid & 15))];
        const float u = __uint_as_float(v.x), w = __uint_as_float(v.y);
        const float t = fminf(fmaxf(__fmaf_rn(u, SORT_INVH, SORT_MAGIC + (float)SORT_CHALF), SORT_MAGIC), SORT_MAGIC + (float)(2 * SORT_CHALF));
        const int c = (int)(__float_as_uint(t) - __float_as_uint(SORT_MAGIC));
        const bool next = i > 0 && c != c_now;
        if (next) {
          store();
          dst = CTB + c;
        }
        c_now = c;
        const float w24 = __fmul_rn(w, 16777216.0f), ou24 = __fmul_rn(w24, u);   // omega u, rounded once, times 2^24
        n = (next ? 0 : n) + __float2int_rn(w24);                                // omega in [0, 1]
        s = (next ? 0 : s) + __float2int_rn(ou24);
        if (DP) {
          q_sum = (next ? 0 : q_sum) + __float2int_rn(__fmul_rn(ou24, u));
        } else {
          const double keep = next ? 0.0 : 1.0, wd = (double)w;
          const double d = (double)__fmaf_rn(u, SORT_INVH, __fsub_rn(SORT_MAGIC + (float)SORT_CHALF, t));      // 256 u - (c - 320): exact in a cell
          const double x = __dmul_rn(wd, d);
          m0 = __fma_rn(m0, keep, wd);
          m1 = __fma_rn(m1, keep, x);
          m2 = __fma_rn(m2, keep, __dmul_rn(x, d));
        }
      }
      store();
    }
    __syncthreads();
    // the owner of a cell adds up its runs: the run of the thread where it begins (its first one when the cell begins at the
    // thread's first position) and the first runs of the threads after that up to the one where it ends
    if (!wide) {
      for (int c = tid; c < SORT_ROWS; c += CTB) {
        const unsigned p0 = hist[c], p1 = hist[c + 1];
        if (p0 == p1) continue;
        const unsigned t0 = p0 >> 4, t1 = (p1 - 1) >> 4;
        const unsigned r = (p0 & 15u) == 0u ? t0 : (unsigned)(CTB + c);
        unsigned long long n = (unsigned)S.run.ns[r].x;
        long long s = S.run.ns[r].y, q = DP ? __double_as_longlong(S.run.m0[r]) : 0;
        double m0 = S.run.m0[r], m1 = DP ? 0.0 : S.run.m1[r], m2 = DP ? 0.0 : S.run.m2[r];
        for (unsigned t = t0 + 1; t <= t1; ++t) {
          n += (unsigned)S.run.ns[t].x; s += S.run.ns[t].y;
          if (DP) q += __double_as_longlong(S.run.m0[t]);
          else { m0 += S.run.m0[t]; m1 += S.run.m1[t]; m2 += S.run.m2[t]; }
        }
        S.accN[c] += n; S.accS[c] += s;
        if (DP) S.accA[0][c] = __longlong_as_double(__double_as_longlong(S.accA[0][c]) + q);
        else { S.accA[0][c] += m0; S.accA[1][c] += m1; S.accA[2][c] += m2; }
      }
    } else {
      // a wide tile: element by element in 64 bits, straight to the global sums
#pragma unroll 1
      for (int i = 0; i < 16; ++i) {
        const uint2 v = S.stage[(unsigned)(16 * tid) + (unsigned)(i ^ (tid & 15))];
        const float u = __uint_as_float(v.x), w = __uint_as_float(v.y);
        if (w == 0.0f) continue;
        const int c = sort_cell(u);
        const float ou = fminf(fmaxf(__fmul_rn(w, u), -256.0f), 256.0f);
        atomicAdd(&ws->cellN[c], (unsigned long long)fix24(w));
        atomicAdd(reinterpret_cast<unsigned long long*>(&ws->cellS[c]), (unsigned long long)fix24(ou));
        if (DP) {
          atomicAdd(reinterpret_cast<unsigned long long*>(&ws->cellQ[c]), (unsigned long long)fix24(__fmul_rn(ou, u)));
        } else {
          const double d = (double)u * 256.0 - (double)(c - SORT_CHALF);
          atomicAdd(&ws->cellA[0][c], (double)w);
          atomicAdd(&ws->cellA[1][c], (double)w * d);
          atomicAdd(&ws->cellA[2][c], (double)w * d * d);
        }
      }
    }
    if (++tiles_since_spill == spill_tiles) {
      spill_cells<DP>(S, ws);               // (a thread clears the cells it owns)
      tiles_since_spill = 0;
    }
  }
  if (tiles_since_spill) spill_cells<DP>(S, ws);
  if (tid == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------------------------------------
// The iterations.  A cell that holds a threshold of the current table ("split cell") is walked element by element; every other
// cell lies inside one entry's interval and is accounted for by its sums.
//   A CTA owns a contiguous range of cache tiles and keeps their cell starts in shared memory over all iterations.  A run is the
//   elements of one split cell in one tile; eight lanes take a run (neighbouring 8-byte elements), four tiles per warp and step,
//   the next step's elements are loaded ahead.  The warps take the runs cell by cell: the sums of a cell (all of it, and the part
//   above its threshold) stay in registers until the warp moves to the next cell, one to three times per iteration.
//   The cells without a threshold are a matter of CTA 0: prefix sums over all cells, built once, make an entry's share of the sums
//   the difference of two of them.  Their distortion comes from the moments about the cells' centres, a cell per thread: what
//   cancels is of the size of a cell, so elements that lie on their entries leave zero and rounding leaves nothing below it (with
//   differences of moments about the origin a layer of seven weight values ended at -2e-13).
//   Every CTA adds its sums to the iteration's global ones, waits (bounded) until all have and then works out the next table for
//   itself: the sums are integers, so all get the same one and nobody has to hand it on.  A sum carries the number of CTAs that have
//   added to it in its top byte, so that neither a fence nor an arrival stands between the additions and their readers.
// What bounds it: the chain of one iteration (the first elements, the sums, global additions, reading them back, table: about 3.7 us;
// 4.5 us with an arrival counter behind a fence, 9 us when the last CTA worked out the table and handed it on) and, for a large pool,
// the latency of the split cells' elements.  Nine iterations on 25 thousand pool blocks 41 us (49 us with the arrival counter, 82 us
// with a warp per tile), on 2 million 97 us (150 us), on 7.3 million 235 us (341 us).  Every warp must have its share of every cell:
// dealt cell by cell, the warps of the outer thresholds waited for those of the inner ones and the 7.3 million took 685 us.
// ---------------------------------------------------------------------------------------------
constexpr int ITB = 768;            // threads of an iteration CTA (one per SM)
constexpr int PRE = 4;              // elements of a run that a lane loads one step ahead
constexpr int MAX_SPLIT = 32;       // a table has at most 31 thresholds, so at most 31 cells hold one
constexpr int LIMBS = 3;            // 64-bit sums modulo 2^64 as 20 + 20 + 24 bits, which native 32-bit shared-memory additions take
constexpr int CTA_COUNT_BIT = 56;   // fewer than 2^27 blocks: a sum of omega stays below 2^55 (see lloyd_iteration_plan)
constexpr unsigned WAIT_POLLS = 1u << 21;      // polls of a few hundred ns: about half a second

struct IterSmem {
  IterDesc d;
  unsigned limb[2][LIMBS][SOP_MAX_ENTRIES];    // this CTA's sums per entry: fix(omega), fix(omega u)
  unsigned long long sum[2][SOP_MAX_ENTRIES];  // the same of cells with several thresholds
  double lane_D[ITB];
  CellEntry entry[MAX_SPLIT];
  unsigned short cell[MAX_SPLIT];
  int n_split, stop, is_last;
  float table[SOP_MAX_ENTRIES];
  // CTA 0: sums over the cells before r
  unsigned long long preN[SORT_ROWS + 1];
  long long preS[SORT_ROWS + 1];
};

// CTA 0: the moments of the thread's cell.
struct CellMoments { double a0, a1, a2; };

// sum omega (u - q)^2 of the cell, q the entry that its elements belong to; zero for a cell that is walked element by element.
__device__ __forceinline__ double cell_distortion(const IterDesc& d, const CellMoments& m, int cell) {
  int j = 0;                                   // thresholds in lower cells (padded with SORT_ROWS from n_entries - 1 on)
#pragma unroll
  for (int step = 16; step >= 1; step >>= 1)
    if (d.thr_cell[j + step - 1] < cell) j += step;
  const double e = 256.0 * (double)d.lut[j] - (double)(cell - SORT_CHALF);
  const double t = m.a2 - e * (2.0 * m.a1 - e * m.a0);
  return d.thr_cell[j] == cell || t < 0.0 ? 0.0 : t * (1.0 / 65536.0);
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v, unsigned lanes = 0xFFFFFFFFu) {      // modulo 2^64, by 32-bit sums of 27-bit limbs
  const unsigned a = __reduce_add_sync(lanes, (unsigned)v & 0x7FFFFFFu), b = __reduce_add_sync(lanes, (unsigned)(v >> 27) & 0x7FFFFFFu),
                 c = __reduce_add_sync(lanes, (unsigned)(v >> 54));
  return (unsigned long long)a + ((unsigned long long)b << 27) + ((unsigned long long)c << 54);
}
__device__ __forceinline__ unsigned limb_of(unsigned long long v, int i) {
  return i == 0 ? (unsigned)v & 0xFFFFFu : i == 1 ? (unsigned)(v >> 20) & 0xFFFFFu : (unsigned)(v >> 40);
}
__device__ __forceinline__ unsigned long long join_limbs(IterSmem& S, int w, int code) {
  return (unsigned long long)S.limb[w][0][code] + ((unsigned long long)S.limb[w][1][code] << 20) + ((unsigned long long)S.limb[w][2][code] << 40);
}

// One warp: the cells that hold thresholds (thresholds ascend, so those of one cell are neighbours).
__device__ void split_cells(IterSmem& S) {
  const int lane = threadIdx.x & 31, ne = S.d.n_entries;
  const bool on = lane < ne - 1;
  const int c = S.d.thr_cell[lane];
  const int cp = __shfl_up_sync(0xFFFFFFFFu, c, 1), cn = __shfl_down_sync(0xFFFFFFFFu, c, 1);
  const bool first = on && (lane == 0 || cp != c);
  const bool single = lane == ne - 2 || cn != c;
  const unsigned fm = __ballot_sync(0xFFFFFFFFu, first);
  if (first) {
    const int idx = __popc(fm & ((1u << lane) - 1u));
    CellEntry e;
    e.thr = S.d.tau[lane];
    e.codes = single ? ((unsigned)lane | ((unsigned)(lane + 1) << 8)) : 0xFFFFu;
    S.cell[idx] = (unsigned short)c;
    S.entry[idx] = e;
  }
  if (lane == 0) S.n_split = __popc(fm);
}

// One warp: the descriptor of a table (entry j of the sorted table, padded with its last value, in lane j): the decision
// thresholds and their lookup cells.  sort_cell is monotone, so an element in a lower cell than a
// threshold's is below the threshold and one in a higher cell is above it: only the elements of the cells listed here need the
// comparison itself.
__device__ void make_desc(IterDesc* d, const float* table, int ne) {
  const int j = threadIdx.x & 31;
  const float t = table_threshold(table, j, ne);
  d->lut[j] = table[j];
  d->tau[j] = t;
  d->thr_cell[j] = j < ne - 1 ? sort_cell(t) : SORT_ROWS;
  if (j == 0) d->n_entries = ne;
}

// One warp: centroids one lane per entry, snapped to bf16, ascending (ties by index); leaves the new table in S.table.
__device__ void new_table(IterSmem& S, unsigned long long n, long long sv) {
  const int j = threadIdx.x & 31, ne = S.d.n_entries;
  float t = S.d.lut[j];                      // lanes from n_entries on hold the last entry's value
  if (j < ne && n) {
    const float cen = __double2float_rn(__ddiv_rn(__ll2double_rn(sv), __ull2double_rn(n)));
    uint32_t b = __float_as_uint(cen);
    b += 0x7FFFu + ((b >> 16) & 1u);
    b &= 0xFFFF0000u;                        // nearest bf16, ties to even
    t = __uint_as_float(b);
  }
  int rank = j;
  const float before = __shfl_up_sync(0xFFFFFFFFu, t, 1);
  if (__any_sync(0xFFFFFFFFu, j > 0 && j < ne && !(before <= t))) {      // (hardly ever: centroids of neighbouring intervals ascend)
    rank = 0;
#pragma unroll 1
    for (int k = 0; k < ne; ++k) {
      const float o = __shfl_sync(0xFFFFFFFFu, t, k);
      rank += o < t || (o == t && k < j) ? 1 : 0;
    }
  }
  if (j < ne) S.table[rank] = t;
  __syncwarp();
  const float top = S.table[ne - 1];
  if (j >= ne) S.table[j] = top;             // padded with the last entry
  __syncwarp();
}

// The whole CTA: adds its share of one iteration to the sums of that iteration and arrives.
template <bool ALL>
__device__ __forceinline__ void iteration_share(const LloydArgs& a, LloydWs* ws, IterSmem& S, const unsigned short* ts,
                                                const CellMoments& mom, unsigned tile0, int T, int it, bool last) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, sub = lane >> 3, ln = lane & 7;
  constexpr int NW = ITB / 32;
  const int n_split = S.n_split, Tc = (T + 3) / 4, total = n_split * Tc;
  double D = 0.0;
  // step x: cell x / Tc, tiles 4 (x % Tc) .. + 3; a warp takes every NW-th, so that each has its share of the cells with long runs
  int l = Tc ? warp / Tc : 0, ch = warp - l * Tc;
  unsigned p0 = 0, p1 = 0;
  uint2 v[PRE];
  const uint2* src = a.cache;
  auto open_run = [&](int x, int lx, int cx) {
    p0 = p1 = 0;
    const int t = 4 * cx + sub;
    if (x < total && t < T) {
      const unsigned short* row = ts + (size_t)t * TS_PITCH + S.cell[lx];
      p0 = row[0] + (unsigned)ln; p1 = row[1];
      src = a.cache + (size_t)(tile0 + (unsigned)t) * TILE_ELEMS;
    }
#pragma unroll
    for (int i = 0; i < PRE; ++i) v[i] = p0 + 8u * i < p1 ? src[tile_slot(p0 + 8u * i)] : make_uint2(0u, 0u);
  };
  open_run(warp, l, ch);
  if (blockIdx.x == 0 && tid < SORT_ROWS) D = cell_distortion(S.d, mom, tid);        // (the first elements are on their way)
  unsigned long long nA = 0, nH = 0;
  long long sA = 0, sH = 0;
#pragma unroll 1
  for (int x = warp; x < total; x += NW) {
    const CellEntry e = S.entry[l];
    const int c_now = S.cell[l], l_now = l;
    unsigned q = p0;
    const unsigned q1 = p1;
    uint2 w[PRE];
#pragma unroll
    for (int i = 0; i < PRE; ++i) w[i] = v[i];
    const uint2* from = src;
    ch += NW;
    while (ch >= Tc) { ch -= Tc; ++l; }
    open_run(x + NW, l, ch);
    // The end cells hold everything beyond the grid (any u), and a cell with several thresholds needs the general search.
    if (e.codes != 0xFFFFu && c_now != 0 && c_now != SORT_ROWS - 1) {
      const float qlo = S.d.lut[e.codes & 0xFFu], qhi = S.d.lut[e.codes >> 8];
#pragma unroll 1
      for (;;) {
        unsigned n = 0, nh = 0;
        int s = 0, sh = 0;
        // |u| <= 1.26: the four terms of a lane stay below 2^31.  An element that is not there reads as (0, 0): its omega is zero.
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
          const float u = __uint_as_float(w[i].x), om = __uint_as_float(w[i].y);
          const bool hi = u > e.thr;
          const float dd = __fsub_rn(u, hi ? qhi : qlo);
          D += (double)__fmul_rn(__fmul_rn(om, dd), dd);
          const float om24 = __fmul_rn(om, 16777216.0f);
          const unsigned ni = __float2uint_rn(om24);             // omega in [0, 1]
          const int si = __float2int_rn(__fmul_rn(om24, u));     // omega u, rounded once, times 2^24
          n += ni; s += si;
          if (hi) { nh += ni; sh += si; }
        }
        nA += n; nH += nh; sA += s; sH += sh;
        q += 8u * PRE;
        if (!__any_sync(0xFFFFFFFFu, q < q1)) break;
#pragma unroll
        for (int i = 0; i < PRE; ++i) w[i] = q + 8u * i < q1 ? from[tile_slot(q + 8u * i)] : make_uint2(0u, 0u);
      }
      if ((l != l_now || x + NW >= total) && !last) {
        const unsigned long long ta = warp_sum64(nA), th = warp_sum64(nH), ua = warp_sum64((unsigned long long)sA), uh = warp_sum64((unsigned long long)sH);
        if (lane < 4 * LIMBS) {
          const int side = lane / (2 * LIMBS), w2 = lane / LIMBS & 1, i = lane % LIMBS;      // below / above the threshold; n / s; limb
          const unsigned long long y = side ? (w2 ? uh : th) : (w2 ? ua - uh : ta - th);
          atomicAdd(&S.limb[w2][i][side ? e.codes >> 8 : e.codes & 0xFFu], limb_of(y, i));
        }
        nA = nH = 0; sA = sH = 0;
      }
    } else {
#pragma unroll 1
      for (; q < q1; q += 8u) {
        const uint2 y = from[tile_slot(q)];
        const float u = __uint_as_float(y.x), om = __uint_as_float(y.y);
        const int code = count_below(S.d.tau, u);
        const float dd = __fsub_rn(u, S.d.lut[code]);
        D += (double)__fmul_rn(__fmul_rn(om, dd), dd);
        if (!last) {
          const unsigned same = __match_any_sync(__activemask(), code);
          const unsigned long long tn = warp_sum64((unsigned long long)fix24(om), same);
          const unsigned long long ts = warp_sum64((unsigned long long)fix24(fminf(fmaxf(__fmul_rn(om, u), -256.0f), 256.0f)), same);
          if (lane == __ffs((int)same) - 1) { atomicAdd(&S.sum[0][code], tn); atomicAdd(&S.sum[1][code], ts); }
        }
      }
      __syncwarp();
    }
  }
  S.lane_D[tid] = D;
  __syncthreads();
  if (warp == 0) {
    const int ne = S.d.n_entries;
    unsigned long long n = join_limbs(S, 0, lane) + S.sum[0][lane], s = join_limbs(S, 1, lane) + S.sum[1][lane];
    // CTA 0: the cells without a threshold between this entry's two
    const int lo = blockIdx.x == 0 && lane < ne ? (lane ? S.d.thr_cell[lane - 1] + 1 : 0) : 0;
    const int hi = blockIdx.x == 0 && lane < ne ? (lane < ne - 1 ? S.d.thr_cell[lane] : SORT_ROWS) : 0;
    if (lo < hi) {
      n += S.preN[hi] - S.preN[lo];
      s += (unsigned long long)(S.preS[hi] - S.preS[lo]);
    }
    if (!last && lane < ne) {
      const unsigned long long one = ALL ? 1ull << CTA_COUNT_BIT : 0ull;
      atomicAdd(&ws->acc[it][0][lane], n + one);
      atomicAdd(&ws->acc[it][1][lane], (s & 0xFFFFFFFFull) + one);
      atomicAdd(&ws->acc[it][2][lane], (unsigned long long)((long long)s >> 32) + one);
    }
    // the rest happens while those are on their way
    S.sum[0][lane] = S.sum[1][lane] = 0ull;
#pragma unroll
    for (int i = 0; i < LIMBS; ++i) S.limb[0][i][lane] = S.limb[1][i][lane] = 0u;
    // (a shorter chain, four sums at a time, had the CTAs poll the sums while they were being added to: 1 us of a pass slower)
    double dsum = 0.0;
#pragma unroll 8
    for (int i = lane; i < ITB; i += 32) dsum += S.lane_D[i];
#pragma unroll
    for (int o = 16; o; o >>= 1) dsum += __shfl_xor_sync(0xFFFFFFFFu, dsum, o);
    if (lane == 0 && dsum != 0.0) atomicAdd(&ws->accD[it], dsum);
    if (!ALL || last) {
      __threadfence();
      __syncwarp();
      if (lane == 0) S.is_last = atomicAdd(&ws->arrive[it], 1u) == gridDim.x - 1 ? 1 : 0;
      __syncwarp();
    }
  }
}

// The sums of one iteration where they count their CTAs (one lane per entry): false while some are missing.
__device__ __forceinline__ bool read_sums(const unsigned long long (*acc)[SOP_MAX_ENTRIES], unsigned ctas, unsigned long long& n, long long& s) {
  const int lane = threadIdx.x & 31;
  unsigned long long v[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v[i]) : "l"(&acc[i][lane]) : "memory");
  const unsigned long long c0 = v[0] >> CTA_COUNT_BIT, c1 = v[1] >> CTA_COUNT_BIT, c2 = (v[2] + (1ull << (CTA_COUNT_BIT - 1))) >> CTA_COUNT_BIT;
  n = v[0] - (c0 << CTA_COUNT_BIT);
  s = (long long)((v[1] - (c1 << CTA_COUNT_BIT)) + ((v[2] - (c2 << CTA_COUNT_BIT)) << 32));      // modulo 2^64
  return c0 == ctas && c1 == ctas && c2 == ctas;
}

// ALL: every iteration in this launch (launched cooperatively: every CTA is resident); else iteration `it0` alone, whose last CTA
// leaves the next table in ws->desc for the next launch.
// The wait is bounded: a CTA that gives up raises ws->error, every CTA then leaves, and the last distortion entry stays -1 (a
// distortion is never negative) so that the caller can tell.
template <bool ALL>
__global__ void __launch_bounds__(ITB, 1) lloyd_iter_kernel(LloydArgs a, LloydWs* ws, double* distortion, int it0, int iters,
                                                           float* out_lut, int smem_tiles) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(16) unsigned char iter_smem[];
  IterSmem& S = *reinterpret_cast<IterSmem*>(iter_smem);
  unsigned short* s_ts = reinterpret_cast<unsigned short*>(iter_smem + ((sizeof(IterSmem) + 15) & ~(size_t)15));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned n_tiles = (ws->list_count + CTB - 1) / CTB;
  const unsigned tile0 = (unsigned)((unsigned long long)blockIdx.x * n_tiles / gridDim.x);
  const int T = (int)((unsigned)((unsigned long long)(blockIdx.x + 1) * n_tiles / gridDim.x) - tile0);
  const unsigned short* ts = a.tile_start + (size_t)tile0 * TS_PITCH;
  if (T <= smem_tiles) {                  // the cell starts of this CTA's tiles, kept over the iterations
    const uint4* from = reinterpret_cast<const uint4*>(ts);
    for (int i = tid; i < T * (TS_PITCH / 8); i += ITB) reinterpret_cast<uint4*>(s_ts)[i] = from[i];
    ts = s_ts;
  }
  {
    constexpr int DW = (int)(sizeof(IterDesc) / sizeof(unsigned));
    if (tid < DW) reinterpret_cast<unsigned*>(&S.d)[tid] = reinterpret_cast<const unsigned*>(&ws->desc)[tid];
  }
  if (tid < 2 * LIMBS * SOP_MAX_ENTRIES) (&S.limb[0][0][0])[tid] = 0u;
  if (tid < 2 * SOP_MAX_ENTRIES) (&S.sum[0][0])[tid] = 0ull;
  CellMoments mom = {0.0, 0.0, 0.0};
  if (blockIdx.x == 0) {
    // prefix sums over the cells, one cell per thread: inside the warps, then the warps' totals
    __shared__ unsigned long long t_n[32];
    __shared__ long long t_s[32];
    static_assert(SORT_ROWS <= ITB, "one cell per thread");
    const bool in = tid < SORT_ROWS;
    unsigned long long n = in ? ws->cellN[tid] : 0ull;
    long long s = in ? ws->cellS[tid] : 0ll;
    if (in) mom = {ws->cellA[0][tid], ws->cellA[1][tid], ws->cellA[2][tid]};
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long un = __shfl_up_sync(0xFFFFFFFFu, n, o);
      const long long us = __shfl_up_sync(0xFFFFFFFFu, s, o);
      if (lane >= o) { n += un; s += us; }
    }
    if (lane == 31) { t_n[warp] = n; t_s[warp] = s; }
    __syncthreads();
    for (int w = 0; w < warp && w < 32; ++w) { n += t_n[w]; s += t_s[w]; }
    if (in) { S.preN[tid + 1] = n; S.preS[tid + 1] = s; }
    if (tid == 0) { S.preN[0] = 0; S.preS[0] = 0; }
  }
  __syncthreads();
  if (warp == 0) split_cells(S);
  __syncthreads();
  for (int it = it0;; ++it) {
    const bool last = it == iters;
    iteration_share<ALL>(a, ws, S, ts, mom, tile0, T, it, last);
    if (warp == 0) {
      bool go = true;
      unsigned long long n = 0;
      long long s = 0;
      if (ALL && !last) {
        for (unsigned polls = 0;;) {
          const bool there = lane >= S.d.n_entries || read_sums(ws->acc[it], gridDim.x, n, s);
          if (__all_sync(0xFFFFFFFFu, there)) break;
          ++polls;
          const bool give_up = polls > WAIT_POLLS || ((polls & 63u) == 0u && *(volatile unsigned*)&ws->error != 0u);
          if (__any_sync(0xFFFFFFFFu, give_up)) { go = false; break; }
        }
        if (!go && lane == 0) atomicExch(&ws->error, 1u);
      } else if (ALL) {
        // CTA 0 waits for everybody's distortions: it reports the result
        if (blockIdx.x == 0 && lane == 0) {
          unsigned polls = 0, seen;
          for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&ws->arrive[it]) : "memory");
            if (seen >= gridDim.x) break;
            if (++polls > WAIT_POLLS || ((polls & 63u) == 0u && *(volatile unsigned*)&ws->error != 0u)) { atomicExch(&ws->error, 1u); go = false; break; }
          }
        }
        go = __shfl_sync(0xFFFFFFFFu, go ? 1 : 0, 0) != 0;
        if (go && blockIdx.x == 0)
          for (int i = lane; i <= iters; i += 32) distortion[i] = __ldcg(&ws->accD[i]);
      } else {
        go = S.is_last != 0;
        __threadfence();
        if (go && lane == 0) distortion[it] = __ldcg(&ws->accD[it]);
        if (go && !last) {
          n = __ldcg(&ws->acc[it][0][lane]);
          s = (long long)(__ldcg(&ws->acc[it][1][lane]) + (__ldcg(&ws->acc[it][2][lane]) << 32));
        }
      }
      if (go && last && (!ALL || blockIdx.x == 0)) out_lut[lane] = lane < S.d.n_entries ? S.d.lut[lane] : 0.0f;
      if (go && !last) {
        new_table(S, n, s);
        make_desc(ALL ? &S.d : &ws->desc, S.table, S.d.n_entries);
        __syncwarp();
        if (ALL) split_cells(S);
      }
      if (lane == 0) S.stop = !ALL || last || !go ? 1 : 0;
    }
    __syncthreads();
    if (S.stop) return;
  }
}

// ---------------------------------------------------------------------------------------------
// Grid-constrained DD-n (pair-search steps 1 and 3: cluster selection by dynamic programming on the grid points of the
// LUT value format).  The histogram is the per-cell sums that pool_cache_kernel has formed -- H = sum fix(omega),
// S = sum fix(omega u), Q = sum fix((omega u) u), integers, so independent of any order.  The cells with H > 0, in
// ascending order, are cut into min(n_entries, cells) runs; a run's code point is the bf16 value nearest to S / H
// (clamped to +-1.25) and it costs Q - 2 q S + q^2 H; the least total cost wins, a tie between cuts goes to the earliest.
//   grid_dp_cost_kernel   the costs of all runs i .. j, which no row of the programme changes: every CTA works out the prefix sums
//                         for itself and takes its share of the 205 thousand divisions
//   grid_dp_rows_kernel   the rows (number of runs) in one cluster of eight CTAs: a CTA keeps the costs of every eighth last cell
//                         in shared memory, a warp takes a last cell, the row's least costs go to all eight CTAs' shared memory
//                         and a cluster barrier ends the row; then the backtrack
// The FP64 operations are written one by one (no contraction), so every comparison sees the same numbers as a sequential evaluation.
// What bounds it: the latency of the rows (about 3 us each).  2048 x 4096, 16 entries: 223 us with one launch per row that worked the
// costs out again and a serial first and last step, 75 us now.
// ---------------------------------------------------------------------------------------------
constexpr int DP_TB = 1024;
constexpr int DP_CL = 8;                                                             // CTAs of the cluster
constexpr int DP_COLS = (SORT_ROWS + DP_CL - 1) / DP_CL;                             // last cells of a CTA
constexpr int DP_SLICE = DP_CL / 2 * DP_COLS * (DP_COLS - 1) + DP_CL * DP_COLS;      // costs of a CTA, at most

// Scratch of the dynamic programme in the workspace: prefix sums of the non-empty cells, the costs by CTA of the cluster.
struct DpScratch {
  int B;
  int pad;
  long long pH[SORT_ROWS + 1], pS[SORT_ROWS + 1], pQ[SORT_ROWS + 1];
  double cost[DP_CL][DP_SLICE];
};

static size_t lloyd_dp_bytes() { return (sizeof(DpScratch) + 255) & ~(size_t)255; }

// the costs of last cell j (starts 0 .. j) in the slice of CTA j % DP_CL: the cells j % DP_CL, j % DP_CL + DP_CL, ... one after the other
__device__ __forceinline__ int dp_column(int j) {
  const int t = j / DP_CL, c = j % DP_CL;
  return DP_CL / 2 * t * (t - 1) + (c + 1) * t;
}

__device__ __forceinline__ double dp_run_cost(const long long* pH, const long long* pS, const long long* pQ, int i, int j, float* q_out) {
  const double h = __ll2double_rn(pH[j + 1] - pH[i]), sm = __ll2double_rn(pS[j + 1] - pS[i]), qq = __ll2double_rn(pQ[j + 1] - pQ[i]);
  const float mean = __double2float_rn(__ddiv_rn(sm, h));
  uint32_t b = __float_as_uint(mean);
  b += 0x7FFFu + ((b >> 16) & 1u);
  b &= 0xFFFF0000u;                                   // nearest bf16, ties to even
  float q = __uint_as_float(b);
  q = fminf(1.25f, fmaxf(-1.25f, q));
  if (q_out) *q_out = q;
  const double qd = (double)q;
  const double a = __dmul_rn(__dmul_rn(2.0, qd), sm);
  const double c = __dmul_rn(__dmul_rn(qd, qd), h);
  return __dadd_rn(__dsub_rn(qq, a), c);
}

__global__ void __launch_bounds__(DP_TB) grid_dp_cost_kernel(const LloydWs* ws, DpScratch* dp) {
  __shared__ long long pre[3][SORT_ROWS + 1];
  __shared__ long long tot[4][32];
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  static_assert(SORT_ROWS <= DP_TB, "one cell per thread");
  long long v[3] = {0, 0, 0};
  if (tid < SORT_ROWS) { v[0] = (long long)ws->cellN[tid]; v[1] = ws->cellS[tid]; v[2] = ws->cellQ[tid]; }
  const bool on = v[0] > 0;
  if (!on) v[1] = v[2] = 0;
  long long n = on ? 1 : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long a = __shfl_up_sync(0xFFFFFFFFu, v[0], o), b = __shfl_up_sync(0xFFFFFFFFu, v[1], o), c = __shfl_up_sync(0xFFFFFFFFu, v[2], o);
    const long long m = __shfl_up_sync(0xFFFFFFFFu, n, o);
    if (lane >= o) { v[0] += a; v[1] += b; v[2] += c; n += m; }
  }
  if (lane == 31) { tot[0][warp] = v[0]; tot[1][warp] = v[1]; tot[2][warp] = v[2]; tot[3][warp] = n; }
  __syncthreads();
  int B = 0;
  for (int w = 0; w < DP_TB / 32; ++w) {
    if (w < warp) { v[0] += tot[0][w]; v[1] += tot[1][w]; v[2] += tot[2][w]; n += tot[3][w]; }
    B += (int)tot[3][w];
  }
  if (on) { pre[0][n] = v[0]; pre[1][n] = v[1]; pre[2][n] = v[2]; }
  if (tid < 3) pre[tid][0] = 0;
  __syncthreads();
  if (blockIdx.x == 0) {
    for (int i = tid; i <= B; i += DP_TB) { dp->pH[i] = pre[0][i]; dp->pS[i] = pre[1][i]; dp->pQ[i] = pre[2][i]; }
    if (tid == 0) dp->B = B;
  }
  // last cells j and B - 1 - j together have B + 1 starts: the CTAs take such pairs
  for (int p = blockIdx.x; 2 * p < B; p += gridDim.x) {
    const int ja = p, jb = B - 1 - p;
    const int n_a = ja + 1, total = jb > ja ? n_a + jb + 1 : n_a;
    for (int x = tid; x < total; x += DP_TB) {
      const int j = x < n_a ? ja : jb, i = x < n_a ? x : x - n_a;
      dp->cost[j % DP_CL][dp_column(j) + i] = dp_run_cost(pre[0], pre[1], pre[2], i, j, nullptr);
    }
  }
}

struct DpSmem {
  double best[2][SORT_ROWS];
  float lut[SOP_MAX_ENTRIES];
  double cost[DP_SLICE];          // CTA 0, after the last row: where the last run starts, [rows][SORT_ROWS] 16-bit numbers
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __cluster_dims__(DP_CL, 1, 1) __launch_bounds__(DP_TB) grid_dp_rows_kernel(const DpScratch* dp, int n_entries,
                                                                                         short* cut, float* out_lut,
                                                                                         double* cost_out) {
  extern __shared__ __align__(16) unsigned char dp_smem[];
  DpSmem& S = *reinterpret_cast<DpSmem*>(dp_smem);
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = (int)blockIdx.x;       // one cluster
  const int B = dp->B, R = min(n_entries, B);
  if (B == 0) {
    if (rank == 0 && tid < SOP_MAX_ENTRIES) out_lut[tid] = 0.0f;
    if (rank == 0 && tid == 0) cost_out[0] = 0.0;
    return;                                            // (the same in every CTA)
  }
  const int n_cols = rank < B ? (B - 1 - rank) / DP_CL + 1 : 0, j_end = rank + DP_CL * n_cols;
  const int n_cost = dp_column(j_end);
  for (int x = tid; x < n_cost; x += DP_TB) S.cost[x] = dp->cost[rank][x];
  for (int j = tid; j < B; j += DP_TB) S.best[0][j] = dp->cost[j % DP_CL][dp_column(j)];        // one run: cells 0 .. j
  cluster_sync();
  for (int r = 1; r < R; ++r) {
    const double* prev = S.best[(r - 1) & 1];
    // a warp per last cell j, the lanes share the starts i of the last run; the least value wins, a tie goes to the smallest i (what
    // a sequential scan from the first start on keeps)
    for (int t = warp; t < n_cols; t += DP_TB / 32) {
      const int j = rank + DP_CL * t;
      if (j < r) continue;
      const double* col = S.cost + dp_column(j);
      double bv = 0.0;
      int bi = -1;
      for (int i = r + lane; i <= j; i += 32) {
        const double v = __dadd_rn(prev[i - 1], col[i]);
        if (bi < 0 || v < bv) { bv = v; bi = i; }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const double ov = __shfl_xor_sync(0xFFFFFFFFu, bv, o);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
        if (oi >= 0 && (bi < 0 || ov < bv || (ov == bv && oi < bi))) { bv = ov; bi = oi; }
      }
      if (lane < DP_CL) {                              // to the shared memory of every CTA of the cluster
        unsigned at;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((unsigned)__cvta_generic_to_shared(&S.best[r & 1][j])), "r"(lane));
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(bv) : "memory");
      }
      if (lane == 0) cut[(size_t)r * SORT_ROWS + j] = (short)bi;
    }
    cluster_sync();
  }
  if (rank != 0) return;
  // the backtrack, the code points in ascending order, the least total cost; with fewer cells than entries the programme stops at
  // the last row that has a cell
  short* s_cut = reinterpret_cast<short*>(S.cost);
  for (int x = tid; x < R * SORT_ROWS; x += DP_TB) s_cut[x] = x < SORT_ROWS ? 0 : __ldcg(cut + x);
  __syncthreads();
  if (warp == 0) {
    int j = B - 1, my_i = 0, my_j = 0;
    for (int r = R - 1; r >= 0; --r) {
      const int i = s_cut[r * SORT_ROWS + j];
      if (lane == r) { my_i = i; my_j = j; }
      j = i - 1;
    }
    float q = __int_as_float(0x7F800000);
    if (lane < R) dp_run_cost(dp->pH, dp->pS, dp->pQ, my_i, my_j, &q);
    int at = 0;                                        // ascending, ties by run
#pragma unroll 1
    for (int k = 0; k < R; ++k) {
      const float o = __shfl_sync(0xFFFFFFFFu, q, k);
      at += o < q || (o == q && k < lane) ? 1 : 0;
    }
    if (lane < R) S.lut[at] = q;
    __syncwarp();
    out_lut[lane] = lane < n_entries ? S.lut[min(lane, R - 1)] : 0.0f;
    if (lane == 0) cost_out[0] = __ddiv_rn(S.best[(R - 1) & 1][B - 1], 16777216.0);
  }
}

int num_sms();

// Grid of the iteration kernels and whether all iterations run in one cooperative launch: they do wherever the device launches
// cooperatively (the CTAs wait for one another between iterations, so the whole grid has to be resident: at most one per SM);
// otherwise there is one launch per iteration.  Four tiles per CTA at least: their split cells' runs keep its 128 groups of eight
// lanes busy for half a step to a step, and a CTA less is an arrival less.
static size_t iter_smem_bytes(int tiles) { return ((sizeof(IterSmem) + 15) & ~(size_t)15) + (size_t)tiles * TS_PITCH * sizeof(unsigned short); }
constexpr size_t ITER_SMEM_MAX = 225 * 1024;

static bool lloyd_iteration_plan(long long NB, long long pool_blocks, int iters, int flags, long long* grid_out) {
  const int sms = num_sms();
  const long long likely = (pool_blocks + CTB - 1) / CTB;           // cache tiles of the pool without ties at its threshold
  long long grid = (likely + 3) / 4;
  if (grid > sms) grid = sms;
  if (grid > 255) grid = 255;                                       // (a byte counts them)
  if (g_tune.iter_ctas > 0 && grid > g_tune.iter_ctas) grid = g_tune.iter_ctas;
  if (grid < 1) grid = 1;
  DeviceFacts* facts = device_facts();
  if (facts->coop_blocks_per_sm < 0) {
    int dev = 0, coop = 0, nb = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
        cudaFuncSetAttribute(lloyd_iter_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ITER_SMEM_MAX) == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, lloyd_iter_kernel<true>, ITB, ITER_SMEM_MAX) == cudaSuccess)
      facts->coop_blocks_per_sm = nb;
    else
      facts->coop_blocks_per_sm = 0;
    cudaGetLastError();
  }
  *grid_out = grid;
  return iters >= 1 && NB < (1ll << 27) && facts->coop_blocks_per_sm >= 1 && !(flags & SOP_LLOYD_LAUNCH_PER_ITERATION);
}

}  // namespace sop

extern "C" {

int sop_dd4_lloyd_launches(long long M, long long K, int iters, int flags, int* launches) {
  if (!launches) return SOP_ERR_NULL;
  if (M < 1 || K < 1 || (K % SOP_G) != 0 || iters < 0 || iters > sop::SOP_MAX_LLOYD_ITERS) return SOP_ERR_RANGE;
  long long grid = 1;
  const bool persistent = sop::lloyd_iteration_plan(M * (K / SOP_G), M * (K / SOP_G), iters, flags, &grid);
  // radix select (three passes, unless the pool is cut by a threshold), set-up, pool list, pool cache, iterations
  // the dynamic programme: the costs, the rows
  *launches = ((flags & SOP_LLOYD_POOL_THRESHOLD) ? 0 : 3) + 3 + ((flags & SOP_LLOYD_GRID_DP) ? 2 : (persistent ? 1 : iters + 1));
  return SOP_OK;
}

int sop_dd4_lloyd_tuning(int cell_spill_tiles, int cache_ctas, int tiles_per_warp, int iter_ctas) {
  using namespace sop;
  if (cell_spill_tiles < 1 || cell_spill_tiles > CELL_SPILL_TILES_MAX || cache_ctas < 0 || tiles_per_warp < 1 ||
      tiles_per_warp > TILES_PER_WARP_MAX || iter_ctas < 0) return SOP_ERR_RANGE;
  g_tune.spill_tiles = cell_spill_tiles;
  g_tune.cache_ctas = cache_ctas;
  g_tune.iter_ctas = iter_ctas;
  return SOP_OK;
}

int sop_dd4_lloyd_workspace(long long M, long long K, size_t* bytes) {
  if (!bytes) return SOP_ERR_NULL;
  if (M < 1 || K < 1 || (K % SOP_G) != 0) return SOP_ERR_SHAPE;
  if (M > (1ll << 31) / (K / SOP_G)) return SOP_ERR_SHAPE;
  *bytes = sop::lloyd_ws_bytes(M, K);
  return SOP_OK;
}

int sop_dd4_lloyd(const void* W_dev, long long M, long long K, long long ldw, const float* c_dev, int g,
                  const sop_scale_fmt* fmt, int k_mode, const sop_search_result* search_dev,
                  const float* block_metric_dev, long long pool_rank, float pool_threshold, int flags,
                  const sop_atom* atoms, int n_atoms,
                  int fmta_index, int iters, float* out_lut_dev, double* distortion_dev,
                  long long* pool_count_dev, void* workspace_dev, size_t workspace_bytes, void* stream) {
  using namespace sop;
  int rc = validate_layer(W_dev, M, K, ldw, c_dev, g);
  if (rc) return rc;
  if (!block_metric_dev || !out_lut_dev || !distortion_dev || !pool_count_dev) return SOP_ERR_NULL;
  if (flags & ~(SOP_LLOYD_POOL_BY_ERROR | SOP_LLOYD_UNIFORM_WEIGHTS | SOP_LLOYD_POOL_THRESHOLD | SOP_LLOYD_LAUNCH_PER_ITERATION | SOP_LLOYD_GRID_DP)) return SOP_ERR_RANGE;
  const bool grid_dp = (flags & SOP_LLOYD_GRID_DP) != 0;
  if (grid_dp && iters != 0) return SOP_ERR_RANGE;        // the dynamic programme replaces the iterations
  const bool by_threshold = (flags & SOP_LLOYD_POOL_THRESHOLD) != 0;
  if (by_threshold && !(pool_threshold == pool_threshold)) return SOP_ERR_RANGE;   // NaN orders nothing
  FmtDev F;
  if ((rc = validate_fmt(fmt, &F))) return rc;
  AtomsDev A;
  if ((rc = validate_atoms(atoms, n_atoms, 0u, nullptr, &A))) return rc;
  const long long NB = M * (K / SOP_G);
  if ((!by_threshold && (pool_rank < 1 || pool_rank > NB)) || iters < 0 || iters > 64) return SOP_ERR_RANGE;
  if (k_mode != SOP_K_FROM_RESULT && (k_mode < -64 || k_mode > 64)) return SOP_ERR_RANGE;
  if ((k_mode == SOP_K_FROM_RESULT || fmta_index == SOP_FMTA_FROM_RESULT) && !search_dev) return SOP_ERR_NULL;
  if (fmta_index != SOP_FMTA_FROM_RESULT && (fmta_index < 0 || fmta_index >= n_atoms)) return SOP_ERR_RANGE;
  if (fmta_index >= 0 && atoms[fmta_index].kind != SOP_KIND_LUT) return SOP_ERR_ALPHABET;
  if (NB * 16 > (1ll << 31)) return SOP_ERR_SHAPE;   // int64 fixed-point sums: at most 2^31 elements
  size_t need = 0;
  sop_dd4_lloyd_workspace(M, K, &need);
  if (!workspace_dev || ((uintptr_t)workspace_dev & 255u) || workspace_bytes < need) return SOP_ERR_WORKSPACE;

  // entries of the table the dynamic programme builds: FMTa's; when FMTa is chosen on the device every table atom must
  // agree on the number (decided here, before the first enqueue)
  int ne = 0;
  if (grid_dp) {
    ne = fmta_index >= 0 ? atoms[fmta_index].n_entries : 0;
    for (int i = 0; i < n_atoms && fmta_index < 0; ++i) {
      if (atoms[i].kind != SOP_KIND_LUT) continue;
      if (ne == 0) ne = atoms[i].n_entries;
      else if (atoms[i].n_entries != ne) return SOP_ERR_ALPHABET;
    }
    if (ne < 2) return SOP_ERR_ALPHABET;
  }

  unsigned char* wsb = (unsigned char*)workspace_dev;
  LloydArgs a;
  a.W = (const uint16_t*)W_dev; a.c = c_dev; a.cosrow_base = block_metric_dev;
  a.M = M; a.K = K; a.ldw = ldw; a.nbk = K / SOP_G; a.NB = NB; a.pool_rank = pool_rank;
  a.k_mode = k_mode; a.fmta_index = fmta_index; a.n_atoms = n_atoms;
  a.flags = flags; a.pool_threshold = pool_threshold;
  a.omega = (float*)(wsb + lloyd_off_omega());
  a.pool_idx = (unsigned*)(wsb + lloyd_off_idx(K));
  a.cache = (uint2*)(wsb + lloyd_off_cache(M, K));
  a.tile_start = (unsigned short*)(wsb + lloyd_off_tiles(M, K));
  LloydWs* ws = (LloydWs*)workspace_dev;
  cudaStream_t st = (cudaStream_t)stream;
  if ((rc = profile_mark(SOP_PROFILE_POOL, 0, st))) return rc;
  const int sms = num_sms();
  long long sg = (NB + LTB * 8 - 1) / (LTB * 8);
  if (sg > sms * 4) sg = sms * 4;
  if (sg < 1) sg = 1;
  SOP_CUDA_TRY(launch(lloyd_init_kernel, 9, INIT_TB, 0, st, a, A, search_dev, ws, distortion_dev, iters));
  if (!by_threshold) {     // radix select of the pool_rank-th worst block (three passes over the ranking keys)
    SOP_CUDA_TRY(launch(select_kernel<0>, sg, LTB, 0, st, a, search_dev, ws));
    SOP_CUDA_TRY(launch(select_kernel<1>, sg, LTB, 0, st, a, search_dev, ws));
    SOP_CUDA_TRY(launch(select_kernel<2>, sg, LTB, 0, st, a, search_dev, ws));
  }
  const long long lg = (NB + LIST_ROUND - 1) / LIST_ROUND;
  SOP_CUDA_TRY(launch(pool_list_kernel, (unsigned)(lg < sms * 6 ? lg : sms * 6), LTB, 0, st, a, ws));

  // (u, omega) of every pool element, once: sorted tiles, cell starts, per-cell sums and moments
  {
    long long cg = (NB + CTB - 1) / CTB;      // one tile per CTA pass
    const long long cg_max = g_tune.cache_ctas > 0 ? g_tune.cache_ctas : (long long)sms * 2;
    if (cg > cg_max) cg = cg_max;
    const size_t stage_bytes = sizeof(CacheSmem);
    DeviceFacts* facts = device_facts();
    if (!facts->lloyd_attr_set) {
      SOP_CUDA_TRY(cudaFuncSetAttribute(pool_cache_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stage_bytes));
      SOP_CUDA_TRY(cudaFuncSetAttribute(pool_cache_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stage_bytes));
      SOP_CUDA_TRY(cudaFuncSetAttribute(grid_dp_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DpSmem)));
      SOP_CUDA_TRY(cudaFuncSetAttribute(lloyd_iter_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ITER_SMEM_MAX));
      facts->lloyd_attr_set = true;
    }
    if (grid_dp) SOP_CUDA_TRY(launch(pool_cache_kernel<true>, cg, CTB, stage_bytes, st, a, F, ws, pool_count_dev, (unsigned)g_tune.spill_tiles));
    else SOP_CUDA_TRY(launch(pool_cache_kernel<false>, cg, CTB, stage_bytes, st, a, F, ws, pool_count_dev, (unsigned)g_tune.spill_tiles));
    SOP_CUDA_TRY(cudaGetLastError());
  }
  if ((rc = profile_mark(SOP_PROFILE_POOL, 1, st))) return rc;
  if (grid_dp) {
    if ((rc = profile_mark(SOP_PROFILE_LLOYD, 0, st))) return rc;
    DpScratch* dp = reinterpret_cast<DpScratch*>(wsb + lloyd_off_dp());
    SOP_CUDA_TRY(launch(grid_dp_cost_kernel, sms, DP_TB, 0, st, ws, dp));
    SOP_CUDA_TRY(launch(grid_dp_rows_kernel, DP_CL, DP_TB, sizeof(DpSmem), st, dp, ne, &ws->dp_cut[0][0], out_lut_dev, distortion_dev));
    if ((rc = profile_mark(SOP_PROFILE_LLOYD, 1, st))) return rc;
    return SOP_OK;
  }
  long long grid = 1;
  const long long expected = by_threshold ? NB : pool_rank;
  const bool persistent = lloyd_iteration_plan(NB, expected, iters, flags, &grid);
  // room for the cell starts of the tiles that a CTA is likely to have (and a few more, for ties); more tiles are read from memory
  int smem_tiles = (int)(((expected + CTB - 1) / CTB + grid - 1) / grid + 4);
  while (smem_tiles > 0 && iter_smem_bytes(smem_tiles) > ITER_SMEM_MAX) --smem_tiles;
  const size_t iter_smem = iter_smem_bytes(smem_tiles);
  if ((rc = profile_mark(SOP_PROFILE_LLOYD, 0, st))) return rc;
  if (persistent) {
    int it0 = 0;
    void* kargs[] = {(void*)&a, (void*)&ws, (void*)&distortion_dev, (void*)&it0, (void*)&iters, (void*)&out_lut_dev, (void*)&smem_tiles};
    SOP_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)lloyd_iter_kernel<true>, dim3((unsigned)grid), dim3(ITB), kargs, iter_smem, st));
  } else {
    for (int it = 0; it <= iters; ++it)
      SOP_CUDA_TRY(launch(lloyd_iter_kernel<false>, grid, ITB, iter_smem, st, a, ws, distortion_dev, it, iters, out_lut_dev, smem_tiles));
  }
  if ((rc = profile_mark(SOP_PROFILE_LLOYD, 1, st))) return rc;
  SOP_CUDA_TRY(cudaGetLastError());
  return SOP_OK;
}

}  // extern "C"
