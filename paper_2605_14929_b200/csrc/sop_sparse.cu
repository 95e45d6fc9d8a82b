// sop_opq_extract and sop_wr_extract: the two sparse side streams on either side of the search.
//
// Both are scans with an ordered compaction: a thread owns one 16-element block, a CTA pass ("tile") 256
// consecutive blocks.  The records of a stream ascend by (row, column), which is the order of the blocks and of
// the elements inside a block, so the place of a block's first record is the exclusive prefix sum of the
// per-block record counts:
//   count kernel    per-tile record counts (one 32-bit sum per tile)
//   tile_scan       one CTA turns them into exclusive offsets, writes the total
//   write kernel    recomputes the per-block counts, scans them inside the CTA and writes records and row starts
// Nothing waits on another CTA.
//
//   opq_mask_kernel     reads W once: per block the outlier mask (binary64 test w_i^2 g > m^2 sum w^2), W_out with
//                       the outliers zeroed, the 16-bit mask, the tile count, and the tile's records (column |
//                       bf16 bits << 16) in order
//   opq_write_kernel    moves the tiles' records to their place in the stream, writes the row starts
//   wr_max_kernel       first decode pass of the packed stream (scale word -> s_hat, codes -> table values, residual
//                       E = w - s_hat q with one rounding, metric |E| c_k): per block the largest metric, of which the
//                       top 11 bits (inverted) are its bin.  The bins go to memory, two bytes per block, and into a
//                       histogram.  At least n_keep elements are as large as the n_keep-th largest block maximum, so
//                       the threshold lies in that value's bin or an earlier one
//   wr_collect_kernel   reads the bins, decodes only the blocks that reach the bound; every element whose bin is not
//                       later than it goes to a candidate list (position, residual, metric): a fraction of a per cent
//                       of the layer.  The bins' memory is left zeroed: it becomes the map of the kept entries
//   wr_select_kernel<1,2>, wr_mark_kernel
//                       over the list: radix select (11 / 11 / 10 bits, the first digit was counted by the collecting
//                       kernel) of the n_keep-th largest metric, then the kept set as one 16-bit mask per block, the
//                       per-tile counts and the largest kept |E|
//   wr_write_kernel     E3M4 codes of E / 2^e, records (column | code << 16): a warp per kept entry of the list counts
//                       the entries before it in its tile's map
// The last CTA of a histogram kernel picks the bin that holds the rank (wr_pick).  When the candidates do not fit their
// list (a layer whose metrics are nearly all alike) the flag that wr_collect_kernel's last CTA sets makes the kernels
// after it decode the whole layer instead.
// The residual is never stored: decoding a block (2.6 bytes per element read) is cheaper than reading 4 bytes.
#include <math.h>
#include <string.h>

#include "sop_device.cuh"

namespace sop {

constexpr int STB = 256;          // threads per CTA = blocks per tile

int num_sms();

struct SparseWs {
  unsigned hist[3][2048];
  unsigned hist_bm[2048];         // histogram of the per-block maxima of the metric (top 11 bits of the inverted key)
  unsigned bm_bin;                // bin of the n_keep-th largest block maximum: the threshold cannot lie in a later bin
  unsigned prefix;                // inverted-key prefix fixed by the selection passes so far
  unsigned tau_bits;              // the threshold metric as fp32 bits (a NaN pattern: nothing is kept)
  unsigned long long rank;        // rank still to find among the keys with that prefix
  unsigned emax_bits;             // max |E| over the kept entries, fp32 bits
  int scale_exp;
  int no_pair;                    // the search result holds no pair: nothing was packed, nothing is corrected
  unsigned n_cand;                // candidates found (may exceed the list's capacity: then the list is not used)
  unsigned overflow;              // 1: the candidates did not fit, the full decode passes do the work
  unsigned done[4];               // CTAs that have added their histogram, per kernel
};

static size_t sparse_tiles_off() { return (sizeof(SparseWs) + 255) & ~(size_t)255; }
static long long sparse_tiles(long long NB) { return (NB + STB - 1) / STB; }
static size_t sparse_masks_off(long long NB) { return sparse_tiles_off() + (((size_t)sparse_tiles(NB) * 4 + 255) & ~(size_t)255); }
// behind the per-block masks, OPQ: the tiles' records
static size_t opq_local_off(long long NB) { return sparse_masks_off(NB) + (((size_t)NB * 2 + 255) & ~(size_t)255); }
// Wr: the candidate list, three 32-bit arrays of wr_cand_cap entries
static size_t wr_cand_off(long long NB) { return sparse_masks_off(NB) + (((size_t)NB * 2 + 255) & ~(size_t)255); }
static unsigned wr_cand_cap(long long NB) { const long long c = NB / 4; return (unsigned)(c > 65536 ? c : 65536); }   // 1/64 of the elements

// exclusive prefix sum of one value per thread over the CTA (STB threads); *total = the CTA's sum
__device__ __forceinline__ unsigned cta_excl_scan(unsigned v, unsigned* s_warp, unsigned* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();                 // s_warp may still be read from the previous tile
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  unsigned base = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < STB / 32; ++w) { const unsigned c = s_warp[w]; tot += c; if (w < warp) base += c; }
  *total = tot;
  return base + incl - v;
}

// In place: tile_sums[t] becomes the number of records before tile t.  One CTA; a thread holds 16 consecutive tiles of a
// chunk of 16384 in registers (four loads in flight, one scan of the CTA per chunk).  The total goes to row_start[M] and
// *count.  With `wr` the kernel also turns the largest kept |E| into the layer exponent of the Wr values.
__global__ void __launch_bounds__(1024) tile_scan_kernel(unsigned* tile_sums, long long n_tiles, unsigned* row_start,
                                                         long long M, long long* count, SparseWs* ws, int wr,
                                                         int* scale_exp_out, float* tau_out) {
  pdl_trigger();
  pdl_wait();
  __shared__ unsigned s_warp[2][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned total = 0;
  int par = 0;
  for (long long c0 = 0; c0 < n_tiles; c0 += 16384, par ^= 1) {
    const long long t0 = c0 + tid * 16;
    uint4* p = reinterpret_cast<uint4*>(tile_sums + t0);         // the array is padded to 256 bytes
    uint4 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = make_uint4(0u, 0u, 0u, 0u);
      const long long i = t0 + 4 * q;
      if (i < n_tiles) {
        v[q] = p[q];
        if (i + 1 >= n_tiles) v[q].y = 0;                        // beyond the end: whatever lies in the padding
        if (i + 2 >= n_tiles) v[q].z = 0;
        if (i + 3 >= n_tiles) v[q].w = 0;
      }
    }
    unsigned local = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) local += v[q].x + v[q].y + v[q].z + v[q].w;
    unsigned incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[par][warp] = incl;
    __syncthreads();
    const unsigned ws_ = s_warp[par][lane];
    unsigned run = total + incl - local + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? ws_ : 0u);
    total += __reduce_add_sync(0xFFFFFFFFu, ws_);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint4 o;
      o.x = run; run += v[q].x;
      o.y = run; run += v[q].y;
      o.z = run; run += v[q].z;
      o.w = run; run += v[q].w;
      if (t0 + 4 * q < n_tiles) p[q] = o;
    }
  }
  if (tid == 0) {
    row_start[M] = total;
    if (count) *count = wr && ws->no_pair ? -1ll : (long long)total;
    if (wr) {
      const float emax = __uint_as_float(ws->emax_bits);
      const int e = emax > 0.0f ? ilogb_pos(layer_pot_scale(emax, 15.5f)) : 0;
      ws->scale_exp = e;
      if (scale_exp_out) *scale_exp_out = e;
      if (tau_out) *tau_out = __uint_as_float(ws->tau_bits);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// OPQ
// ---------------------------------------------------------------------------------------------
constexpr unsigned OPQ_LOCAL = STB;       // records of a tile kept at hand: one per block (a tile with more reads them from W again)

struct OpqArgs {
  const uint16_t* W;
  uint16_t* W_out;
  long long M, K, ldw, ldo, nbk, NB;
  double m2;                      // the threshold squared
  unsigned short* masks;          // workspace: one 16-bit outlier mask per block
  unsigned* tile_sums;            // workspace
  unsigned* local;                // workspace: OPQ_LOCAL records per tile
  unsigned* row_start;
  unsigned* records;
  long long capacity;
};

// A tile per step, the next tile's elements loaded before this one's arithmetic, one barrier per tile (the warps' counts
// are double-buffered).
// What bounds it: DRAM, 300 MB in 55 us at 8192 x 8192, of which the input's copy without outliers is 268 MB.
__global__ void __launch_bounds__(STB) opq_mask_kernel(OpqArgs a) {
  pdl_trigger();
  pdl_wait();
  __shared__ unsigned s_cnt[2][STB / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned NB = (unsigned)a.NB, nbk = (unsigned)a.nbk, n_tiles = (NB + STB - 1) / STB;   // the block count fits 31 bits
  uint4 v0, v1;
  unsigned m = 0, j = 0;
  auto fetch = [&](unsigned tile) {
    const unsigned blk = tile * STB + tid;
    if (tile < n_tiles && blk < NB) {
      m = blk / nbk; j = blk - m * nbk;
      const uint4* p = reinterpret_cast<const uint4*>(a.W + (long long)m * a.ldw + (long long)j * SOP_G);
      v0 = *p; v1 = p[1];
    }
  };
  fetch(blockIdx.x);
  int par = 0;
  for (unsigned tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, par ^= 1) {
    const unsigned blk = tile * STB + tid;
    uint32_t wb[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
    const unsigned cm = m, cj = j;
    fetch(tile + gridDim.x);
    unsigned mask = 0;
    if (blk < NB) {
      double sq[16], s2 = 0.0;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const double w = (double)((i & 1) ? bf16hi(wb[i >> 1]) : bf16lo(wb[i >> 1]));
        sq[i] = __dmul_rn(w, w);                 // exact: a bf16 value has 8 significant bits
        s2 = __dadd_rn(s2, sq[i]);               // element order
      }
      const double rhs = __dmul_rn(a.m2, s2);
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (__dmul_rn(sq[i], 16.0) > rhs) {
          mask |= 1u << i;
          wb[i >> 1] &= (i & 1) ? 0x0000FFFFu : 0xFFFF0000u;
        }
      uint4* q = reinterpret_cast<uint4*>(a.W_out + (long long)cm * a.ldo + (long long)cj * SOP_G);
      q[0] = make_uint4(wb[0], wb[1], wb[2], wb[3]);
      q[1] = make_uint4(wb[4], wb[5], wb[6], wb[7]);
      a.masks[blk] = (unsigned short)mask;
    }
    const unsigned mine = (unsigned)__popc(mask);
    const unsigned cnt = __reduce_add_sync(0xFFFFFFFFu, mine);
    if (lane == 0) s_cnt[par][warp] = cnt;
    __syncthreads();
    const unsigned other = lane < STB / 32 ? s_cnt[par][lane] : 0u;
    const unsigned sum = __reduce_add_sync(0xFFFFFFFFu, other);
    if (tid == 0) a.tile_sums[tile] = sum;
    if (cnt && sum <= OPQ_LOCAL) {
      unsigned incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
      }
      unsigned pos = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? other : 0u) + incl - mine;
      const uint16_t* p = a.W + (long long)cm * a.ldw + (long long)cj * SOP_G;
      for (unsigned rest = mask; rest; rest &= rest - 1u, ++pos) {
        const int i = __ffs((int)rest) - 1;
        a.local[(size_t)tile * OPQ_LOCAL + pos] = (cj * SOP_G + (unsigned)i) | ((unsigned)p[i] << 16);
      }
    }
  }
}

// A warp per tile: the tile's records lie together already and move to their place in the stream; the masks are read only
// where a row starts inside the tile, or where the tile has more records than its share of the workspace.
// 11 us at 8192 x 8192 with 1.3 million records (32 us when the values were read from W once more: their sectors are all of W).
__global__ void __launch_bounds__(STB) opq_write_kernel(OpqArgs a) {
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned NB = (unsigned)a.NB, nbk = (unsigned)a.nbk, n_tiles = (NB + STB - 1) / STB;   // the block count fits 31 bits
  for (unsigned tile = blockIdx.x * (STB / 32) + (tid >> 5); tile < n_tiles; tile += gridDim.x * (STB / 32)) {
    const unsigned base = a.tile_sums[tile];
    const unsigned cnt = (tile + 1 < n_tiles ? a.tile_sums[tile + 1] : a.row_start[a.M]) - base;
    const unsigned t0 = tile * STB;
    if (cnt > OPQ_LOCAL) {
      // the tile's records did not fit their share: from the masks and W, 32 neighbouring blocks at a time
      unsigned run = base;
      for (unsigned blk = t0 + lane; blk < t0 + STB; blk += 32) {
        const unsigned mask = blk < NB ? (unsigned)a.masks[blk] : 0u, m = blk / nbk, j = blk - m * nbk;
        const unsigned mine = (unsigned)__popc(mask);
        unsigned incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          if (lane >= o) incl += t;
        }
        unsigned pos = run + incl - mine;
        run += __shfl_sync(0xFFFFFFFFu, incl, 31);
        if (blk < NB && j == 0) a.row_start[m] = pos;
        const uint16_t* p = a.W + (long long)m * a.ldw + (long long)j * SOP_G;
        for (unsigned rest = mask; rest; rest &= rest - 1u, ++pos) {
          const int i = __ffs((int)rest) - 1;
          if ((long long)pos < a.capacity) a.records[pos] = (j * SOP_G + (unsigned)i) | ((unsigned)p[i] << 16);
        }
      }
      continue;
    }
    const unsigned* from = a.local + (size_t)tile * OPQ_LOCAL;
    for (unsigned i = lane; i < cnt; i += 32)
      if ((long long)base + i < a.capacity) a.records[base + i] = from[i];
    const unsigned jt = t0 % nbk;
    if (jt == 0 && lane == 0) a.row_start[t0 / nbk] = base;
    if (jt + min((unsigned)STB, NB - t0) <= nbk) continue;          // no other row starts here
    const unsigned b0 = t0 + 8 * lane;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (b0 < NB) v = *reinterpret_cast<const uint4*>(a.masks + b0);      // the array is padded to 256 bytes
    const unsigned n_here = b0 < NB ? (NB - b0 < 8u ? NB - b0 : 8u) : 0u;
    unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if ((unsigned)e >= n_here) u[e >> 1] &= (e & 1) ? 0x0000FFFFu : 0xFFFF0000u;
    const unsigned mine = (unsigned)(__popc(u[0]) + __popc(u[1]) + __popc(u[2]) + __popc(u[3]));
    unsigned incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += t;
    }
    unsigned pos = base + incl - mine;
    unsigned m = b0 / nbk, j = b0 - m * nbk;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if ((unsigned)e < n_here) {
        if (j == 0) a.row_start[m] = pos;
        pos += (unsigned)__popc((u[e >> 1] >> (16 * (e & 1))) & 0xFFFFu);
        if (++j == nbk) { j = 0; ++m; }
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Wr
// ---------------------------------------------------------------------------------------------
struct WrArgs {
  const uint16_t* W;
  const float* c;
  long long M, K, ldw, nbk, NB;
  int index_a, index_b, k_mode, use_sign;
  int container_bits, word_sign_bits, meta_bits;
  const unsigned char* codes;
  const unsigned* words;
  long long n_keep;
  unsigned* tile_sums;
  unsigned* row_start;
  unsigned* records;
  long long capacity;
  unsigned short* kept;           // workspace: per block the 16-bit mask of kept entries (candidate path)
  unsigned* cand_pos;             // workspace: candidate list: element position blk * 16 + i,
  unsigned* cand_e;               //   residual bits,
  unsigned* cand_m;               //   metric bits
  unsigned cand_cap;
};

struct WrCand { int kind, neg, scope, k, sign_pos, y, bias; float tmax; };

// what a CTA needs to decode the stream: the (up to two) tables and their atoms' parameters
struct WrShared {
  float lutv[2][32];
  float lut4[32];                 // two tables of up to 16 entries side by side: 32 banks, no conflict between the tables
  WrCand cand[2];
  float pot[2];
  int n_bits;
  int no_pair;
};

// value of the code sign | E | M of a floating-point element grid with y mantissa bits and the given bias
__device__ __forceinline__ float fp_grid_decode(uint32_t code, int sign_pos, int y, int bias) {
  const uint32_t mag = code & ((1u << sign_pos) - 1u);
  const uint32_t E = mag >> y, Mm = mag & ((1u << y) - 1u);
  const float v = ldexp_once(E ? ((1u << y) + Mm) : Mm, (int)(E ? E : 1u) - bias - y);
  return ((code >> sign_pos) & 1u) ? -v : v;
}

// the scale a scale code stands for: the tail of scale_quantize
__device__ __forceinline__ float scale_decode(uint32_t code, int k, const FmtDev& f) {
  const int E = (int)(code >> f.y);
  const uint32_t Mm = code & ((1u << f.y) - 1u);
  const uint32_t mant = E ? ((1u << f.y) + Mm) : Mm;
  return mant ? ldexp_once(mant, (E ? E : 1) - f.bias - f.y - k) : 0.0f;
}

// the first warp of every CTA; the caller synchronises afterwards
__device__ void wr_setup(const WrArgs& a, const AtomsDev& A, const sop_search_result* res, WrShared& sh) {
  const int lane = threadIdx.x;
  if (lane >= 32) return;
  int ia = a.index_a, ib = a.index_b;
  const bool from_result = ia == SOP_PAIR_FROM_RESULT;
  if (from_result) {
    ia = a.use_sign ? res->best_sa : res->best_a;
    ib = a.use_sign ? res->best_sb : res->best_b;
  }
  // a result without a pair: the packer wrote nothing, so there is nothing to correct
  const int no_pair = from_result && (ia < 0 || ib < 0 || ia >= A.n_atoms || ib >= A.n_atoms ||
                                      (a.use_sign && (ia + 1 >= A.n_atoms || ib + 1 >= A.n_atoms))) ? 1 : 0;
  ia = max(0, min(A.n_atoms - 1, ia));
  int nb = 1;
  if (ib != SOP_NO_ATOM) { ib = max(0, min(A.n_atoms - 1, ib)); nb = 2; }
  if (lane == 0) { sh.no_pair = no_pair; sh.n_bits = A.atoms[ia].n_bits; }
  if (lane < nb) {
    const int idx = lane ? ib : ia;
    const sop_atom& at = A.atoms[idx];
    WrCand cd;
    cd.kind = at.kind; cd.neg = at.negated; cd.scope = at.scope; cd.tmax = at.tmax;
    cd.k = a.k_mode == SOP_K_FROM_RESULT ? res->k[idx] : a.k_mode;
    if (at.kind == SOP_KIND_FP_E2M3) { cd.sign_pos = 5; cd.y = 3; cd.bias = 1; }
    else if (at.kind == SOP_KIND_FP_E4M3) { cd.sign_pos = 7; cd.y = 3; cd.bias = 7; }
    else { cd.sign_pos = at.grid_exp_bits + at.grid_man_bits; cd.y = at.grid_man_bits; cd.bias = at.grid_bias; }
    sh.cand[lane] = cd;
    sh.pot[lane] = at.scope == 0 ? layer_pot_scale(res ? res->layer_absmax : 0.0f, at.tmax) : 0.0f;
  }
  for (int t = 0; t < nb; ++t) {
    const int idx = t ? ib : ia;
    const sop_atom& at = A.atoms[idx];
    const bool dd = (A.dd_mask >> idx) & 1u;
    const int e = min(lane, (at.kind == SOP_KIND_LUT ? at.n_entries : 1) - 1);
    const float v = at.kind == SOP_KIND_LUT ? (dd ? A.dd_lut[e] : at.lut[e]) : 0.0f;
    sh.lutv[t][lane] = v;
    if (lane < 16) sh.lut4[16 * t + lane] = v;
  }
}

// One block's inputs as they lie in memory: the loads of a block can be issued a step ahead of its arithmetic.
template <bool LUT4>
struct WrRaw {
  uint4 v0, v1;                   // 16 elements
  uint2 c4;                       // n = 4: the codes
  unsigned long long lo, hi;      // else: the 16 n-bit payload as one little-endian integer
  unsigned w0, w1;                // the 32-bit words that hold the scale word (container of 12 bits), or the word
};

template <bool LUT4>
__device__ __forceinline__ WrRaw<LUT4> wr_fetch(const WrArgs& a, int n_bits, unsigned blk, const uint16_t* wrow) {
  WrRaw<LUT4> r;
  const uint4* p = reinterpret_cast<const uint4*>(wrow);
  r.v0 = *p; r.v1 = p[1];
  r.w1 = 0;
  const int b = a.container_bits;
  if (b == 16) r.w0 = (unsigned)*(reinterpret_cast<const unsigned short*>(a.words) + blk);
  else if (b == 8) r.w0 = (unsigned)*(reinterpret_cast<const unsigned char*>(a.words) + blk);
  else {
    const unsigned long long bit = (unsigned long long)blk * 12u;
    const unsigned* q = a.words + (bit >> 5);
    r.w0 = *q;
    if (((unsigned)bit & 31u) > 20u) r.w1 = q[1];
  }
  if constexpr (LUT4) {
    r.c4 = *(reinterpret_cast<const uint2*>(a.codes) + blk);
  } else {
    const int n = n_bits;
    const unsigned char* cp = a.codes + (size_t)blk * 2 * n;
    r.lo = r.hi = 0;
    if (n == 4) {
      const uint2 t = *reinterpret_cast<const uint2*>(cp);
      r.lo = (unsigned long long)t.x | ((unsigned long long)t.y << 32);
    } else if (n == 8) {
      const uint4 t = *reinterpret_cast<const uint4*>(cp);
      r.lo = (unsigned long long)t.x | ((unsigned long long)t.y << 32);
      r.hi = (unsigned long long)t.z | ((unsigned long long)t.w << 32);
    } else {
      const unsigned short* sp = reinterpret_cast<const unsigned short*>(cp);
      for (int i = 0; i < n; ++i) {
        const unsigned long long v = (unsigned long long)sp[i];
        if (i < 4) r.lo |= v << (16 * i); else r.hi |= v << (16 * (i - 4));
      }
    }
  }
  return r;
}

__device__ __forceinline__ void wr_weights(const WrArgs& a, unsigned j, float (&c)[16]) {
  const float4* cq = reinterpret_cast<const float4*>(a.c + (size_t)j * SOP_G);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 v = cq[q];
    c[4 * q] = v.x; c[4 * q + 1] = v.y; c[4 * q + 2] = v.z; c[4 * q + 3] = v.w;
  }
}

// The residual E_i = w_i - s_hat q_i (one rounding) and the metric |E_i| c_k of one block.
// LUT4: both codebooks are tables of at most 16 entries (the common case): constant shifts, no kind test per element.
template <bool LUT4>
__device__ __forceinline__ void wr_decode(const WrArgs& a, const FmtDev& F, const WrShared& sh, unsigned blk, const WrRaw<LUT4>& r,
                                          const float (&c)[16], float (&E)[16], float (&met)[16]) {
  const uint32_t wb[8] = {r.v0.x, r.v0.y, r.v0.z, r.v0.w, r.v1.x, r.v1.y, r.v1.z, r.v1.w};
  const int b = a.container_bits;
  const unsigned word = b == 12 ? __funnelshift_r(r.w0, r.w1, (blk * 12u) & 31u) & 0xFFFu : r.w0;
  // the scale word: sign, scale code, selector
  unsigned sgn = 0, sel = 0, scode;
  const unsigned cmask = (1u << (b - a.word_sign_bits - a.meta_bits)) - 1u;
  if (a.word_sign_bits) { sgn = word >> (b - 1); scode = (word >> a.meta_bits) & cmask; sel = a.meta_bits >= 1 ? (word & 1u) : 0u; }
  else if (a.meta_bits >= 1) { sel = word >> (b - 1); scode = (word >> (a.meta_bits - 1)) & cmask; }
  else scode = word & cmask;
  if (a.index_b == SOP_NO_ATOM) sel = 0;
  float s_hat;
  if (sh.cand[sel].scope == 0) {
    uint32_t mb = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) { mb = max(mb, wb[q] & 0x7FFFu); mb = max(mb, (wb[q] >> 16) & 0x7FFFu); }
    s_hat = mb ? sh.pot[sel] : 0.0f;
  } else {
    s_hat = scale_decode(scode, sh.cand[sel].k, F);
  }
  // (-s) q = s (-q): the sign of a negated table goes to the scale
  const float ns = (sgn != 0) == (sh.cand[sel].neg != 0) ? -s_hat : s_hat;
  if constexpr (LUT4) {
    const char* tab = reinterpret_cast<const char*>(sh.lut4 + 16 * sel);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t cw = i < 8 ? r.c4.x : r.c4.y;
      const int s = 4 * (i & 7) - 2;
      const uint32_t off = (s < 0 ? cw << 2 : cw >> s) & 60u;
      const float q = *reinterpret_cast<const float*>(tab + off);
      const float w = (i & 1) ? bf16hi(wb[i >> 1]) : bf16lo(wb[i >> 1]);
      E[i] = __fmaf_rn(ns, q, w);
      met[i] = __fmul_rn(fabsf(E[i]), c[i]);
    }
  } else {
    const WrCand cd = sh.cand[sel];
    const int n = sh.n_bits;
    const unsigned emask = (1u << n) - 1u;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int pos = i * n;
      unsigned long long v;
      if (pos < 64) { v = r.lo >> pos; if (pos + n > 64) v |= r.hi << (64 - pos); }
      else v = r.hi >> (pos - 64);
      const uint32_t code = (uint32_t)v & emask;
      const float q = cd.kind == SOP_KIND_LUT ? sh.lutv[sel][code & 31u] : fp_grid_decode(code, cd.sign_pos, cd.y, cd.bias);
      const float w = (i & 1) ? bf16hi(wb[i >> 1]) : bf16lo(wb[i >> 1]);
      E[i] = __fmaf_rn(ns, q, w);
      met[i] = __fmul_rn(fabsf(E[i]), c[i]);
    }
  }
}

// a block that is not next to the one before it: all of the above in one
template <bool LUT4>
__device__ __forceinline__ void wr_block(const WrArgs& a, const FmtDev& F, const WrShared& sh, unsigned blk, float (&E)[16], float (&met)[16]) {
  const unsigned m = blk / (unsigned)a.nbk, j = blk - m * (unsigned)a.nbk;   // the block count fits 31 bits
  const WrRaw<LUT4> r = wr_fetch<LUT4>(a, sh.n_bits, blk, a.W + (long long)m * a.ldw + (long long)j * SOP_G);
  float c[16];
  wr_weights(a, j, c);
  wr_decode<LUT4>(a, F, sh, blk, r, c, E, met);
}

// the metric as a key whose ascending order is the metric's descending order (the metric is never negative;
// a NaN counts as zero)
__device__ __forceinline__ unsigned wr_key(float met) {
  return ~(met > 0.0f ? __float_as_uint(met) : 0u);
}

struct WrPick {
  unsigned long long warp[STB / 32];
  unsigned long long before;
  int bin;
  int last;
};

// Adds a CTA's histogram to the layer's; true in the CTA that comes last (all threads of the CTA call it).
__device__ __forceinline__ bool wr_flush(const unsigned* hist, unsigned* out, unsigned* done, WrPick& s) {
  __syncthreads();
  for (int i = threadIdx.x; i < 2048; i += STB)
    if (hist[i]) atomicAdd(&out[i], hist[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s.last = atomicAdd(done, 1u) + 1u == gridDim.x;
  __syncthreads();
  if (s.last) __threadfence();
  return s.last;
}

// The last CTA of a histogram kernel: the bin that holds the rank, the prefix and the rank inside it for the next
// pass; after the last pass the threshold itself.  Pass -1: the bin of the n_keep-th largest block maximum.  A rank
// beyond the histogram's total (no pair to correct, so the histogram is empty) leaves a NaN threshold: nothing
// compares >= to it.
__device__ void wr_pick(SparseWs* ws, int pass, long long n_keep, WrPick& s) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned long long rank = pass <= 0 ? (unsigned long long)n_keep : ws->rank;
  const unsigned prev = pass > 0 ? ws->prefix : 0u;
  const unsigned* h = (pass < 0 ? ws->hist_bm : ws->hist[pass]) + 8 * tid;     // pass 2 counts 1024 bins, the rest stays zero
  const uint4 h0 = __ldcg(reinterpret_cast<const uint4*>(h)), h1 = __ldcg(reinterpret_cast<const uint4*>(h) + 1);
  const unsigned b[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
  unsigned long long local = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) local += b[i];
  unsigned long long incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s.warp[warp] = incl;
  if (tid == 0) { s.bin = -1; s.before = 0; }
  __syncthreads();
  unsigned long long excl = incl - local;
  for (int w = 0; w < warp; ++w) excl += s.warp[w];
  if (local && excl < rank && rank <= excl + local) {
    int i = 0;
    while (rank > excl + b[i]) excl += b[i++];
    s.bin = 8 * tid + i; s.before = excl;
  }
  __syncthreads();
  if (tid == 0 && pass < 0) {
    // fewer blocks than entries to keep: no bound, every bin counts
    ws->bm_bin = s.bin < 0 ? 2047u : (unsigned)s.bin;
  } else if (tid == 0) {
    if (s.bin < 0) {
      ws->prefix = 0xFFFFFFFFu; ws->rank = 0; ws->tau_bits = 0x7FC00000u;
    } else {
      const unsigned pre = (prev << (pass < 2 ? 11 : 10)) | (unsigned)s.bin;
      ws->prefix = pre;
      ws->rank = rank - s.before;
      if (pass == 2) ws->tau_bits = ~pre;
    }
  }
}

// First decode pass.  A thread stays in its block column and steps down the rows (the grid's threads cover `rows` whole
// rows), so that the sixteen channel weights stay in registers; the next row's block is loaded before this one's
// arithmetic.
// What bounds it: instruction issue (67 % of the slots) beside 184 MB of DRAM traffic; 50 us at 8192 x 8192, 28 us of which the bytes need
// (82 us with a block per thread in storage order, weights re-read per block, and both tables in the same sixteen banks).
template <bool LUT4>
__global__ void __launch_bounds__(STB, LUT4 ? 4 : 2) wr_max_kernel(WrArgs a, AtomsDev A, FmtDev F, const sop_search_result* res,
                                                                   SparseWs* ws, unsigned rows) {
  pdl_trigger();
  __shared__ WrShared sh;
  __shared__ WrPick pk;
  __shared__ unsigned hist[2048];
  const int tid = threadIdx.x;
  for (int i = tid; i < 2048; i += STB) hist[i] = 0;
  pdl_wait();
  wr_setup(a, A, res, sh);
  __syncthreads();
  const unsigned nbk = (unsigned)a.nbk, NB = (unsigned)a.NB, S = rows * nbk;
  const unsigned t = blockIdx.x * STB + tid;
  if (t < S && !sh.no_pair) {
    const unsigned m0 = t / nbk, j = t - m0 * nbk;
    const uint16_t* wrow = a.W + (long long)m0 * a.ldw + (long long)j * SOP_G;
    const long long step = (long long)rows * a.ldw;
    const int n_bits = LUT4 ? 4 : sh.n_bits;
    float c[16];
    wr_weights(a, j, c);
    unsigned blk = t;
    WrRaw<LUT4> r = wr_fetch<LUT4>(a, n_bits, blk, wrow);        // rows <= M: the first block is there
    while (true) {
      const WrRaw<LUT4> cur = r;
      const unsigned at = blk;
      const bool more = S < NB && blk < NB - S;
      blk += S; wrow += step;
      if (more) r = wr_fetch<LUT4>(a, n_bits, blk, wrow);
      float E[16], met[16];
      wr_decode<LUT4>(a, F, sh, at, cur, c, E, met);
      float bm = 0.0f;
#pragma unroll
      for (int i = 0; i < 16; ++i) bm = fmaxf(bm, met[i]);       // fmaxf drops a NaN
      const unsigned bin = wr_key(bm) >> 21;
      a.kept[at] = (unsigned short)bin;
      // most blocks share a handful of bins: one addition per distinct bin of the warp
      const unsigned same = __match_any_sync(__activemask(), bin);
      if ((__ffs((int)same) - 1) == (tid & 31)) atomicAdd(&hist[bin], (unsigned)__popc(same));
      if (!more) break;
    }
  }
  if (wr_flush(hist, ws->hist_bm, &ws->done[0], pk)) wr_pick(ws, -1, a.n_keep, pk);
}

__device__ __forceinline__ bool wr_kept(float met, float tau) { return met >= tau && met > 0.0f; }

// The stored value of a residual: the E3M4 code (bias 3, 4 mantissa bits, largest 15.5) of E / 2^e.  The quotient is
// formed by two exact multiplications by powers of two (|E| / 2^e <= 15.5; a quotient below the fp32 normal range is
// far below half the smallest E3M4 step and rounds to zero either way).
struct WrValue {
  float f1, f2;
  GridDev g;
  __device__ explicit WrValue(int e) {
    const int e1 = max(-100, min(100, -e));
    f1 = pow2f_int(e1); f2 = pow2f_int(max(-120, min(120, -e - e1)));
    g.min_eb = 125; g.sh = 19; g.vpos = 15.5f; g.vneg = 15.5f;
  }
  __device__ __forceinline__ uint32_t code(float E) const {
    return grid_code(grid_quantize(__fmul_rn(__fmul_rn(E, f1), f2), g), g, 7);
  }
};

// The candidates.  A warp reads the bins of 1024 blocks, lists those that reach the bound and decodes them 32 at a time:
// a lane counts its block's candidates, the warp reserves room for all of them with one addition to the list's counter,
// every lane writes its own.  Beyond the capacity nothing is written; the counter keeps counting, which is how the
// overflow is seen.  The bins are replaced by zeros (the map of the kept entries starts empty), the tile counts as well.
// Reading the bins instead of decoding the layer once more: 22 us instead of 104 at 8192 x 8192 (30 MB instead of 176); the latency of
// the chain bins -> block -> list bounds it.
constexpr int WR_BPL = 32;               // blocks per lane and step
template <bool LUT4>
__global__ void __launch_bounds__(STB) wr_collect_kernel(WrArgs a, AtomsDev A, FmtDev F, const sop_search_result* res,
                                                         SparseWs* ws) {
  pdl_trigger();
  __shared__ WrShared sh;
  __shared__ WrPick pk;
  __shared__ unsigned hist[2048];
  __shared__ unsigned short s_list[STB / 32][32 * WR_BPL];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < 2048; i += STB) hist[i] = 0;
  pdl_wait();
  wr_setup(a, A, res, sh);
  __syncthreads();
  if (blockIdx.x == 0 && tid == 0) ws->no_pair = sh.no_pair;
  const unsigned bm_bin = ws->bm_bin, NB = (unsigned)a.NB;
  const unsigned n_tasks = (NB + 32 * WR_BPL - 1) / (32 * WR_BPL), n_tiles = (NB + STB - 1) / STB;
  for (unsigned task = blockIdx.x * (STB / 32) + warp; task < n_tasks; task += gridDim.x * (STB / 32)) {
    const unsigned b0 = task * (32 * WR_BPL);
    uint4 v[WR_BPL / 8];
    uint4* map = reinterpret_cast<uint4*>(a.kept + b0);          // the array is padded to 256 bytes
#pragma unroll
    for (int q = 0; q < WR_BPL / 8; ++q)
      if (b0 + (q * 32 + lane) * 8 < NB) v[q] = map[q * 32 + lane];
    unsigned hit = 0;                                            // bit 8 q + e: block (32 q + lane) 8 + e
#pragma unroll
    for (int q = 0; q < WR_BPL / 8; ++q) {
      const unsigned first = b0 + (q * 32 + lane) * 8;
      if (first < NB) {
        const unsigned u[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (((u[e >> 1] >> (16 * (e & 1))) & 0xFFFFu) <= bm_bin && first + e < NB) hit |= 1u << (8 * q + e);
        map[q * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (lane < 32 * WR_BPL / STB && b0 / STB + lane < n_tiles) a.tile_sums[b0 / STB + lane] = 0;
    if (sh.no_pair) continue;
    unsigned at = 0, total;
    {
      const unsigned mine = (unsigned)__popc(hit);
      unsigned incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
      }
      total = __shfl_sync(0xFFFFFFFFu, incl, 31);
      at = incl - mine;
    }
    for (unsigned rest = hit; rest; rest &= rest - 1u) {
      const int i = __ffs((int)rest) - 1;
      s_list[warp][at++] = (unsigned short)(((i >> 3) * 32 + lane) * 8 + (i & 7));
    }
    __syncwarp();
    for (unsigned r0 = 0; r0 < total; r0 += 32) {
      float E[16], met[16];
      unsigned in = 0, blk = 0;
      if (r0 + lane < total) {
        blk = b0 + s_list[warp][r0 + lane];
        wr_block<LUT4>(a, F, sh, blk, E, met);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const unsigned bin = wr_key(met[i]) >> 21;
          if (bin <= bm_bin) { in |= 1u << i; atomicAdd(&hist[bin], 1u); }
        }
      }
      const unsigned mine = (unsigned)__popc(in);
      unsigned incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
      }
      unsigned base = 0;
      if (lane == 31) base = atomicAdd(&ws->n_cand, incl);
      base = __shfl_sync(0xFFFFFFFFu, base, 31);
      unsigned to = base + incl - mine;
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if ((in >> i) & 1u) {
          if (to < a.cand_cap) {
            a.cand_pos[to] = blk * 16u + (unsigned)i;
            a.cand_e[to] = __float_as_uint(E[i]);
            a.cand_m[to] = __float_as_uint(met[i]);
          }
          ++to;
        }
    }
    __syncwarp();
  }
  if (wr_flush(hist, ws->hist[0], &ws->done[1], pk)) {
    if (tid == 0) ws->overflow = *(volatile unsigned*)&ws->n_cand > a.cand_cap ? 1u : 0u;
    wr_pick(ws, 0, a.n_keep, pk);
  }
}

// The second and third digit of the threshold: over the candidate list, or over the layer when it overflowed.
template <int PASS, bool LUT4>
__global__ void __launch_bounds__(STB) wr_select_kernel(WrArgs a, AtomsDev A, FmtDev F, const sop_search_result* res,
                                                        SparseWs* ws) {
  pdl_trigger();
  __shared__ WrShared sh;
  __shared__ WrPick pk;
  __shared__ unsigned hist[2048];
  const int tid = threadIdx.x;
  for (int i = tid; i < 2048; i += STB) hist[i] = 0;
  pdl_wait();
  const unsigned prefix = ws->prefix;
  auto add = [&](float met) {
    const unsigned key = wr_key(met);
    if (PASS == 1) { if ((key >> 21) == prefix) atomicAdd(&hist[(key >> 10) & 2047u], 1u); }
    else { if ((key >> 10) == prefix) atomicAdd(&hist[key & 1023u], 1u); }
  };
  if (!ws->overflow) {
    __syncthreads();
    const unsigned n = ws->n_cand;
    for (unsigned i = blockIdx.x * STB + tid; i < n; i += gridDim.x * STB) add(__uint_as_float(a.cand_m[i]));
  } else {
    wr_setup(a, A, res, sh);
    __syncthreads();
    if (!sh.no_pair)
      for (long long blk = (long long)blockIdx.x * STB + tid; blk < a.NB; blk += (long long)gridDim.x * STB) {
        float E[16], met[16];
        wr_block<LUT4>(a, F, sh, (unsigned)blk, E, met);
#pragma unroll
        for (int i = 0; i < 16; ++i) add(met[i]);
      }
  }
  if (wr_flush(hist, ws->hist[PASS], &ws->done[1 + PASS], pk)) wr_pick(ws, PASS, a.n_keep, pk);
}

// The kept candidates: their bit in the per-block masks (two blocks per 32-bit word), their tile's record count, the
// largest |E| among them.  After an overflow: the counts and the largest |E| from the layer.
template <bool LUT4>
__global__ void __launch_bounds__(STB) wr_mark_kernel(WrArgs a, AtomsDev A, FmtDev F, const sop_search_result* res,
                                                      SparseWs* ws) {
  pdl_trigger();
  __shared__ WrShared sh;
  __shared__ unsigned s_cnt;
  const int tid = threadIdx.x;
  pdl_wait();
  const float tau = __uint_as_float(ws->tau_bits);
  unsigned emax = 0;
  if (!ws->overflow) {
    const unsigned n = ws->n_cand;
    unsigned* map = reinterpret_cast<unsigned*>(a.kept);
    for (unsigned i = blockIdx.x * STB + tid; i < n; i += gridDim.x * STB) {
      const unsigned pos = a.cand_pos[i], e = a.cand_e[i];
      if (!wr_kept(__uint_as_float(a.cand_m[i]), tau)) continue;
      atomicOr(&map[pos >> 5], 1u << (pos & 31u));
      atomicAdd(&a.tile_sums[pos >> 12], 1u);          // a tile is 256 blocks of 16 elements
      emax = max(emax, e & 0x7FFFFFFFu);
    }
  } else {
    wr_setup(a, A, res, sh);
    __syncthreads();
    const long long n_tiles = (a.NB + STB - 1) / STB;
    for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
      if (tid == 0) s_cnt = 0;
      __syncthreads();
      const long long blk = tile * STB + tid;
      unsigned cnt = 0;
      if (blk < a.NB && !sh.no_pair) {
        float E[16], met[16];
        wr_block<LUT4>(a, F, sh, (unsigned)blk, E, met);
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (wr_kept(met[i], tau)) { ++cnt; emax = max(emax, __float_as_uint(fabsf(E[i]))); }
      }
      cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
      if ((tid & 31) == 0 && cnt) atomicAdd(&s_cnt, cnt);
      __syncthreads();
      if (tid == 0) a.tile_sums[tile] = s_cnt;
      __syncthreads();
    }
  }
  emax = __reduce_max_sync(0xFFFFFFFFu, emax);
  if ((tid & 31) == 0 && emax) atomicMax(&ws->emax_bits, emax);
}

// Bits of the map before `pos` inside its tile (4096 bits, a warp reads them in one go): `word` is the lane's 16 bytes.
__device__ __forceinline__ unsigned wr_bits_before(const uint4& v, unsigned pos, int lane) {
  const unsigned u[4] = {v.x, v.y, v.z, v.w};
  const int n = (int)(pos & 4095u) - 128 * lane;
  unsigned cnt = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int left = n - 32 * k;
    cnt += (unsigned)__popc(left >= 32 ? u[k] : left > 0 ? u[k] & ((1u << left) - 1u) : 0u);
  }
  return __reduce_add_sync(0xFFFFFFFFu, cnt);
}

// The records.  The kept entries of the list: a record's place is its tile's offset plus the map's bits before it, which
// a warp counts together; four entries' maps are in flight at once.  The row starts come from the map in the same way.
// 17 us at 8192 x 8192 with 67 thousand kept entries (64 us for a pass over the map that decodes the blocks with a kept entry), bounded by
// latency.
// After an overflow: every block is decoded and its entries are compared with the threshold.
template <bool LUT4>
__global__ void __launch_bounds__(STB) wr_write_kernel(WrArgs a, AtomsDev A, FmtDev F, const sop_search_result* res,
                                                       const SparseWs* ws) {
  pdl_trigger();
  __shared__ WrShared sh;
  __shared__ unsigned s_warp[STB / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  pdl_wait();
  const float tau = __uint_as_float(ws->tau_bits);
  const WrValue V(ws->scale_exp);
  if (!ws->overflow) {
    const unsigned n = ws->n_cand, nbk = (unsigned)a.nbk, wid = blockIdx.x * (STB / 32) + (tid >> 5), n_warps = gridDim.x * (STB / 32);
    for (unsigned m = wid; m < (unsigned)a.M; m += n_warps) {
      const unsigned b = m * nbk;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (lane * 8 < (b & 255u)) v = *(reinterpret_cast<const uint4*>(a.kept + (b & ~255u)) + lane);
      const unsigned base = a.tile_sums[b >> 8];
      const unsigned cnt = wr_bits_before(v, b * 16u, lane);
      if (lane == 0) a.row_start[m] = base + cnt;
    }
    for (unsigned i0 = wid * 32; i0 < n; i0 += n_warps * 32) {
      bool keep = false;
      unsigned pos = 0, rec = 0;
      if (i0 + lane < n) {
        pos = a.cand_pos[i0 + lane];
        const float e = __uint_as_float(a.cand_e[i0 + lane]);
        keep = wr_kept(__uint_as_float(a.cand_m[i0 + lane]), tau);
        const unsigned blk = pos >> 4;
        rec = ((blk % nbk) * SOP_G + (pos & 15u)) | (V.code(e) << 16);
      }
      const unsigned first = keep ? a.tile_sums[pos >> 12] : 0u;
      unsigned before = 0;
      for (unsigned rest = __ballot_sync(0xFFFFFFFFu, keep); rest; ) {
        int src[4];
        unsigned p[4];
        uint4 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          src[q] = rest ? __ffs((int)rest) - 1 : -1;
          rest &= rest - 1u;                                      // 0 stays 0
          p[q] = __shfl_sync(0xFFFFFFFFu, pos, src[q] & 31);
          v[q] = make_uint4(0u, 0u, 0u, 0u);
          if (src[q] >= 0 && 128u * lane < (p[q] & 4095u)) v[q] = *(reinterpret_cast<const uint4*>(a.kept + ((p[q] >> 4) & ~255u)) + lane);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const unsigned cnt = wr_bits_before(v[q], p[q], lane);
          if (lane == src[q]) before = cnt;
        }
      }
      if (keep && (long long)first + before < a.capacity) a.records[first + before] = rec;
    }
    return;
  }
  wr_setup(a, A, res, sh);
  __syncthreads();
  const long long n_tiles = (a.NB + STB - 1) / STB;
  for (long long tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const long long blk = tile * STB + tid;
    float E[16], met[16];
    unsigned keep = 0;
    long long m = 0, j = 0;
    if (blk < a.NB) {
      m = (long long)((unsigned)blk / (unsigned)a.nbk); j = blk - m * a.nbk;
      if (!sh.no_pair) {
        wr_block<LUT4>(a, F, sh, (unsigned)blk, E, met);
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (wr_kept(met[i], tau)) keep |= 1u << i;
      }
    }
    unsigned tot;
    const unsigned excl = cta_excl_scan((unsigned)__popc(keep), s_warp, &tot);
    if (blk >= a.NB) continue;
    unsigned pos = a.tile_sums[tile] + excl;
    if (j == 0) a.row_start[m] = pos;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if ((keep >> i) & 1u) {
        if ((long long)pos < a.capacity) a.records[pos] = (unsigned)(j * SOP_G + i) | (V.code(E[i]) << 16);
        ++pos;
      }
  }
}

}  // namespace sop

extern "C" {

int sop_opq_threshold(double q, int max_order, double* m_out) {
  if (!m_out) return SOP_ERR_NULL;
  if (!(q > 0.0 && q < 1.0) || max_order < 1) return SOP_ERR_RANGE;
  // (2 Phi(m) - 1)^M = q with 2 Phi(m) - 1 = erf(m / sqrt 2): solve erf(m / sqrt 2) = q^(1/M) by bisection
  const double target = exp(log(q) / (double)max_order);
  double lo = 0.0, hi = 16.0;
  for (int it = 0; it < 128; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (erf(mid * 0.70710678118654752440) < target) lo = mid; else hi = mid;
  }
  *m_out = 0.5 * (lo + hi);
  return SOP_OK;
}

int sop_opq_workspace(long long M, long long K, size_t* bytes) {
  if (!bytes) return SOP_ERR_NULL;
  if (M < 1 || K < 1 || (K % SOP_G) != 0 || M > (1ll << 31) / (K / SOP_G)) return SOP_ERR_SHAPE;
  const long long NB = M * (K / SOP_G);
  *bytes = sop::opq_local_off(NB) + (size_t)sop::sparse_tiles(NB) * sop::OPQ_LOCAL * 4;
  return SOP_OK;
}

int sop_opq_extract(const void* W_dev, long long M, long long K, long long ldw, int g, double m,
                    void* W_out_dev, long long ldo, unsigned* row_start_dev, unsigned* records_dev, long long capacity,
                    long long* count_dev, void* workspace_dev, size_t workspace_bytes, void* stream) {
  using namespace sop;
  if (!W_dev || !W_out_dev || !row_start_dev || !count_dev) return SOP_ERR_NULL;
  if (g != SOP_G || M < 1 || K < 1 || (K % SOP_G) != 0 || ldw < K || (ldw % 8) != 0 || ldo < K || (ldo % 8) != 0) return SOP_ERR_SHAPE;
  if (((uintptr_t)W_dev & 15u) || ((uintptr_t)W_out_dev & 15u)) return SOP_ERR_SHAPE;
  if (M > (1ll << 31) / (K / SOP_G) || K > 65536) return SOP_ERR_SHAPE;       // the record holds the column in 16 bits
  if (W_out_dev == W_dev) return SOP_ERR_RANGE;                               // the stream is written from the untouched input
  if (!(m > 0.0) || !(m < 1.0e6)) return SOP_ERR_RANGE;
  if (capacity < 0 || (capacity > 0 && !records_dev)) return SOP_ERR_NULL;
  size_t need = 0;
  sop_opq_workspace(M, K, &need);
  if (!workspace_dev || ((uintptr_t)workspace_dev & 255u) || workspace_bytes < need) return SOP_ERR_WORKSPACE;
  OpqArgs a;
  a.W = (const uint16_t*)W_dev; a.W_out = (uint16_t*)W_out_dev; a.M = M; a.K = K; a.ldw = ldw; a.ldo = ldo;
  a.nbk = K / SOP_G; a.NB = M * a.nbk; a.m2 = m * m;
  unsigned char* wsb = (unsigned char*)workspace_dev;
  a.tile_sums = (unsigned*)(wsb + sparse_tiles_off());
  a.masks = (unsigned short*)(wsb + sparse_masks_off(a.NB));
  a.local = (unsigned*)(wsb + opq_local_off(a.NB));
  a.row_start = row_start_dev; a.records = records_dev; a.capacity = capacity;
  cudaStream_t st = (cudaStream_t)stream;
  const long long n_tiles = sparse_tiles(a.NB);
  const long long cap = (long long)num_sms() * 8;
  const int grid = (int)(n_tiles < cap ? n_tiles : cap);
  int rc;
  if ((rc = profile_mark(SOP_PROFILE_OPQ, 0, st))) return rc;
  SOP_CUDA_TRY(launch(opq_mask_kernel, grid, STB, 0, st, a));
  SOP_CUDA_TRY(launch(tile_scan_kernel, 1, 1024, 0, st, a.tile_sums, n_tiles, row_start_dev, M, count_dev, (SparseWs*)workspace_dev, 0, nullptr, nullptr));
  SOP_CUDA_TRY(launch(opq_write_kernel, grid, STB, 0, st, a));
  SOP_CUDA_TRY(cudaGetLastError());
  if ((rc = profile_mark(SOP_PROFILE_OPQ, 1, st))) return rc;
  return SOP_OK;
}

int sop_wr_workspace(long long M, long long K, size_t* bytes) {
  if (!bytes) return SOP_ERR_NULL;
  if (M < 1 || K < 1 || (K % SOP_G) != 0 || M > (1ll << 31) / (K / SOP_G)) return SOP_ERR_SHAPE;
  const long long NB = M * (K / SOP_G);
  *bytes = sop::wr_cand_off(NB) + 3 * (((size_t)sop::wr_cand_cap(NB) * 4 + 255) & ~(size_t)255);
  return SOP_OK;
}

int sop_wr_extract(const void* W_dev, long long M, long long K, long long ldw, const float* c_dev, int g,
                   const sop_scale_fmt* fmt, const sop_atom* atoms, int n_atoms, const float* dd_lut_dev, unsigned dd_mask,
                   int index_a, int index_b, int k_mode, const sop_search_result* search_dev, int use_sign,
                   int container_bits, int word_sign_bits, const unsigned char* codes_dev, const unsigned char* words_dev,
                   long long n_keep, unsigned* row_start_dev, unsigned* records_dev, long long capacity,
                   long long* count_dev, int* scale_exp_dev, float* tau_dev, void* workspace_dev, size_t workspace_bytes,
                   void* stream) {
  using namespace sop;
  int rc = validate_layer(W_dev, M, K, ldw, c_dev, g);
  if (rc) return rc;
  if (!codes_dev || !words_dev || !row_start_dev || !count_dev || !scale_exp_dev) return SOP_ERR_NULL;
  if (K > 65536) return SOP_ERR_SHAPE;                                        // the record holds the column in 16 bits
  FmtDev F;
  if ((rc = validate_fmt(fmt, &F))) return rc;
  AtomsDev A;
  if ((rc = validate_atoms(atoms, n_atoms, dd_mask, dd_lut_dev, &A))) return rc;
  if (use_sign != 0 && use_sign != 1) return SOP_ERR_FORMAT;
  if (word_sign_bits != 0 && word_sign_bits != 1) return SOP_ERR_FORMAT;
  if (container_bits != 8 && container_bits != 12 && container_bits != 16) return SOP_ERR_FORMAT;
  const int meta = container_bits - word_sign_bits - fmt->exp_bits - fmt->man_bits;
  if (meta < 0 || (use_sign && !word_sign_bits)) return SOP_ERR_FORMAT;
  const bool from_result = index_a == SOP_PAIR_FROM_RESULT;
  if (from_result) {
    if (!search_dev) return SOP_ERR_NULL;
    if (index_b == SOP_NO_ATOM) return SOP_ERR_RANGE;
  } else {
    if (index_a < 0 || index_a >= n_atoms) return SOP_ERR_RANGE;
    if (index_b != SOP_NO_ATOM && (index_b < 0 || index_b >= n_atoms)) return SOP_ERR_RANGE;
    if (index_b != SOP_NO_ATOM && (atoms[index_a].n_bits != atoms[index_b].n_bits || atoms[index_a].kind != SOP_KIND_LUT ||
                                   atoms[index_b].kind != SOP_KIND_LUT)) return SOP_ERR_ALPHABET;
    if (use_sign && atoms[index_a].kind != SOP_KIND_LUT) return SOP_ERR_ALPHABET;
    if (atoms[index_a].kind == SOP_KIND_FP_GRID && (atoms[index_a].grid_exp_bits < 1 || atoms[index_a].n_bits > 8)) return SOP_ERR_ALPHABET;
  }
  if (index_b != SOP_NO_ATOM && meta < 1) return SOP_ERR_FORMAT;
  if (k_mode == SOP_K_FROM_RESULT) { if (!search_dev) return SOP_ERR_NULL; }
  else if (k_mode < -64 || k_mode > 64) return SOP_ERR_RANGE;
  bool need_wmax = false;
  for (int i = 0; i < n_atoms; ++i) need_wmax |= atoms[i].scope == 0;
  if (need_wmax && !search_dev) return SOP_ERR_NULL;
  if (((uintptr_t)codes_dev & 15u) || ((uintptr_t)words_dev & 3u)) return SOP_ERR_SHAPE;
  if (from_result) {
    int n_bits = 0;
    for (int i = 0; i < n_atoms; ++i)
      if (atoms[i].kind == SOP_KIND_LUT) { if (!n_bits) n_bits = atoms[i].n_bits; else if (atoms[i].n_bits != n_bits) return SOP_ERR_ALPHABET; }
    if (!n_bits) return SOP_ERR_ALPHABET;
  }
  if (n_keep < 1 || n_keep > M * K) return SOP_ERR_RANGE;
  if (capacity < 0 || (capacity > 0 && !records_dev)) return SOP_ERR_NULL;
  size_t need = 0;
  sop_wr_workspace(M, K, &need);
  if (!workspace_dev || ((uintptr_t)workspace_dev & 255u) || workspace_bytes < need) return SOP_ERR_WORKSPACE;

  WrArgs a;
  a.W = (const uint16_t*)W_dev; a.c = c_dev; a.M = M; a.K = K; a.ldw = ldw; a.nbk = K / SOP_G; a.NB = M * a.nbk;
  a.index_a = index_a; a.index_b = index_b; a.k_mode = k_mode; a.use_sign = use_sign;
  a.container_bits = container_bits; a.word_sign_bits = word_sign_bits; a.meta_bits = meta;
  a.codes = codes_dev; a.words = (const unsigned*)words_dev; a.n_keep = n_keep;
  unsigned char* wsb = (unsigned char*)workspace_dev;
  SparseWs* ws = (SparseWs*)workspace_dev;
  a.tile_sums = (unsigned*)(wsb + sparse_tiles_off());
  a.row_start = row_start_dev; a.records = records_dev; a.capacity = capacity;
  a.kept = (unsigned short*)(wsb + sparse_masks_off(a.NB));
  a.cand_cap = wr_cand_cap(a.NB);
  {
    const size_t one = ((size_t)a.cand_cap * 4 + 255) & ~(size_t)255;
    a.cand_pos = (unsigned*)(wsb + wr_cand_off(a.NB));
    a.cand_e = (unsigned*)(wsb + wr_cand_off(a.NB) + one);
    a.cand_m = (unsigned*)(wsb + wr_cand_off(a.NB) + 2 * one);
  }
  cudaStream_t st = (cudaStream_t)stream;
  const long long n_tiles = sparse_tiles(a.NB);
  const long long cap = (long long)num_sms() * 4;
  const int grid = (int)(n_tiles < cap ? n_tiles : cap);
  // wr_max_kernel: as many whole rows as the CTAs that fit the device at once have threads for
  const long long fit = cap * STB / a.nbk;
  const unsigned rows = (unsigned)(fit < 1 ? 1 : fit < M ? fit : M);
  const int mgrid = (int)((rows * a.nbk + STB - 1) / STB);
  // (a memset, not clear(), which ends the chain of early starts between the packer and the first decode pass: with clear() here a pass over
  // 8192 x 8192 with both streams takes 1078 us instead of 1056, in three comparisons.  Why has not been established; elsewhere clear() wins.)
  SOP_CUDA_TRY(cudaMemsetAsync(ws, 0, sizeof(SparseWs), st));
  if ((rc = profile_mark(SOP_PROFILE_WR, 0, st))) return rc;
  // both codebooks tables of at most 16 entries: the decode with constant shifts (a pair taken from a search result is
  // always a pair of tables, and n_bits is then the alphabet's)
  bool lut4 = true;
  if (from_result) {
    for (int i = 0; i < n_atoms; ++i)
      if (atoms[i].kind == SOP_KIND_LUT && atoms[i].n_bits != 4) lut4 = false;
  } else {
    lut4 = atoms[index_a].kind == SOP_KIND_LUT && atoms[index_a].n_bits == 4 &&
           (index_b == SOP_NO_ATOM || (atoms[index_b].kind == SOP_KIND_LUT && atoms[index_b].n_bits == 4));
  }
#define SOP_WR_LAUNCHES(L4)                                                                             \
  do {                                                                                                  \
    SOP_CUDA_TRY(launch(wr_max_kernel<L4>, mgrid, STB, 0, st, a, A, F, search_dev, ws, rows));          \
    SOP_CUDA_TRY(launch(wr_collect_kernel<L4>, grid, STB, 0, st, a, A, F, search_dev, ws));             \
    SOP_CUDA_TRY(launch(wr_select_kernel<1, L4>, grid, STB, 0, st, a, A, F, search_dev, ws));           \
    SOP_CUDA_TRY(launch(wr_select_kernel<2, L4>, grid, STB, 0, st, a, A, F, search_dev, ws));           \
    SOP_CUDA_TRY(launch(wr_mark_kernel<L4>, grid, STB, 0, st, a, A, F, search_dev, ws));                \
    SOP_CUDA_TRY(launch(tile_scan_kernel, 1, 1024, 0, st, a.tile_sums, n_tiles, row_start_dev, M, count_dev, ws, 1, scale_exp_dev, tau_dev)); \
    SOP_CUDA_TRY(launch(wr_write_kernel<L4>, grid, STB, 0, st, a, A, F, search_dev, ws));               \
  } while (0)
  if (lut4) SOP_WR_LAUNCHES(true); else SOP_WR_LAUNCHES(false);
#undef SOP_WR_LAUNCHES
  SOP_CUDA_TRY(cudaGetLastError());
  if ((rc = profile_mark(SOP_PROFILE_WR, 1, st))) return rc;
  return SOP_OK;
}

}  // extern "C"
