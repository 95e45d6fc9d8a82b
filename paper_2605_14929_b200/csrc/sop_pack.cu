// sop_pack: materialise the chosen codebook(s): per block the best of the (up to four) candidates -- read off
// the per-block cosines of the sweep where they are given, else re-evaluated with the same arithmetic -- is
// encoded: 2n bytes of codes plus one b-bit scale word (sign, exponent, mantissa, selector).  Reads W once,
// writes ~n/8 + b/128 bytes per element; bound by instruction issue (the encode), not by bytes.  Table codes
// come from a uniform cell grid on u where the table allows it, else from a binary search over the thresholds.
// pack_winner_kernel serves choices whose cosines or errors a sweep has written; pack_kernel evaluates the candidates itself.
#include <string.h>

#include "sop_device.cuh"

namespace sop {

constexpr int PTB = 256;

struct PackArgs {
  const uint16_t* W;
  const float* c;
  long long M, K, ldw, nbk, NB;
  int index_a, index_b, k_mode, use_sign;
  int container_bits, word_sign_bits, meta_bits;
  unsigned char* codes;
  unsigned* words;       // zeroed before the kernel; filled with atomicOr
  unsigned long long* counts;
  const float* block_cos;   // optional [n_atoms x NB]: per-block cosines (or errors, with select_err) of an earlier sweep
  int select_err;           // 1: the smallest block error wins instead of the largest block cosine
  int cos_neg_a, cos_neg_b; // rows of the negated variants of index_a / index_b (-1: unknown, evaluate instead)
};

constexpr int KIND_LUT16 = 100;   // inside this file: a LUT of at most 16 entries (a four-step search is enough)
constexpr int KIND_LUT_CELL = 101; // inside this file: a LUT whose codes come from a uniform cell grid on u (one look-up, one compare)
constexpr int CELL_ROWS_MAX = 1025;
constexpr float CELL_MAGIC = 12582912.0f;   // 1.5 * 2^23: adding it leaves rint(x) in the low mantissa bits

// cell grid of a table: cell = rint(u * invh) + c_half, clamped to [0, 2 c_half]
struct PackCand { int table; int kind; int neg; int scope; int k; float tmax; GridDev grid; int sign_pos; float invh; int c_half; };

// One candidate on one block, everything in registers; same operation order as the sweep kernel.
// The 16 codes come back as bytes, four per word (element i in byte i % 4 of word i / 4).
// METRIC: 1 = with the block cosine, 2 = with the block squared error (in cos_out).
template <int METRIC, int KIND>
__device__ __forceinline__ void eval_block_kind(const float (&w)[16], const float (&c)[16], const float* tau,
                                                const float* lutv, int neg, float rcp, float s_hat,
                                                float& cos_out, uint32_t (&code4)[4], const GridDev grid = GridDev(), int sign_pos = 0,
                                                const uint2* cells = nullptr, float invh = 0.0f, int c_half = 0) {
  float qn[4], qd[4], qw[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float an = 0.0f, ad = 0.0f, aw = 0.0f;
    uint32_t packed = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = 4 * h + r;
      const float u = __fmul_rn(w[i], rcp);
      float q;
      uint32_t code;
      if (KIND == KIND_LUT_CELL) {
        // the cell holds at most one decision threshold: the code is the number of thresholds below the cell, plus one
        // when u lies above the cell's own threshold (+inf when it has none)
        const float uu = neg ? -u : u;
        const float t = fminf(fmaxf(__fmaf_rn(uu, invh, CELL_MAGIC + (float)c_half), CELL_MAGIC), CELL_MAGIC + (float)(2 * c_half));
        const uint2 e = cells[__float_as_uint(t) - __float_as_uint(CELL_MAGIC)];
        code = e.y + (uu > __uint_as_float(e.x) ? 1u : 0u);
        q = neg ? -lutv[code] : lutv[code];
      } else if (KIND == SOP_KIND_LUT || KIND == KIND_LUT16) {
        code = (uint32_t)(KIND == KIND_LUT16 ? count_below<4>(tau, neg ? -u : u) : count_below<5>(tau, neg ? -u : u));
        q = neg ? -lutv[code] : lutv[code];
      } else if (KIND == SOP_KIND_FP_E2M3) {
        q = fp_quantize<SOP_KIND_FP_E2M3>(u);
        code = fp_code<SOP_KIND_FP_E2M3>(q);
      } else if (KIND == SOP_KIND_FP_GRID) {
        q = grid_quantize(u, grid);
        code = grid_code(q, grid, sign_pos);      // at most 8 bits: the host refuses wider grids here
      } else {
        q = fp_quantize<SOP_KIND_FP_E4M3>(u);
        code = fp_code<SOP_KIND_FP_E4M3>(q);
      }
      packed |= code << (8 * r);
      if (METRIC == 1) {
        const float cw = __fmul_rn(c[i], w[i]);
        const float cq = __fmul_rn(c[i], q);
        aw = __fmaf_rn(cw, w[i], aw);
        ad = __fmaf_rn(cq, w[i], ad);
        an = __fmaf_rn(cq, q, an);
      } else {
        const float e = __fmaf_rn(-s_hat, q, w[i]);     // w - s q with one rounding, as the sweep forms it
        an = __fmaf_rn(e, e, an);
      }
    }
    qn[h] = an; qd[h] = ad; qw[h] = aw;
    code4[h] = packed;
  }
  cos_out = METRIC == 1 ? block_cosine(quad_tree(qw), quad_tree(qn), quad_tree(qd)) : quad_tree(qn);
}

// the quantiser kind is decided once per block, outside the element loops: a kind test inside them lets
// the compiler hoist the FP-grid arithmetic into the table path
template <int METRIC>
__device__ __forceinline__ void eval_block_regs(const float (&w)[16], const float (&c)[16], const float* tau,
                                                const float* lutv, int kind, int neg, float rcp, float s_hat,
                                                float& cos_out, uint32_t (&code4)[4], const GridDev grid, int sign_pos,
                                                const uint2* cells, float invh, int c_half) {
  if (kind == KIND_LUT_CELL) eval_block_kind<METRIC, KIND_LUT_CELL>(w, c, tau, lutv, neg, rcp, s_hat, cos_out, code4, grid, sign_pos, cells, invh, c_half);
  else if (kind == KIND_LUT16) eval_block_kind<METRIC, KIND_LUT16>(w, c, tau, lutv, neg, rcp, s_hat, cos_out, code4);
  else if (kind == SOP_KIND_LUT) eval_block_kind<METRIC, SOP_KIND_LUT>(w, c, tau, lutv, neg, rcp, s_hat, cos_out, code4);
  else if (kind == SOP_KIND_FP_GRID) eval_block_kind<METRIC, SOP_KIND_FP_GRID>(w, c, tau, lutv, neg, rcp, s_hat, cos_out, code4, grid, sign_pos);
  else if (kind == SOP_KIND_FP_E2M3) eval_block_kind<METRIC, SOP_KIND_FP_E2M3>(w, c, tau, lutv, neg, rcp, s_hat, cos_out, code4);
  else eval_block_kind<METRIC, SOP_KIND_FP_E4M3>(w, c, tau, lutv, neg, rcp, s_hat, cos_out, code4);
}

// Every candidate of the choice is evaluated here.
__global__ void __launch_bounds__(PTB, 1) pack_kernel(PackArgs a, AtomsDev A, FmtDev F, const sop_search_result* res) {
  pdl_trigger();
  pdl_wait();
  __shared__ float lutv[2][32], tau[2][32];
  __shared__ uint2 cells[2][CELL_ROWS_MAX];       // per table and cell: {the cell's threshold (+inf: none), thresholds below the cell}
  __shared__ PackCand base[2];
  __shared__ int s_nb, s_nbits;
  __shared__ float s_pot[2];
  __shared__ unsigned s_cnt[2];
  __shared__ int s_idx[2];   // the two atoms
  __shared__ int s_no_pair;  // the search result holds no pair to pack
  const int tid = threadIdx.x;
  if (tid == 0) {
    int ia = a.index_a, ib = a.index_b;
    const bool from_result = ia == SOP_PAIR_FROM_RESULT;
    if (ia == SOP_PAIR_FROM_RESULT) {
      ia = a.use_sign ? res->best_sa : res->best_a;
      ib = a.use_sign ? res->best_sb : res->best_b;
    }
    // a result without a pair (singles-only search, no signed table, one base atom): nothing is packed and the
    // counts say so; with use_sign the second atom of each must exist too (the negation follows its atom)
    s_no_pair = from_result && (ia < 0 || ib < 0 || ia >= A.n_atoms || ib >= A.n_atoms ||
                                (a.use_sign && (ia + 1 >= A.n_atoms || ib + 1 >= A.n_atoms))) ? 1 : 0;
    ia = max(0, min(A.n_atoms - 1, ia));
    int nb = 1;
    if (ib != SOP_NO_ATOM) { ib = max(0, min(A.n_atoms - 1, ib)); nb = 2; }
    s_nb = nb;
    s_nbits = A.atoms[ia].n_bits;
    const float wmax = res ? res->layer_absmax : 0.0f;
    for (int t = 0; t < nb; ++t) {
      const int idx = t ? ib : ia;
      const sop_atom& at = A.atoms[idx];
      base[t].table = t; base[t].kind = (at.kind == SOP_KIND_LUT && at.n_entries <= 16) ? KIND_LUT16 : at.kind; base[t].neg = at.negated; base[t].scope = at.scope; base[t].tmax = at.tmax;
      base[t].k = a.k_mode == SOP_K_FROM_RESULT ? res->k[idx] : a.k_mode;
      base[t].grid.min_eb = 128 - at.grid_bias; base[t].grid.sh = 23 - at.grid_man_bits;
      base[t].grid.vpos = at.tmax; base[t].grid.vneg = at.grid_neg_max;
      base[t].sign_pos = at.grid_exp_bits + at.grid_man_bits;
      base[t].invh = 0.0f; base[t].c_half = 0;
      s_pot[t] = at.scope == 0 ? layer_pot_scale(wmax, at.tmax) : 0.0f;
      s_idx[t] = idx;
    }
    s_cnt[0] = s_cnt[1] = 0;
  }
  __syncthreads();
  if (s_no_pair) {
    if (a.counts && blockIdx.x == 0 && tid < 2) a.counts[tid] = ~0ull;     // {-1, -1}
    return;
  }
  const int nb = s_nb, n = s_nbits, b = a.container_bits;
  // table values and decision thresholds of the (up to two) tables: one thread per entry
  if (tid < 32 * nb) {
    const int t = tid >> 5, j = tid & 31, idx = s_idx[t];
    const sop_atom& at = A.atoms[idx];
    const bool dd = (A.dd_mask >> idx) & 1u;
    const int ne = at.kind == SOP_KIND_LUT ? at.n_entries : 2;
    lutv[t][j] = at.kind == SOP_KIND_LUT ? (dd ? A.dd_lut[min(j, ne - 1)] : at.lut[min(j, ne - 1)]) : 0.0f;
    __syncwarp();
    tau[t][j] = table_threshold(lutv[t], j, ne);
  }
  __syncthreads();
  // Cell grids of the tables.  A grid of width h <= (smallest gap between two thresholds) / 2 puts at most one threshold
  // into a cell's closed interval [(k - 1/2) h, (k + 1/2) h]; the first and last cells lie beyond every threshold.  A
  // table with repeated thresholds, or one that would need more than CELL_ROWS_MAX cells, keeps the binary search.
  if (tid < nb) {
    const int t = tid;
    PackCand cd = base[t];
    const int ne = A.atoms[s_idx[t]].kind == SOP_KIND_LUT ? A.atoms[s_idx[t]].n_entries : 0;
    if (ne >= 2) {
      float gap = __int_as_float(0x7F800000), reach = 0.0f;
      bool ok = true;
      for (int j = 0; j < ne - 1; ++j) {
        reach = fmaxf(reach, fabsf(tau[t][j]));
        if (j + 1 < ne - 1) {
          const float g = __fsub_rn(tau[t][j + 1], tau[t][j]);
          if (!(g > 0.0f)) ok = false;
          gap = fminf(gap, g);
        }
      }
      if (ne == 2) gap = 1.0f;
      if (ok && gap > 0.0f && reach < 1.0e6f) {
        const int eh = ilogb_pos(gap) - 1;                       // h = 2^eh <= gap / 2
        if (eh >= -20 && eh <= 20) {
          const float h = pow2f_int(eh);
          const float rows_half = ceilf(__fdiv_rn(reach, h)) + 1.0f;
          if (2.0f * rows_half + 1.0f <= (float)CELL_ROWS_MAX) {
            cd.invh = pow2f_int(-eh);
            cd.c_half = (int)rows_half;
            cd.kind = KIND_LUT_CELL;
          }
        }
      }
    }
    base[t] = cd;
  }
  __syncthreads();
  for (int t = 0; t < nb; ++t) {
    if (base[t].kind != KIND_LUT_CELL) continue;
    const int ch = base[t].c_half, ne = A.atoms[s_idx[t]].n_entries;
    const float h = __fdiv_rn(1.0f, base[t].invh);
    for (int r = tid; r <= 2 * ch; r += PTB) {
      const float lo = __fmul_rn((float)(r - ch) - 0.5f, h), hi = __fmul_rn((float)(r - ch) + 0.5f, h);   // exact: small integers and halves times a power of two
      unsigned below = 0;
      float thr = __int_as_float(0x7F800000);
      for (int j = 0; j < ne - 1; ++j) {
        const float tj = tau[t][j];
        if (r > 0 && tj < lo) ++below;
        else if (r == 2 * ch || tj <= hi) thr = fminf(thr, tj);
      }
      cells[t][r] = make_uint2(__float_as_uint(thr), below);
    }
  }
  __syncthreads();

  const int n_sign = a.use_sign ? 2 : 1;
  unsigned my_sel = 0, my_neg = 0;
  const unsigned nbk32 = (unsigned)a.nbk, NB32 = (unsigned)a.NB;       // the block count fits 31 bits
  // the weights of a block are loaded one iteration ahead
  auto fetch = [&](unsigned blk, uint4& v0, uint4& v1) {
    const unsigned m = blk / nbk32, j = blk - m * nbk32;
    const uint4* p = reinterpret_cast<const uint4*>(a.W + (long long)m * a.ldw + (long long)j * SOP_G);
    v0 = *p; v1 = p[1];
  };
  const unsigned stride = gridDim.x * PTB;
  uint4 nv0 = make_uint4(0u, 0u, 0u, 0u), nv1 = nv0;
  if (blockIdx.x * PTB + tid < NB32) fetch(blockIdx.x * PTB + tid, nv0, nv1);
  for (unsigned blk = blockIdx.x * PTB + tid; blk < NB32; blk += stride) {
    const unsigned j = blk % nbk32;
    const uint4 v0 = nv0, v1 = nv1;
    if (blk + stride < NB32) fetch(blk + stride, nv0, nv1);
    const uint32_t wb[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
    float w[16], c[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) { w[2 * i] = bf16lo(wb[i]); w[2 * i + 1] = bf16hi(wb[i]); }
    const float4* cp = reinterpret_cast<const float4*>(a.c + j * SOP_G);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 v = cp[q];
      c[4 * q] = v.x; c[4 * q + 1] = v.y; c[4 * q + 2] = v.z; c[4 * q + 3] = v.w;
    }
    // bf16 magnitudes order like their bit patterns: the maximum of the sixteen 15-bit patterns, two per word at a time
    uint32_t mb = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) mb = __vmaxu2(mb, wb[q] & 0x7FFF7FFFu);
    mb = max(mb & 0xFFFFu, mb >> 16);
    const float amax = __uint_as_float(mb << 16);
    float best_cos = 0.0f;
    uint32_t best_scode = 0, best4[4] = {0u, 0u, 0u, 0u};
    int pick = -1;
    for (int t = 0; t < nb; ++t) {
      const PackCand cd = base[t];
      float s_hat;
      uint32_t sc = 0;
      if (cd.scope == 0) {
        s_hat = amax > 0.0f ? s_pot[t] : 0.0f;
      } else {
        const float sigma = cd.tmax == 1.0f ? amax : __fdiv_rn(amax, cd.tmax);
        const QScale qs = scale_quantize(sigma, cd.k, F);
        s_hat = qs.s_hat;
        sc = qs.code;
      }
      const float rcp = s_hat > 0.0f ? __frcp_rn(s_hat) : 0.0f;
      for (int sg = 0; sg < n_sign; ++sg) {
        float cs;
        uint32_t c4[4];
        if (a.select_err) eval_block_regs<2>(w, c, tau[t], lutv[t], cd.kind, sg ? 1 - cd.neg : cd.neg, rcp, s_hat, cs, c4, cd.grid, cd.sign_pos, cells[t], cd.invh, cd.c_half);
        else eval_block_regs<1>(w, c, tau[t], lutv[t], cd.kind, sg ? 1 - cd.neg : cd.neg, rcp, s_hat, cs, c4, cd.grid, cd.sign_pos, cells[t], cd.invh, cd.c_half);
        if (pick < 0 || (a.select_err ? cs < best_cos : cs > best_cos)) {
          best_cos = cs; best_scode = sc; pick = 2 * t + sg;
#pragma unroll
          for (int h = 0; h < 4; ++h) best4[h] = c4[h];
        }
      }
    }
    const unsigned sel = pick >> 1, sgn = pick & 1;
    my_sel += sel; my_neg += sgn;
    // codes: 16 n-bit fields, little-endian, 2n bytes
    unsigned long long lo = 0, hi = 0;   // 128-bit accumulator
    if (n == 4) {
      uint32_t h16[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const uint32_t y = (best4[h] | (best4[h] >> 4)) & 0x00FF00FFu;   // bytes 0 and 2 hold two codes each
        h16[h] = (y | (y >> 8)) & 0xFFFFu;
      }
      lo = (unsigned long long)(h16[0] | (h16[1] << 16)) | ((unsigned long long)(h16[2] | (h16[3] << 16)) << 32);
    } else
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int pos = i * n;
      const unsigned long long v = (unsigned long long)((best4[i >> 2] >> (8 * (i & 3))) & 0xFFu);
      if (pos < 64) {
        lo |= v << pos;
        if (pos + n > 64) hi |= v >> (64 - pos);
      } else {
        hi |= v << (pos - 64);
      }
    }
    unsigned short* dst = reinterpret_cast<unsigned short*>(a.codes + (size_t)blk * 2 * n);
    if (n == 4) {
      *reinterpret_cast<uint2*>(dst) = make_uint2((unsigned)lo, (unsigned)(lo >> 32));
    } else if (n == 8) {
      *reinterpret_cast<uint4*>(dst) = make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
    } else {
      for (int i = 0; i < n; ++i) dst[i] = (unsigned short)((i < 4 ? lo >> (16 * i) : hi >> (16 * (i - 4))) & 0xFFFFu);
    }
    // scale word
    unsigned word;
    if (a.word_sign_bits) word = (sgn << (b - 1)) | (best_scode << a.meta_bits) | (a.meta_bits >= 1 ? sel : 0u);
    else if (a.meta_bits >= 1) word = (sel << (b - 1)) | (best_scode << (a.meta_bits - 1));
    else word = best_scode;
    const long long bit = (long long)blk * b;
    const long long wi = bit >> 5;
    const int sh = (int)(bit & 31);
    if (b == 16) {
      reinterpret_cast<unsigned short*>(a.words)[blk] = (unsigned short)word;
    } else if (b == 8) {
      reinterpret_cast<unsigned char*>(a.words)[blk] = (unsigned char)word;
    } else if (word) {
      atomicOr(&a.words[wi], word << sh);
      if (sh + b > 32) atomicOr(&a.words[wi + 1], word >> (32 - sh));
    }
  }
  if (a.counts) {
    atomicAdd(&s_cnt[0], my_sel);
    atomicAdd(&s_cnt[1], my_neg);
    __syncthreads();
    if (tid < 2 && s_cnt[tid]) atomicAdd(&a.counts[tid], (unsigned long long)s_cnt[tid]);
  }
}

// ---------------------------------------------------------------------------------------------
// The packer where the winner of each block can be read off a sweep's values: only the winner is encoded.
//   Table codes: a uniform grid of PCELLS cells on u; a cell's entry holds its one threshold and the codes below and above it, so an
//   element costs a look-up, a comparison and a byte permutation.  Entries are stored eight times (lanes l, l + 8, ... share a copy).
//   A table with two different thresholds in one cell is searched instead.
//   E2M3 and E4M3 codes are what the conversion instructions return.
//   The codes of a block leave as whole 32-bit words wherever 16 n bits (of two blocks for odd n) are a multiple of 32; 12-bit scale
//   words are gathered eight blocks at a time by shuffles.
// What bounds it: instruction issue (70 to 74 % of the slots) with the shared-memory wavefronts of the grid look-ups (63 %) close behind;
// 230 MB of DRAM traffic would take 35 us at 8192 x 8192, where it takes 76 us (the general kernel: 95 us).  The whole
// pass over 14336 x 4096 in E2M3 fell from 288 to 201 us with it, of which 10 us come from code width and candidate count being template
// parameters.
// ---------------------------------------------------------------------------------------------
constexpr int PCELLS = 320, PCOPIES = 8;
constexpr float PMAGIC = 12582912.0f;   // 1.5 * 2^23: adding it leaves rint(x) in the low mantissa bits

struct PackTable {       // of each of the two atoms
  float tmax, pot, inv_range;
  int neg, k, slow, block_scope;
  unsigned fast_lo, fast_span;         // patterns of sigma that take the one-addition rounding (see scale_quantize)
  unsigned code_off;                   // scale code = (rounded pattern >> (23 - y)) - code_off there
};

__device__ __forceinline__ unsigned pack_cell(float u, float inv_range) {
  return __float_as_uint(__fmaf_rn(__saturatef(__fmaf_rn(u, inv_range, 0.5f)), (float)PCELLS, PMAGIC));      // cell number + bits of PMAGIC
}

// KIND: SOP_KIND_LUT (any pair or single table), SOP_KIND_FP_E2M3, SOP_KIND_FP_E4M3 or SOP_KIND_FP_GRID (a single format).  N: bits of a code (0: as the
// atom says).  NC: candidates of the choice, 1, 2 (a pair, or a table and its negation) or 4.
template <int KIND, int N, int NC>
__global__ void __launch_bounds__(PTB, 4) pack_winner_kernel(PackArgs a, AtomsDev A, FmtDev F, const sop_search_result* res) {
  constexpr bool LUT = KIND == SOP_KIND_LUT;
  __shared__ __align__(16) uint2 cells[LUT ? 2 * (PCELLS + 1) * PCOPIES : 1];      // {threshold, code below | code above << 8}
  __shared__ float tau[2][32], lutv[2][32];
  __shared__ unsigned short tcell[2][32];
  __shared__ PackTable tab[2];
  __shared__ int s_idx[2], s_row[4];
  __shared__ unsigned s_cnt[2];
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31;
  // the pair (as pack_kernel resolves it)
  int ia = a.index_a, ib = a.index_b;
  const bool from_result = ia == SOP_PAIR_FROM_RESULT;
  if (from_result) {
    ia = a.use_sign ? res->best_sa : res->best_a;
    ib = a.use_sign ? res->best_sb : res->best_b;
    if (ia < 0 || ib < 0 || ia >= A.n_atoms || ib >= A.n_atoms || (a.use_sign && (ia + 1 >= A.n_atoms || ib + 1 >= A.n_atoms))) {
      if (a.counts && blockIdx.x == 0 && tid < 2) a.counts[tid] = ~0ull;     // {-1, -1}: the result holds no pair
      // the words as the other packer leaves them: a stream of 12-bit words cleared, else the last 32 bits
      const unsigned long long n_words = ((unsigned long long)a.NB * (unsigned)a.container_bits + 31ull) / 32ull;
      unsigned long long i = (unsigned long long)blockIdx.x * PTB + (unsigned)tid;
      if (a.container_bits != 12) i += n_words - 1ull;
      for (; i < n_words; i += (unsigned long long)gridDim.x * PTB) a.words[i] = 0u;
      return;
    }
  }
  const int nb = ib == SOP_NO_ATOM ? 1 : 2;
  const int n = N ? N : A.atoms[ia].n_bits, b = a.container_bits;
  if (tid < 2) {
    s_cnt[tid] = 0;
    const int idx = tid && nb == 2 ? ib : ia;
    s_idx[tid] = idx;
    const sop_atom& at = A.atoms[idx];
    PackTable t;
    t.tmax = at.tmax; t.neg = at.negated; t.block_scope = at.scope != 0; t.slow = 0;
    t.k = a.k_mode == SOP_K_FROM_RESULT ? res->k[idx] : a.k_mode;
    t.pot = at.scope == 0 ? layer_pot_scale(res->layer_absmax, at.tmax) : 0.0f;
    t.inv_range = __fdiv_rn(0.4f, at.tmax);                          // the cells cover |u| <= 1.25 tmax, the end cells everything beyond
    const int e0 = max(F.emin + 127 - t.k, 4), e1 = min(F.emax + 127 - t.k, 250);      // normal, below the top binade, reciprocal normal
    const bool ok = F.y >= 1 && e1 > e0;
    t.fast_lo = ok ? (unsigned)e0 << 23 : 0u;
    t.fast_span = ok ? (unsigned)(e1 - e0) << 23 : 0u;
    t.code_off = (unsigned)(127 - t.k - F.bias) << F.y;               // (modulo 2^32)
    tab[tid] = t;
    // from a search result with signs, a and b are base atoms and each is followed by its negation
    s_row[2 * tid] = idx;
    s_row[2 * tid + 1] = from_result ? idx + 1 : (tid ? a.cos_neg_b : a.cos_neg_a);
  }
  if (LUT) {
    __syncthreads();
    if (tid < 64) {
      const int t = tid >> 5, j = tid & 31, idx = s_idx[t], ne = A.atoms[idx].n_entries;
      lutv[t][j] = ((A.dd_mask >> idx) & 1u) ? A.dd_lut[min(j, ne - 1)] : A.atoms[idx].lut[min(j, ne - 1)];
      __syncwarp();
      const float x = table_threshold(lutv[t], j, ne);
      tau[t][j] = x;
      const unsigned c = x < __int_as_float(0x7F800000) ? pack_cell(x, tab[t].inv_range) - __float_as_uint(PMAGIC) : 0xFFFFu;
      tcell[t][j] = (unsigned short)c;
      __syncwarp();
      if (j < 31 && c != 0xFFFFu && c == tcell[t][j + 1] && tau[t][j + 1] != x) tab[t].slow = 1;
    }
    __syncthreads();
    for (int i = tid; i < nb * (PCELLS + 1); i += PTB) {
      const int t = i / (PCELLS + 1), c = i - t * (PCELLS + 1);
      int lo = 0, hi = 0;                    // thresholds in lower cells; in this cell or lower ones
#pragma unroll
      for (int step = 16; step >= 1; step >>= 1) {
        if ((int)tcell[t][lo + step - 1] < c) lo += step;
        if ((int)tcell[t][hi + step - 1] <= c) hi += step;
      }
      const uint2 e = make_uint2(__float_as_uint(hi > lo ? tau[t][lo] : __int_as_float(0x7F800000)), (unsigned)lo | ((unsigned)hi << 8));
      for (int x = 0; x < PCOPIES; ++x) cells[i * PCOPIES + ((x + i) & (PCOPIES - 1))] = e;      // (neighbouring threads in different banks)
    }
  }
  __syncthreads();

  const bool signs = NC == 4 || (NC == 2 && a.use_sign);      // the candidates are a table and its negation, once or twice
  const unsigned nbk = (unsigned)a.nbk, NB = (unsigned)a.NB;       // the block count fits 31 bits
  const bool packed_rows = a.ldw == a.K;
  GridDev grid = {};
  int sign_pos = 0;
  if (KIND == SOP_KIND_FP_GRID) {
    const sop_atom& at = A.atoms[ia];
    grid.min_eb = 128 - at.grid_bias; grid.sh = 23 - at.grid_man_bits; grid.vpos = at.tmax; grid.vneg = at.grid_neg_max;
    sign_pos = at.grid_exp_bits + at.grid_man_bits;
  }
  const unsigned flip = a.select_err ? 0x80000000u : 0u;      // errors are compared as their negatives
  const float* row[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) row[q] = a.block_cos + (size_t)s_row[signs ? q : 2 * q] * a.NB;
  const int sh = 23 - F.y;
  const unsigned half = (1u << (sh - 1)) - 1u, mask = (1u << sh) - 1u;
  unsigned my_sel = 0, my_neg = 0;
  // the loads of a block are issued one iteration ahead; whole warps run (the shuffles need them), lanes beyond the last block idle
  uint4 nv0, nv1;
  float ncs[NC];
  auto fetch = [&](unsigned blk) {
    nv0 = nv1 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int q = 0; q < NC; ++q) ncs[q] = 0.0f;
    if (blk < NB) {
      const uint16_t* p = a.W + (size_t)blk * SOP_G;
      if (!packed_rows) { const unsigned m = blk / nbk; p = a.W + (long long)m * a.ldw + (long long)(blk - m * nbk) * SOP_G; }
      nv0 = *reinterpret_cast<const uint4*>(p); nv1 = *(reinterpret_cast<const uint4*>(p) + 1);
      if (NC > 1) {
#pragma unroll
        for (int q = 0; q < NC; ++q) ncs[q] = __uint_as_float(__float_as_uint(row[q][blk]) ^ flip);
      }
    }
  };
  const unsigned stride = gridDim.x * PTB;
  const unsigned base0 = blockIdx.x * PTB + (unsigned)(tid & ~31);
  fetch(base0 + lane);
#pragma unroll 1
  for (unsigned base = base0; base < NB; base += stride) {
    const unsigned blk = base + lane;
    const bool on = blk < NB;
    uint32_t wb[8] = {nv0.x, nv0.y, nv0.z, nv0.w, nv1.x, nv1.y, nv1.z, nv1.w};
    // the winner in the priority order a, (-a), b, (-b): ties keep the earlier
    int pick = 0;
    float best = ncs[0];
#pragma unroll
    for (int q = 1; q < NC; ++q)
      if (ncs[q] > best) { best = ncs[q]; pick = q; }
    if (stride < NB - base) fetch(blk + stride);
    const int t = NC == 1 ? 0 : signs ? pick >> 1 : pick, sg = NC > 1 && signs ? pick & 1 : 0;
    uint32_t mb = 0;       // the maximum of the sixteen 15-bit magnitude patterns, two per word at a time
#pragma unroll
    for (int q = 0; q < 8; ++q) mb = __vmaxu2(mb, wb[q] & 0x7FFF7FFFu);
    mb = max(mb & 0xFFFFu, mb >> 16);
    const float amax = __uint_as_float(mb << 16);
    const PackTable& T = tab[t];
    const float sigma = T.tmax == 1.0f ? amax : __fdiv_rn(amax, T.tmax);
    const unsigned sb = __float_as_uint(sigma);
    float rcp;
    unsigned scode = 0;
    if (T.block_scope && sb - T.fast_lo < T.fast_span) {
      const unsigned rb = (sb + half + ((sb >> sh) & 1u)) & ~mask;
      scode = (rb >> sh) - T.code_off;
      rcp = reciprocal_scale(__uint_as_float(rb));
    } else {
      float s_hat;
      if (!T.block_scope) s_hat = amax > 0.0f ? T.pot : 0.0f;
      else { const QScale qs = scale_quantize(sigma, T.k, F); s_hat = qs.s_hat; scode = qs.code; }
      rcp = s_hat > 0.0f ? __frcp_rn(s_hat) : 0.0f;
    }
    if (KIND == SOP_KIND_FP_E4M3 && isinf(rcp)) saturate_zeros(wb);
    uint32_t code4[4];       // sixteen codes as bytes
    if (LUT) {
      const float r = (sg ? 1 - T.neg : T.neg) ? -rcp : rcp;       // a negated table runs on -u
      if (!T.slow) {
        const float inv_range = T.inv_range;
        const unsigned at = (unsigned)(t * (PCELLS + 1) * PCOPIES + (lane & (PCOPIES - 1))) - __float_as_uint(PMAGIC) * PCOPIES;      // modulo 2^32
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          uint32_t c4 = 0;
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int i = 4 * h + x;
            const float u = __fmul_rn((i & 1) ? bf16hi(wb[i >> 1]) : bf16lo(wb[i >> 1]), r);
            const uint2 e = cells[at + pack_cell(u, inv_range) * PCOPIES];
            // byte x of the word: the code below or above the threshold
            const unsigned below = x == 0 ? 0x3214u : x == 1 ? 0x3240u : x == 2 ? 0x3410u : 0x4210u;
            c4 = __byte_perm(c4, e.y, u > __uint_as_float(e.x) ? below + (1u << (4 * x)) : below);
          }
          code4[h] = c4;
        }
      } else {
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          code4[h] = 0;
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int i = 4 * h + x;
            code4[h] |= (uint32_t)count_below(tau[t], __fmul_rn((i & 1) ? bf16hi(wb[i >> 1]) : bf16lo(wb[i >> 1]), r)) << (8 * x);
          }
        }
      }
    } else if (KIND == SOP_KIND_FP_GRID) {
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        code4[h] = 0;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int i = 4 * h + x;
          const float u = __fmul_rn((i & 1) ? bf16hi(wb[i >> 1]) : bf16lo(wb[i >> 1]), rcp);
          code4[h] |= grid_code(grid_quantize(u, grid), grid, sign_pos) << (8 * x);      // at most 8 bits: the host refuses wider grids here
        }
      }
    } else {
      constexpr int FORMAT = KIND == SOP_KIND_FP_E4M3 ? SOP_KIND_FP_E4M3 : SOP_KIND_FP_E2M3;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        uint32_t lo2, hi2;
        fp_quantize2<FORMAT>(__fmul_rn(bf16lo(wb[2 * h]), rcp), __fmul_rn(bf16hi(wb[2 * h]), rcp), lo2);
        fp_quantize2<FORMAT>(__fmul_rn(bf16lo(wb[2 * h + 1]), rcp), __fmul_rn(bf16hi(wb[2 * h + 1]), rcp), hi2);
        code4[h] = lo2 | (hi2 << 16);
      }
    }
    if (on) { my_sel += (unsigned)t; my_neg += (unsigned)sg; }
    // codes: sixteen n-bit fields, little-endian, 2 n bytes
    if (n == 4) {
      uint32_t h16[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const uint32_t y = (code4[h] | (code4[h] >> 4)) & 0x00FF00FFu;
        h16[h] = (y | (y >> 8)) & 0xFFFFu;
      }
      if (on) *reinterpret_cast<uint2*>(a.codes + (size_t)blk * 8) = make_uint2(h16[0] | (h16[1] << 16), h16[2] | (h16[3] << 16));
    } else if (n == 8) {
      if (on) *reinterpret_cast<uint4*>(a.codes + (size_t)blk * 16) = make_uint4(code4[0], code4[1], code4[2], code4[3]);
    } else if (n == 6) {
      uint32_t v[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const uint32_t y = (code4[h] & 0x003F003Fu) | ((code4[h] >> 2) & 0x0FC00FC0u);
        v[h] = (y & 0xFFFu) | ((y >> 16) << 12);
      }
      if (on) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(a.codes + (size_t)blk * 12);
        dst[0] = v[0] | (v[1] << 24); dst[1] = (v[1] >> 8) | (v[2] << 16); dst[2] = (v[2] >> 16) | (v[3] << 8);
      }
    } else if (n == 5) {
      uint32_t v[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const uint32_t y = (code4[h] & 0x001F001Fu) | ((code4[h] >> 3) & 0x03E003E0u);
        v[h] = (y & 0x3FFu) | ((y >> 16) << 10);
      }
      const uint32_t w0 = v[0] | (v[1] << 20), w1 = (v[1] >> 12) | (v[2] << 8) | (v[3] << 28), w2 = v[3] >> 4;      // 80 bits
      // two blocks make five words: the even lane stores three of them, the odd lane two
      const uint32_t o0 = __shfl_down_sync(0xFFFFFFFFu, w0, 1);
      if (on) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(a.codes + (size_t)(blk & ~1u) * 10);
        if (!(blk & 1u)) {
          dst[0] = w0; dst[1] = w1;
          if (blk + 1u < NB) dst[2] = w2 | (o0 << 16);
          else reinterpret_cast<uint16_t*>(dst)[4] = (uint16_t)w2;
        } else {
          dst[3] = (w0 >> 16) | (w1 << 16); dst[4] = (w1 >> 16) | (w2 << 16);
        }
      }
    } else if (on) {
      unsigned long long lo = 0, hi = 0;   // 128-bit accumulator
      for (int i = 0; i < 16; ++i) {
        const int pos = i * n;
        const uint32_t word = i < 4 ? code4[0] : i < 8 ? code4[1] : i < 12 ? code4[2] : code4[3];
        const unsigned long long y = (unsigned long long)((word >> (8 * (i & 3))) & 0xFFu);
        if (pos < 64) { lo |= y << pos; if (pos + n > 64) hi |= y >> (64 - pos); }
        else hi |= y << (pos - 64);
      }
      unsigned short* dst = reinterpret_cast<unsigned short*>(a.codes + (size_t)blk * 2 * n);
      for (int i = 0; i < n; ++i) dst[i] = (unsigned short)((i < 4 ? lo >> (16 * i) : hi >> (16 * (i - 4))) & 0xFFFFu);
    }
    // scale word
    const unsigned sel = (unsigned)t, sgn = (unsigned)sg;
    unsigned word;
    if (a.word_sign_bits) word = (sgn << (b - 1)) | (scode << a.meta_bits) | (a.meta_bits >= 1 ? sel : 0u);
    else if (a.meta_bits >= 1) word = (sel << (b - 1)) | (scode << (a.meta_bits - 1));
    else word = scode;
    if (b == 16) {
      if (on) reinterpret_cast<unsigned short*>(a.words)[blk] = (unsigned short)word;
    } else if (b == 8) {
      if (on) reinterpret_cast<unsigned char*>(a.words)[blk] = (unsigned char)word;
    } else {
      // eight blocks make three words: lane x < 3 of a group of eight takes the blocks that reach into word x
      if (!on) word = 0;
      const int x = lane & 7, first = 32 * x / 12;
      unsigned out = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const unsigned w = __shfl_sync(0xFFFFFFFFu, word, (lane & ~7) + ((first + i) & 7));
        const int to = (first + i) * 12 - 32 * x;
        if (x < 3 && first + i < 8 && to < 32) out |= to >= 0 ? w << to : w >> -to;
      }
      const unsigned long long wi = (unsigned long long)((base + (unsigned)(lane & ~7)) / 8u) * 3u + (unsigned)x;
      if (x < 3 && wi * 32u < (unsigned long long)NB * 12u) a.words[wi] = out;
    }
  }
  // the stream's last 32 bits are whole
  if (blockIdx.x == 0 && tid < 4 && b != 12) {
    const unsigned long long end = (unsigned long long)NB * (unsigned)(b / 8), at = end + (unsigned)tid;
    if (at < ((end + 3ull) & ~3ull)) reinterpret_cast<unsigned char*>(a.words)[at] = 0;
  }
  if (a.counts) {
    my_sel = __reduce_add_sync(0xFFFFFFFFu, my_sel);
    my_neg = __reduce_add_sync(0xFFFFFFFFu, my_neg);
    if (lane == 0 && my_sel) atomicAdd(&s_cnt[0], my_sel);
    if (lane == 0 && my_neg) atomicAdd(&s_cnt[1], my_neg);
    __syncthreads();
    if (tid < 2 && s_cnt[tid]) atomicAdd(&a.counts[tid], (unsigned long long)s_cnt[tid]);
  }
}

int num_sms();

}  // namespace sop

extern "C" {

int sop_pack(const void* W_dev, long long M, long long K, long long ldw, const float* c_dev, int g,
             const sop_scale_fmt* fmt, const sop_atom* atoms, int n_atoms, const float* dd_lut_dev,
             unsigned dd_mask, int index_a, int index_b, int k_mode, const sop_search_result* search_dev,
             int use_sign, int container_bits, int word_sign_bits, unsigned char* codes_dev,
             unsigned char* words_dev, long long* counts_dev, const float* block_metric_dev, int flags, void* stream) {
  using namespace sop;
  const float* block_cos_dev = block_metric_dev;
  if (flags & ~SOP_PACK_SELECT_MSE) return SOP_ERR_RANGE;
  int rc = validate_layer(W_dev, M, K, ldw, c_dev, g);
  if (rc) return rc;
  if (!codes_dev || !words_dev) return SOP_ERR_NULL;
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
  }
  const bool pair = index_b != SOP_NO_ATOM;
  if (pair && meta < 1) return SOP_ERR_FORMAT;     // the selector needs a metabit
  // a parametric grid is packed as sign | E | M in at most 8 bits; wider grids and grids without such a code are swept only
  if (!from_result && atoms[index_a].kind == SOP_KIND_FP_GRID &&
      (atoms[index_a].grid_exp_bits < 1 || atoms[index_a].n_bits > 8)) return SOP_ERR_ALPHABET;
  if (k_mode == SOP_K_FROM_RESULT) { if (!search_dev) return SOP_ERR_NULL; }
  else if (k_mode < -64 || k_mode > 64) return SOP_ERR_RANGE;
  bool need_wmax = false;
  for (int i = 0; i < n_atoms; ++i) need_wmax |= atoms[i].scope == 0;
  if (need_wmax && !search_dev) return SOP_ERR_NULL;  // the layer power-of-two scale comes from a previous search
  if (((uintptr_t)codes_dev & 15u) || ((uintptr_t)words_dev & 3u)) return SOP_ERR_SHAPE;
  // every atom that can be picked must share n_bits with the first LUT atom when the pair comes from the device
  int n_bits = from_result ? 0 : atoms[index_a].n_bits;
  if (from_result) {
    for (int i = 0; i < n_atoms; ++i)
      if (atoms[i].kind == SOP_KIND_LUT) { if (!n_bits) n_bits = atoms[i].n_bits; else if (atoms[i].n_bits != n_bits) return SOP_ERR_ALPHABET; }
    if (!n_bits) return SOP_ERR_ALPHABET;
  }

  PackArgs a;
  a.W = (const uint16_t*)W_dev; a.c = c_dev; a.M = M; a.K = K; a.ldw = ldw; a.nbk = K / SOP_G; a.NB = M * a.nbk;
  a.index_a = index_a; a.index_b = index_b; a.k_mode = k_mode; a.use_sign = use_sign;
  a.container_bits = container_bits; a.word_sign_bits = word_sign_bits; a.meta_bits = meta;
  a.codes = codes_dev; a.words = (unsigned*)words_dev; a.counts = (unsigned long long*)counts_dev;
  a.block_cos = block_cos_dev;
  a.select_err = (flags & SOP_PACK_SELECT_MSE) ? 1 : 0;
  a.cos_neg_a = a.cos_neg_b = -1;
  if (block_cos_dev && use_sign && !from_result) {
    // row of the negated variant of an explicitly given atom: same table and scale reference, opposite sign
    auto find_neg = [&](int i) {
      for (int j = 0; j < n_atoms; ++j)
        if (j != i && atoms[j].kind == atoms[i].kind && atoms[j].negated != atoms[i].negated && atoms[j].tmax == atoms[i].tmax &&
            atoms[j].n_entries == atoms[i].n_entries && ((dd_mask >> j) & 1u) == ((dd_mask >> i) & 1u) &&
            (((dd_mask >> i) & 1u) || memcmp(atoms[j].lut, atoms[i].lut, sizeof(float) * atoms[i].n_entries) == 0))
          return j;
      return -1;
    };
    a.cos_neg_a = find_neg(index_a);
    if (index_b != SOP_NO_ATOM) a.cos_neg_b = find_neg(index_b);
  }
  cudaStream_t st = (cudaStream_t)stream;
  const size_t word_bytes = (size_t)((a.NB * container_bits + 7) / 8);
  // 12-bit words are merged into the stream with 32-bit atomicOr (the caller's buffer holds whole 32-bit
  // words and starts from zero); 8- and 16-bit words are stored directly, only the padding is cleared
  const size_t padded = (word_bytes + 3) & ~(size_t)3;
  const bool negs_known = !use_sign || from_result || (a.cos_neg_a >= 0 && (!pair || a.cos_neg_b >= 0));
  const int kind = from_result ? SOP_KIND_LUT : atoms[index_a].kind;
  const bool winner = block_cos_dev && negs_known;       // (pack_winner_kernel writes whole words)
  if (winner) {}
  else if (container_bits == 12) SOP_CUDA_TRY(cudaMemsetAsync(words_dev, 0, padded, st));
  else SOP_CUDA_TRY(cudaMemsetAsync(words_dev + padded - 4, 0, 4, st));
  if (counts_dev) SOP_CUDA_TRY(clear(counts_dev, 2 * sizeof(long long), st));
  long long grid = (a.NB + PTB - 1) / PTB;
  const int sms = num_sms();
  const long long resident = (long long)sms * 4;
  if (grid > resident) grid = resident;      // one wave of resident CTAs: the table set-up runs once per CTA
  if ((rc = profile_mark(SOP_PROFILE_PACK, 0, st))) return rc;
#define SOP_PACK(KD, NN, C) SOP_CUDA_TRY(launch(pack_winner_kernel<KD, NN, C>, grid, PTB, 0, st, a, A, F, search_dev))
#define SOP_PACK_LUT(NN) do { if (n_cand == 4) SOP_PACK(SOP_KIND_LUT, NN, 4); else if (n_cand == 2) SOP_PACK(SOP_KIND_LUT, NN, 2); else SOP_PACK(SOP_KIND_LUT, NN, 1); } while (0)
  const int n_cand = (pair ? 2 : 1) * (use_sign ? 2 : 1);
  if (winner && kind == SOP_KIND_FP_E2M3) SOP_PACK(SOP_KIND_FP_E2M3, 6, 1);
  else if (winner && kind == SOP_KIND_FP_E4M3) SOP_PACK(SOP_KIND_FP_E4M3, 8, 1);
  else if (winner && kind == SOP_KIND_FP_GRID) SOP_PACK(SOP_KIND_FP_GRID, 0, 1);
  else if (winner && n_bits == 4) SOP_PACK_LUT(4);
  else if (winner && n_bits == 5) SOP_PACK_LUT(5);
  else if (winner) SOP_PACK_LUT(0);
#undef SOP_PACK_LUT
#undef SOP_PACK
  else SOP_CUDA_TRY(launch(pack_kernel, grid, PTB, 0, st, a, A, F, search_dev));
  if ((rc = profile_mark(SOP_PROFILE_PACK, 1, st))) return rc;
  SOP_CUDA_TRY(cudaGetLastError());
  return SOP_OK;
}

}  // extern "C"
