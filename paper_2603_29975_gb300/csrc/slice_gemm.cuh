// Slice-pair GEMM on the sm_103a tensor cores with the fused reconstruction epilogue
// (paper Sec. 2.2: low-precision products of slice pairs, accumulated in higher precision).
//
// Operands are the fp16 digit planes written by split.cu: A [batch][h][S][rowsA][8] and B
// [batch][h][S][rowsB][8], h over the 16-byte K halves.  One CTA computes a 128 x BN tile of the stacked real
// product (m x 2n) for every slice pair at once:
//
//   * warp 0 (one lane) streams K-blocks of 16 with TMA: one box of two halves of S slices of A
//     (128 rows) and one of B (BN rows) per pipeline stage, in runs of 2 KB and BN x 16 bytes, which
//     land as the unswizzled core-matrix layout of the MMA descriptors;
//   * warp 1 (one elected lane) issues tcgen05.mma kind::f16 for every pair (s, t) of the pair set,
//     accumulating pair products of the same weight class g = s + t into one FP32 TMEM
//     accumulator per group (G groups x BN columns of the 512); where the groups are accumulated
//     already, the partners of each A slice share one MMA over the stacked B slices, and around a
//     chunk's boundary the groups go in two parts, so that one part is drained while the tensor
//     cores work on the other;
//   * warp 2 finds the CTA's tiles ahead of the others and leaves them in a ring;
//   * warps 4..19 drain the accumulators.  Every product of two digits is an integer of
//     magnitude <= 2^14 and each accumulator receives at most 1024 of them per "exactness
//     chunk" of K, so every FP32 value is an exact integer <= 2^24.  The epilogue brings it into
//     the low bits of a 32-bit word by one FP32 addition and adds groups in pairs, each with its
//     weight of 8 (g_max - g) bits, into 64-bit integers: one per output element when the exact
//     sum fits, else one per run of four groups (128-bit sums in the run-time schedules of many
//     groups or a very long K).  After the last chunk their exact sum times 2^(e_i + f_j + c) is
//     rounded once to binary64 (the int64 -> binary64 conversion of a 64-bit sum, integer
//     operations on three 32-bit words or 128 bits otherwise), then stored (C = Z), or subtracted
//     from C (LU update), or combined with alpha/beta.
// No floating-point instruction touches the products' sums before that one rounding; the
// only binary64 arithmetic after it is the subtraction / alpha-beta combination per element.
#pragma once

#include <type_traits>

#include "ozk_params.cuh"

namespace ozk {

constexpr int GEMM_BM = 128;
constexpr int GEMM_EPI_WARPS = 16;
// warpgroup 0 (warps 0..3): TMA producer (warp 0), MMA issuer (warp 1), tiles (warp 2), an idle warp; it
// hands registers to the four epilogue warpgroups (setmaxnreg), whose exact sums of 16 outputs
// need more than the 96 registers a thread of a 20-warp CTA starts with
constexpr int GEMM_CTRL_WARPS = 4;
constexpr int GEMM_THREADS = (GEMM_CTRL_WARPS + GEMM_EPI_WARPS) * 32;
constexpr int GEMM_CTRL_REGS = 64, GEMM_EPI_REGS = 104;
constexpr int GEMM_SMEM_MAX = 227 * 1024;        // shared memory of a CTA (all of it dynamic)

// Exact sums at the ends of the binary64 exponent range, one rounding in 128 bits.
static __device__ __noinline__ double round_far(long long H, long long L, int s8, int E) {
  return round_scaled_dev((static_cast<__int128>(H) << s8) + static_cast<__int128>(L), E);
}

// RN-even of (H 2^S8 + L) 2^E for int64 H, L and E such that every nonzero result is a normal number
// (S8 <= 32; H + L 2^-S8 stays below 2^63 in magnitude, as the plan of the product checks by bounding H
// and L by 0.99 2^63; S8 = 0: |H| < 2^63, no L).
//   S8 = 0: the int64 -> binary64 conversion is that rounding, and the scaling an addition to the
// exponent field.
//   S8 > 0: 32-bit integer operations: the sum as a two's-complement integer of three words (h1, h0,
// lw) = T 2^(32 - S8), its magnitude, the leading one brought to bit 31 of the first word (after
// dropping a zero first word), the 53-bit significand with its rounding bit and the sticky rest.
// About 35 operations of a pipe that runs 64 a clock per SM (4540 cycles for a tile's 8192 sums by
// themselves).  The conversion of T jammed to 62 bits leaves 22 of them but runs at 2 a clock per SM
// on the FP64 pipe (4410 cycles), which the update C - RN(Z) needs as well: the update of
// 6144 x 6144 outputs with K = 192 took 20.1 us per 128 x 64 tile that way and 18.1 this way (S = 7).
// ehi: round_ehi.
template <int S8>
__device__ __forceinline__ double round_hl(unsigned long long H, unsigned long long L, uint32_t ehi) {
  if constexpr (S8 == 0) {
    const double d = __ll2double_rn(static_cast<long long>(H));
    const uint32_t dh = static_cast<uint32_t>(__double2hiint(d));
    return dh ? __hiloint2double(static_cast<int>(dh + ehi), __double2loint(d)) : 0.0;
  } else {
    const unsigned long long Hp = H + static_cast<unsigned long long>(static_cast<long long>(L) >> S8);
    uint32_t h0 = static_cast<uint32_t>(Hp), h1 = static_cast<uint32_t>(Hp >> 32);
    uint32_t lw = static_cast<uint32_t>(L) << (32 - S8);
    const uint32_t s = static_cast<uint32_t>(static_cast<int>(h1) >> 31);
    // magnitude: (~T) + 1 for negative T
    asm("{\n\tadd.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, 0;\n\taddc.u32 %2, %5, 0;\n\t}"
        : "=r"(lw), "=r"(h0), "=r"(h1) : "r"(lw ^ s), "r"(h0 ^ s), "r"(h1 ^ s), "r"(s & 1u));
    uint32_t eadj = ehi;
    if (h1 == 0u) {
      h1 = h0;
      h0 = lw;
      lw = 0u;
      eadj -= 32u << 20;
    }
    if (h1 == 0u) {                                          // |T| 2^(32 - S8) < 2^32 (T = 0, above all)
      h1 = h0;
      h0 = 0u;
      eadj -= 32u << 20;
    }
    const int lz = __clz(static_cast<int>(h1));
    const uint32_t n1 = __funnelshift_l(h0, h1, lz), n0 = __funnelshift_l(lw, h0, lz), rest = lw << (lz & 31);
    // significand n1:n0 (leading one at bit 63): 53 bits, then the rounding bit and 10 more in n0
    const uint32_t m1 = n1 >> 11, m0 = __funnelshift_r(n0, n1, 11);
    uint32_t t = n0 << 21;
    if (rest != 0u) t |= 1u;
    // + 1 when t + (m0 & 1) > 2^31: the carry out of t + (2^31 - 1) + (m0 & 1)
    uint32_t lo, hi;
    asm("{\n\t.reg .u32 c;\n\tadd.cc.u32 c, %2, %3;\n\taddc.cc.u32 %0, %4, 0;\n\taddc.u32 %1, %5, 0;\n\t}"
        : "=r"(lo), "=r"(hi) : "r"(t), "r"(0x7FFFFFFFu + (m0 & 1u)), "r"(m0), "r"(m1 + eadj - (static_cast<uint32_t>(lz) << 20)));
    // T = 0: +0
    return h1 == 0u ? 0.0 : __hiloint2double(static_cast<int>(hi ^ (s & 0x80000000u)), static_cast<int>(lo));
  }
}
// E for round_hl, in the exponent field, and the sign bit when -RN is wanted.  S8 > 0: a leading one
// at bit 31 - lz of h1 has the weight 2^(E + 63 + S8 - lz), and the significand's own leading one adds
// one to the exponent field.
template <int S8>
__device__ __forceinline__ uint32_t round_ehi(int E, bool neg) {
  return (static_cast<uint32_t>(S8 > 0 ? E + 63 + S8 + 1022 : E) << 20) + (neg ? 0x80000000u : 0u);
}
// The row and column exponents whose sums are within round_hl's range for sums T below 2^96.
__device__ __forceinline__ bool exponent_near(int e) { return static_cast<unsigned>(e + 500) <= 950u; }

// Exact FP32 integer accumulator values (|v| <= 2^24) folded into 64-bit sums.  When the values are
// below 2^22 in magnitude, one FP32 add puts the integer into the low mantissa bits (x + 1.5 2^23
// lies in [2^23, 2^24), where the spacing is 1), and two groups combine in 32 bits, 256 v + u with
// |256 v + u| < 2^31, before the one 64-bit multiply-add.  Larger values (they need sums of hundreds
// of near-maximal digit products) take the conversion unit, which delivers 16 a clock per SM.
// Whether the values are small is known beforehand for short K (the magic mask).  Otherwise they are
// folded as if they were, with a running maximum of their magnitudes (one three-input maximum per
// two values), one vote per part of the accumulators, and a second reading that adds the difference
// if it says no: with the check, vote and branch at every pair of groups, a 128 x 64 tile of K = 64
// took 8.8 us instead of 6.5 (S = 7, C = Z).
// The 32-bit parts enter as unsigned numbers with the constant of their magic additions still in
// (0x4B400000 + v, and 0x8B400000 + 256 v + u modulo 2^32, neither of which wraps for |v|, |u| <
// 2^22); the sums start at minus those constants (FoldPlan::bias).
constexpr uint32_t MAGIC_ONE = 0x4B400000u, MAGIC_PAIR = 0x8B400000u;     // 1.5 2^23; 257 times it mod 2^32
__device__ __forceinline__ uint32_t magic_bits(uint32_t v) { return __float_as_uint(__uint_as_float(v) + 12582912.0f); }
__device__ __forceinline__ int acc_to_int(uint32_t bits, bool magic) {
  return magic ? static_cast<int>(magic_bits(bits) - MAGIC_ONE) : __float2int_rn(__uint_as_float(bits));
}
__device__ __forceinline__ float max_abs3(float m, uint32_t a, uint32_t b) {
  return fmaxf(m, fmaxf(fabsf(__uint_as_float(a)), fabsf(__uint_as_float(b))));
}
template <int N>
__device__ __forceinline__ float max_abs(float m, const uint32_t (&v)[N]) {
#pragma unroll
  for (int j = 0; j < N; j += 2) m = max_abs3(m, v[j], v[j + 1]);
  return m;
}
// x += r 2^W
template <int W>
__device__ __forceinline__ void add_shifted(unsigned long long& x, uint32_t r) {
  if constexpr (W == 0) x += r;
  else asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(x) : "r"(r), "n"(1 << W));
}
// X[j] += (256 v_j + u_j + MAGIC_PAIR) 2^W, |v_j|, |u_j| < 2^22
template <int W, int N>
__device__ __forceinline__ void fold_pair(unsigned long long* X, const uint32_t (&v)[N], const uint32_t (&u)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) add_shifted<W>(X[j], (magic_bits(v[j]) << 8) + magic_bits(u[j]));
}
// X[j] += (v_j + MAGIC_ONE) 2^W, |v_j| < 2^22
template <int W, int N>
__device__ __forceinline__ void fold_one(unsigned long long* X, const uint32_t (&v)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) add_shifted<W>(X[j], magic_bits(v[j]));
}
// what the true values would have added, less what fold_pair and fold_one did add
template <int W, int N>
__device__ __forceinline__ void refold_pair(unsigned long long* X, const uint32_t (&v)[N], const uint32_t (&u)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const long long t = static_cast<long long>(__float2int_rn(__uint_as_float(v[j]))) * 256 +
                        __float2int_rn(__uint_as_float(u[j])) + static_cast<long long>(MAGIC_PAIR);
    const uint32_t had = (magic_bits(v[j]) << 8) + magic_bits(u[j]);
    X[j] += static_cast<unsigned long long>(t - static_cast<long long>(had)) << W;
  }
}
template <int W, int N>
__device__ __forceinline__ void refold_one(unsigned long long* X, const uint32_t (&v)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const long long t = static_cast<long long>(__float2int_rn(__uint_as_float(v[j]))) + static_cast<long long>(MAGIC_ONE);
    X[j] += static_cast<unsigned long long>(t - static_cast<long long>(magic_bits(v[j]))) << W;
  }
}

// One MMA from descriptor words: with a compile-time schedule, two 32-bit additions and the
// tcgen05.mma itself.
__device__ __forceinline__ void mma_f16_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc,
                                           uint32_t accumulate) {
  const uint64_t ad = (static_cast<uint64_t>(hi) << 32) | a_lo;
  const uint64_t bd = (static_cast<uint64_t>(hi) << 32) | b_lo;
  mma_f16(d_tmem, ad, bd, idesc, accumulate);
}

// The groups [0, split_group(G)) are the first part of the accumulators, the others the second: the
// two are finished, drained and overwritten half a chunk apart (see the MMA issuer).
__host__ __device__ constexpr int split_group(int G) { return G >= 6 ? 4 : (G + 1) / 2; }

// MMAs of one K-block on the groups [G0, G1) of the triangular pair set.  The B slices sit back to
// back in shared memory (slice t at row (t - 1) BN) and group g = s + t - 2 at TMEM column g BN, so
// A_s x [B_t0 .. B_t1]^T is a single MMA of N = (t1 - t0 + 1) BN columns (in two even pieces above
// N = 256; an MMA of fewer than about 96 columns costs as much as one of 96).  FIRST: first K-block
// of an exactness chunk -- slice s = 1 pairs with every t, so its MMAs overwrite every group
// (accumulate = 0); the later slices accumulate onto it.
template <int S, int BN, int G0, int G1, bool FIRST>
__device__ __forceinline__ void issue_groups(uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi) {
#pragma unroll
  for (int s = 1; s <= S; ++s) {
    const int t0 = G0 + 2 - s > 1 ? G0 + 2 - s : 1, t1 = S + 1 - s < G1 + 1 - s ? S + 1 - s : G1 + 1 - s;
    const int ncols = (t1 - t0 + 1) * BN;
    if (ncols <= 0) continue;
    const int np = ncols > 256 ? (ncols / 2 + 15) / 16 * 16 : ncols;
#pragma unroll
    for (int c0 = 0; c0 < ncols; c0 += np) {
      const int n = ncols - c0 < np ? ncols - c0 : np;
      mma_f16_lo(tmem + (s + t0 - 2) * BN + c0, a_lo + (s - 1) * GEMM_BM, b_lo + (t0 - 1) * BN + c0, hi,
                 idesc_f16_f32(GEMM_BM, n), (FIRST && s == 1) ? 0u : 1u);
    }
  }
}

// One K-block of MMAs for every pair of the full pair set, pair by pair in the order of their groups
// in a chunk's first K-block (the first pair of each group overwrites its accumulator), stacked as
// above in the others.
template <int S, int BN>
__device__ __forceinline__ void issue_kblock_full(bool first, uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi) {
  if (first) {
#pragma unroll
    for (int g = 2; g <= 2 * S; ++g) {
      bool lead = true;
#pragma unroll
      for (int s = 1; s <= S; ++s) {
        const int t = g - s;
        if (t < 1 || t > S) continue;
        mma_f16_lo(tmem + (g - 2) * BN, a_lo + (s - 1) * GEMM_BM, b_lo + (t - 1) * BN, hi, idesc_f16_f32(GEMM_BM, BN),
                   lead ? 0u : 1u);
        lead = false;
      }
    }
    return;
  }
#pragma unroll
  for (int s = 1; s <= S; ++s)
#pragma unroll
    for (int c0 = 0; c0 < S * BN; c0 += 256) {
      const int n = S * BN - c0 < 256 ? S * BN - c0 : 256;
      mma_f16_lo(tmem + (s - 1) * BN + c0, a_lo + (s - 1) * GEMM_BM, b_lo + c0, hi, idesc_f16_f32(GEMM_BM, n), 1u);
    }
}

// Runtime schedule (slice counts and pair sets without a compile-time one, Ozaki-II's products).
template <int BN>
__device__ __forceinline__ void issue_runtime(const GemmParams& p, bool firstkb, uint32_t tmem, uint32_t a_lo,
                                              uint32_t b_lo, uint32_t hi) {
  for (int pi = 0; pi < p.npairs; ++pi) {
    const uint32_t s = p.ps[pi], t = p.pt[pi], g = p.pg[pi];
    mma_f16_lo(tmem + g * BN, a_lo + s * GEMM_BM, b_lo + t * BN, hi, idesc_f16_f32(GEMM_BM, BN),
               firstkb && p.pfirst[pi] ? 0u : 1u);
  }
}

enum GroupPart : int { PART_FIRST = 0, PART_SECOND = 1, PART_ALL = 2 };

template <int S, int BN, int PART>
__device__ __forceinline__ void issue_tri(bool first, uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi) {
  constexpr int GA = split_group(S);
  constexpr int G0 = PART == PART_SECOND ? GA : 0, G1 = PART == PART_FIRST ? GA : S;
  if (first) issue_groups<S, BN, G0, G1, true>(tmem, a_lo, b_lo, hi);
  else issue_groups<S, BN, G0, G1, false>(tmem, a_lo, b_lo, hi);
}

// Whether the launch's K-blocks may be issued in parts (compile-time triangular schedules).
template <int BN>
__device__ __forceinline__ bool in_parts(const GemmParams& p, int S) {
  if (p.diag_pairs || p.fullset) return false;
  if constexpr (BN == 64) return true;
  return S == 9 || S == 10;
}

template <int BN, int PART>
__device__ __forceinline__ void issue_dispatch(const GemmParams& p, int S, bool first, uint32_t tmem,
                                               uint32_t a_lo, uint32_t b_lo, uint32_t hi) {
#define OZK_TRI(SS) case SS: issue_tri<SS, BN, PART>(first, tmem, a_lo, b_lo, hi); return
#define OZK_FULL(SS) case SS: issue_kblock_full<SS, BN>(first, tmem, a_lo, b_lo, hi); return
  if (in_parts<BN>(p, S)) {
    if constexpr (BN == 64) {
      switch (S) { OZK_TRI(1); OZK_TRI(2); OZK_TRI(3); OZK_TRI(4); OZK_TRI(5); OZK_TRI(6); OZK_TRI(7); OZK_TRI(8); default: break; }
    } else {
      // 32-column tiles: S = 9 (the selector's largest regular choice) and S = 10 (its fallback)
      switch (S) { OZK_TRI(9); OZK_TRI(10); default: break; }
    }
  }
  if constexpr (BN == 64) {
    if (p.fullset && !p.diag_pairs)
      switch (S) { OZK_FULL(1); OZK_FULL(2); OZK_FULL(3); OZK_FULL(4); default: break; }
  }
#undef OZK_TRI
#undef OZK_FULL
  issue_runtime<BN>(p, first, tmem, a_lo, b_lo, hi);
}

// Tiles of one problem of a batched GEMM (m rows, n2 stacked columns) with a skip box
// [0, km) x [0, kn) (rows, complex columns) whose outputs are neither computed nor written: the
// part beside the box, rows [0, km) x stacked columns [2 kn, n2), in ku x xu tiles of a grid
// that starts at row 0 and stacked column 2 kn (the last tile row clipped at row km, mu), then
// the part below it, rows [km, m) x all columns, in nl x ntx tiles of a grid that starts at row
// km (m0l).  Each part's grid starts at the box edge, so a strip of one tile's width beside or
// below the box takes one tile row or column, not two.  Without a box (km or kn zero) the whole
// grid is the second part.
struct BoxTiles { int ku, xu, mu, n0u, nl, ntx, m0l; };
__host__ __device__ __forceinline__ BoxTiles box_tiles(int m, int n2, int km, int kn, int BN) {
  BoxTiles b;
  b.ntx = (n2 + BN - 1) / BN;
  if (km > 0 && kn > 0) {
    b.mu = km < m ? km : m;
    b.ku = (b.mu + GEMM_BM - 1) / GEMM_BM;
    b.n0u = 2 * kn;
    b.xu = n2 > b.n0u ? (n2 - b.n0u + BN - 1) / BN : 0;
    b.m0l = km;
    b.nl = m > km ? (m - km + GEMM_BM - 1) / GEMM_BM : 0;
  } else {
    b.mu = 0; b.ku = 0; b.n0u = 0; b.xu = 0; b.m0l = 0;
    b.nl = (m + GEMM_BM - 1) / GEMM_BM;
  }
  return b;
}

// One tile (work unit) as the kernel's roles need it: written by the tile warp into a ring of slots
// in shared memory while earlier tiles run, so that neither the search for the tile's problem nor
// the loads of its exponents and row pointers stand between two tiles of the epilogue (they took
// 2900 to 3800 cycles of each 128 x 64 tile when every role found its own).
struct RowInfo { double2* C; int ld; int grow; };       // row r at C[j ld]; C null: not written
template <int BN>
struct TileInfo {
  int end;                         // no more tiles: the other fields are unset
  int za, ra, n0;                  // operand plane; first plane row and stacked column of the tile
  int kb0, kb1;                    // K-blocks of the unit
  int sp;                          // split-K: the unit's K slice (its partial sums go to p.part)
  int z, row0;                     // problem; first row of the tile in it
  int rows, n2;                    // rows of the problem in the tile; stacked columns of the problem
  int skip_rows, skip_cols;        // rows [0, skip_rows) of the tile skip complex columns below skip_cols
  int pad[3];
  int e[GEMM_BM];                  // row exponents plus base_exp
  int f[BN / 2];                   // column exponents
  RowInfo row[GEMM_BM];
};
constexpr int GEMM_TILE_SLOTS = 4;

struct EpiCtx {
  int row, n2, n0, c0, skip_n, er;
  int sp;
  int grow;              // row of the output matrix (the diagonal test of EPI_IMINUS)
  int jlim;              // complex columns of the output row's matrix
  uint32_t tbase;
  double2* C;            // output row: element j at C[j ld]
  const int* f;          // column exponents of the tile (shared memory)
  long long ld;
  bool rowok;
};

// output pointer, leading dimension and matrix row of row `row` of problem z (row `pr` of operand
// plane za)
__device__ __forceinline__ RowInfo out_row(const GemmParams& p, bool single, int z, int row, int za, int pr) {
  RowInfo o;
  if (p.crow) {
    const int as = pr / p.crow_b, rl = pr - as * p.crow_b;
    const int a = p.crow_perm ? p.crow_perm[as] : as;
    const long long crow = static_cast<long long>(za) * p.crow_b + rl;
    o.ld = p.crow_n ? p.crow_n[a] : p.ldc1;
    o.C = (p.crow_n && crow >= o.ld) ? nullptr : p.crow[a] + crow;
    o.grow = static_cast<int>(crow);
  } else {
    o.C = (single ? p.C1 : p.C[z]) + row;
    o.ld = single ? p.ldc1 : p.ldc[z];
    o.grow = row;
  }
  return o;
}

// Waits of the epilogue for the accumulators of one tile: its exactness chunks complete one after
// the other, each in two parts (acc_full; chunk counter cc, running over the CTA's tiles).
struct ChunkWait {
  uint64_t* acc_full;
  int nchunks;
  uint32_t* cc;
  int* status;
  volatile int* abort_flag;
  __device__ __forceinline__ bool part(int i) {
    if (!mbar_wait(&acc_full[i], *cc & 1, status, abort_flag)) return false;
    tc_fence_after();
    return true;
  }
};

// Release every group accumulator of every chunk of a tile without reading it (a warp with no
// output in the tile).
template <int G>
__device__ __forceinline__ bool release_unread(uint64_t* acc_empty, ChunkWait& cw, int lane) {
  for (int c = 0; c < cw.nchunks; ++c, ++*cw.cc) {
#pragma unroll
    for (int gi = 0; gi < G; ++gi) {
      if (gi == 0 && !cw.part(0)) return false;
      if (gi == split_group(G) && !cw.part(1)) return false;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[gi]);
    }
  }
  return true;
}

// Reads of one tile's chunk: step i takes 8 of the thread's 16 columns (half i & 1) of the groups
// gi(i), gi(i) + 1 (ng(i) of them): groups in pairs that cross neither the accumulators' parts nor
// the halves H ([0, NH)) and L ([NH, G)) of the sums.
template <int G, int NH>
struct FoldPlan {
  __host__ __device__ static constexpr int bound(int g) {        // end of the run of groups that g is in
    const int a = split_group(G);
    int e = G;
    if (g < a && a < e) e = a;
    if (g < NH && NH < e) e = NH;
    return e;
  }
  __host__ __device__ static constexpr int gi(int i) {
    int g = 0;
    for (int k = 0; k < i / 2 && g < G; ++k) g += bound(g) - g >= 2 ? 2 : 1;
    return g;
  }
  __host__ __device__ static constexpr int ng(int i) { return bound(gi(i)) - gi(i) >= 2 ? 2 : 1; }
  __host__ __device__ static constexpr bool more(int i) { return gi(i) < G; }
  __host__ __device__ static constexpr int first_step(int g) {
    int i = 0;
    while (gi(i) < g) i += 2;
    return i;
  }
  // weight (bits) of the step's last group in its half of the sums
  __host__ __device__ static constexpr int shift(int i) { return 8 * ((gi(i) < NH ? NH : G) - gi(i) - ng(i)); }
  // the constants that a chunk's steps add to the sums of groups [lo, hi)
  __host__ __device__ static constexpr unsigned long long bias(int lo, int hi) {
    unsigned long long b = 0;
    for (int i = 0; more(i); i += 2)
      if (gi(i) >= lo && gi(i) < hi)
        b += static_cast<unsigned long long>(ng(i) == 2 ? MAGIC_PAIR : MAGIC_ONE) << shift(i);
    return b;
  }
};
// Steps I .. of the groups below GE, folded as small values (REDO: corrected); `early`: every group
// is released as soon as its columns are read.
template <int G, int NH, int I, int GE, bool REDO>
__device__ __forceinline__ void fold_steps(const EpiCtx& x, uint64_t* acc_empty, int lane, bool early, float& big,
                                           unsigned long long (&H)[16], unsigned long long (&L)[16]) {
  using P = FoldPlan<G, NH>;
  if constexpr (P::gi(I) < GE) {
    constexpr int BN = 64, gi = P::gi(I), ng = P::ng(I), half = I & 1;
    uint32_t v[8], u[8];
    tmem_ld8(x.tbase + gi * BN + 8 * half, v);
    if constexpr (ng == 2) tmem_ld8(x.tbase + (gi + 1) * BN + 8 * half, u);
    tmem_wait_ld();
    unsigned long long* X = (gi < NH ? H : L) + 8 * half;
    if constexpr (REDO) {
      if constexpr (ng == 2) refold_pair<P::shift(I)>(X, v, u);
      else refold_one<P::shift(I)>(X, v);
    } else {
      if (half == 1 && early) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&acc_empty[gi]);
          if constexpr (ng == 2) mbar_arrive(&acc_empty[gi + 1]);
        }
      }
      big = max_abs(big, v);
      if constexpr (ng == 2) big = max_abs(big, u);
      if constexpr (ng == 2) fold_pair<P::shift(I)>(X, v, u);
      else fold_one<P::shift(I)>(X, v);
    }
    fold_steps<G, NH, I + 1, GE, REDO>(x, acc_empty, lane, early, big, H, L);
  }
}
// Groups [G0, GE) of one chunk (a part of the accumulators).  A part without groups (the second one
// of G = 1) is not waited for: nothing it releases would hold the issuer back, which could complete
// that barrier's phase of the next chunk too before a slow warp had seen this one's.
template <int G, int NH, int G0, int GE>
__device__ __forceinline__ bool fold_part(const EpiCtx& x, uint64_t* acc_empty, int lane, uint32_t magic_mask,
                                          ChunkWait& cw, unsigned long long (&H)[16], unsigned long long (&L)[16]) {
  if constexpr (G0 < GE) {
    if (!cw.part(G0 == 0 ? 0 : 1)) return false;
    constexpr int I0 = FoldPlan<G, NH>::first_step(G0);
    constexpr uint32_t need = ((1u << (GE - G0)) - 1u) << G0;
    const bool known = (magic_mask & need) == need;
    float big = 0.0f;
    fold_steps<G, NH, I0, GE, false>(x, acc_empty, lane, known, big, H, L);
    if (!known) {
      if (__any_sync(0xffffffffu, !(big < 4194304.0f)))
        fold_steps<G, NH, I0, GE, true>(x, acc_empty, lane, false, big, H, L);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
#pragma unroll
        for (int g = G0; g < GE; ++g) mbar_arrive(&acc_empty[g]);
      }
    }
  }
  return true;
}

// One complex output: (zr, zi), z rounded (EPI_IMINUS: -Z rounded), becomes the value to store; c the
// old value of C (UPDATE).
template <bool UPDATE>
__device__ __forceinline__ void combine(const GemmParams& p, double& zr, double& zi, double2 c, bool diag) {
  if (UPDATE && p.mode == EPI_LU) {
    zr = c.x - zr;
    zi = c.y - zi;
  } else if (!UPDATE && p.mode == EPI_IMINUS) {
    if (diag) zr = 1.0 + zr;                              // off the diagonal 0 - RN(Z) = RN(-Z)
  } else if (UPDATE || !p.unit_alpha) {
    const double xr = p.ar * zr - p.ai * zi, xi = p.ar * zi + p.ai * zr;
    zr = UPDATE ? xr + (p.br * c.x - p.bi * c.y) : xr;
    zi = UPDATE ? xi + (p.br * c.y + p.bi * c.x) : xi;
  }
}

// Epilogue of one 128 x 64 tile for G <= 8 groups (compile-time) over the tile's exactness
// chunks: the exact sum of the group values v_g (|v| <= 2^24 per chunk) is H 2^(8 NL) + L with
// H = the first NH = min(G, 4) groups and L = the rest (F64: the whole sum fits 64 bits, NL = 0 and
// H takes every group, G <= 5), each accumulated over the chunks in 64 bits.  A thread owns one row and
// 16 stacked columns (8 complex).  The groups are read two at a time.  Where their values are known to be
// small (magic mask), a pair is released as soon as it is read; otherwise a part's groups are released
// together, after the vote on their values and the second reading it may ask for.  Either way the MMAs of
// the next chunk or tile start on them while the rest is folded, rounded and written.  The outputs are
// rounded and combined in two halves of 4 complex columns.
// Returns false if a wait gave up.
// UPDATE: the mode combines with C (a separate instance: the values' registers would spill the others).
template <int G, bool F64, bool KS, bool UPDATE>
__device__ __forceinline__ bool epilogue_fast(const GemmParams& p, const EpiCtx& x, uint64_t* acc_empty,
                                              uint32_t magic_mask, int lane, ChunkWait& cw) {
  constexpr int NH = F64 ? G : (G < 4 ? G : 4);
  constexpr int NL = G - NH;
  constexpr int S8 = 8 * NL;
  const int jc0 = (x.n0 + x.c0) / 2;                  // this thread's 8 complex columns
  const int jend = min(min(jc0 + 8, (x.n2 + 1) / 2), x.jlim);
  const bool active = x.rowok && max(jc0, x.skip_n) < jend;
  if (!__any_sync(0xffffffffu, active)) return release_unread<G>(acc_empty, cw, lane);
  double2* Cp = x.C + jc0 * x.ld;
  auto wanted = [&](int jj) { return active && jc0 + jj < jend && jc0 + jj >= x.skip_n; };
  // C's values go straight to registers, requested when those of the sums' halves become free: copies
  // into shared memory (cp.async, by the threads themselves or by a warp of its own) arrive only after
  // 4 to 8 us beside the tensor pipe's operand reads, and values requested before the drain spill the
  // sums
  auto load_c = [&](int half, double2 (&cv)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      cv[q] = UPDATE && wanted(4 * half + q) ? Cp[(4 * half + q) * x.ld] : make_double2(0.0, 0.0);
  };
  if constexpr (UPDATE) {
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (wanted(q)) asm volatile("prefetch.global.L2 [%0];" ::"l"(Cp + q * x.ld));
  }
  unsigned long long H[16], L[16];
  const unsigned long long bh = 0ull - static_cast<unsigned long long>(cw.nchunks) * FoldPlan<G, NH>::bias(0, NH);
  const unsigned long long bl = 0ull - static_cast<unsigned long long>(cw.nchunks) * FoldPlan<G, NH>::bias(NH, G);
#pragma unroll
  for (int j = 0; j < 16; ++j) { H[j] = bh; L[j] = bl; }
  for (int c = 0; c < cw.nchunks; ++c) {
    if (!fold_part<G, NH, 0, split_group(G)>(x, acc_empty, lane, magic_mask, cw, H, L)) return false;
    if (!fold_part<G, NH, split_group(G), G>(x, acc_empty, lane, magic_mask, cw, H, L)) return false;
    ++*cw.cc;
  }
  if constexpr (KS) {
    // split K: the exact 64-bit halves of this unit's partial sums, column-major (coalesced over
    // the warp's rows); finish_split adds the units and rounds once
    if (x.rowok) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int col = x.n0 + x.c0 + j;
        if (col < x.n2)
          p.part[(static_cast<long long>(x.sp) * x.n2 + col) * p.m1 + x.row] =
              make_longlong2(static_cast<long long>(H[j]), static_cast<long long>(L[j]));
      }
    }
    return true;
  }
  const bool neg = !UPDATE && p.mode == EPI_IMINUS;
  const int* f = x.f + x.c0 / 2;                      // (zero past the problem's columns)
  bool near = exponent_near(x.er);
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) near = near && exponent_near(f[jj]);
  if (!__all_sync(0xffffffffu, near)) {
    // exponents at the ends of the binary64 range: one output at a time, rounded in 128 bits
#pragma unroll 1
    for (int jj = 0; jj < 8; ++jj) {
      unsigned long long hr = 0, lr = 0, hi = 0, li = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q == jj) { hr = H[2 * q]; lr = L[2 * q]; hi = H[2 * q + 1]; li = L[2 * q + 1]; }
      const int E = x.er + f[jj], jc = jc0 + jj;
      double zr = round_far(static_cast<long long>(neg ? 0ull - hr : hr), static_cast<long long>(neg ? 0ull - lr : lr), S8, E);
      double zi = round_far(static_cast<long long>(neg ? 0ull - hi : hi), static_cast<long long>(neg ? 0ull - li : li), S8, E);
      if (!wanted(jj)) continue;
      combine<UPDATE>(p, zr, zi, UPDATE ? Cp[jj * x.ld] : make_double2(0.0, 0.0), jc == x.grow);
      Cp[jj * x.ld] = make_double2(zr, zi);
    }
    return true;
  }
  // the first half's subtractions (FP64 pipe) stand before the second half's roundings (integer
  // pipes), and its stores after them, so that the two can overlap
  auto round_half = [&](int half, double (&z)[8]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t ehi = round_ehi<S8>(x.er + f[4 * half + q], neg);
#pragma unroll
      for (int h = 0; h < 2; ++h) z[2 * q + h] = round_hl<S8>(H[8 * half + 2 * q + h], L[8 * half + 2 * q + h], ehi);
    }
  };
  auto combine_half = [&](int half, double (&z)[8], const double2 (&cv)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) combine<UPDATE>(p, z[2 * q], z[2 * q + 1], cv[q], jc0 + 4 * half + q == x.grow);
  };
  auto store_half = [&](int half, const double (&z)[8]) {
    double2* d = Cp + 4 * half * x.ld;
#pragma unroll
    for (int q = 0; q < 4; ++q, d += x.ld) {
      if (wanted(4 * half + q)) *d = make_double2(z[2 * q], z[2 * q + 1]);
    }
  };
  double z0[8], z1[8];
  double2 c0[4], c1[4];
  load_c(0, c0);
  round_half(0, z0);
  combine_half(0, z0, c0);
  load_c(1, c1);
  round_half(1, z1);
  store_half(0, z0);
  combine_half(1, z1, c1);
  store_half(1, z1);
  return true;
}

// Epilogue of one 128 x 32 tile for G = 9 or 10 groups (S = 9, 10): as epilogue_fast with the groups
// in quads, each folded into a 64-bit sum per stacked column (8 columns a thread), combined to the
// 128-bit sum and rounded at the end of the tile.  Taken with a 128-bit shift and add and the
// conversion unit per accumulator and chunk instead, the drains bound 2048^3 at S = 10: 6.0 ms.
template <int G>
struct WidePlan {
  __host__ __device__ static constexpr int quad_end(int g) { return (g / 4) * 4 + 4 < G ? (g / 4) * 4 + 4 : G; }
  __host__ __device__ static constexpr int ng(int g) { return quad_end(g) - g >= 2 ? 2 : 1; }
  __host__ __device__ static constexpr int shift(int g) { return 8 * (quad_end(g) - g - ng(g)); }
  __host__ __device__ static constexpr unsigned long long bias(int quad) {
    unsigned long long b = 0;
    for (int g = 4 * quad; g < G && g < 4 * quad + 4; g += ng(g))
      b += static_cast<unsigned long long>(ng(g) == 2 ? MAGIC_PAIR : MAGIC_ONE) << shift(g);
    return b;
  }
};
template <int G, int GI, int GE, bool REDO>
__device__ __forceinline__ void wide_steps(uint32_t tbase, uint64_t* acc_empty, int lane, bool early, float& big,
                                           unsigned long long (&X)[3][8]) {
  using P = WidePlan<G>;
  if constexpr (GI < GE) {
    constexpr int BN = 32, ng = P::ng(GI);
    uint32_t v[8], u[8];
    tmem_ld8(tbase + GI * BN, v);
    if constexpr (ng == 2) tmem_ld8(tbase + (GI + 1) * BN, u);
    tmem_wait_ld();
    if constexpr (REDO) {
      if constexpr (ng == 2) refold_pair<P::shift(GI)>(X[GI / 4], v, u);
      else refold_one<P::shift(GI)>(X[GI / 4], v);
    } else {
      if (early) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&acc_empty[GI]);
          if constexpr (ng == 2) mbar_arrive(&acc_empty[GI + 1]);
        }
      }
      big = max_abs(big, v);
      if constexpr (ng == 2) big = max_abs(big, u);
      if constexpr (ng == 2) fold_pair<P::shift(GI)>(X[GI / 4], v, u);
      else fold_one<P::shift(GI)>(X[GI / 4], v);
    }
    wide_steps<G, GI + ng, GE, REDO>(tbase, acc_empty, lane, early, big, X);
  }
}
template <int G, int G0, int GE>
__device__ __forceinline__ bool wide_part(uint32_t tbase, uint64_t* acc_empty, int lane, uint32_t magic_mask,
                                          ChunkWait& cw, unsigned long long (&X)[3][8]) {
  if (!cw.part(G0 == 0 ? 0 : 1)) return false;
  constexpr uint32_t need = ((1u << (GE - G0)) - 1u) << G0;
  const bool known = (magic_mask & need) == need;
  float big = 0.0f;
  wide_steps<G, G0, GE, false>(tbase, acc_empty, lane, known, big, X);
  if (!known) {
    if (__any_sync(0xffffffffu, !(big < 4194304.0f))) wide_steps<G, G0, GE, true>(tbase, acc_empty, lane, false, big, X);
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
#pragma unroll
      for (int g = G0; g < GE; ++g) mbar_arrive(&acc_empty[g]);
    }
  }
  return true;
}
// the exact sums T of the thread's 8 columns over the tile's chunks
template <int G>
__device__ __forceinline__ bool wide_sums(uint32_t tbase, uint64_t* acc_empty, int lane, uint32_t magic_mask, ChunkWait& cw,
                                          __int128 (&T)[8]) {
  unsigned long long X[3][8];
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int j = 0; j < 8; ++j) X[q][j] = 0ull - static_cast<unsigned long long>(cw.nchunks) * WidePlan<G>::bias(q);
  for (int c = 0; c < cw.nchunks; ++c) {
    if (!wide_part<G, 0, split_group(G)>(tbase, acc_empty, lane, magic_mask, cw, X)) return false;
    if (!wide_part<G, split_group(G), G>(tbase, acc_empty, lane, magic_mask, cw, X)) return false;
    ++*cw.cc;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j)
    T[j] = (static_cast<__int128>(static_cast<long long>(X[0][j])) << (8 * (G - 4))) +
           (static_cast<__int128>(static_cast<long long>(X[1][j])) << (8 * (G - 8))) +
           static_cast<__int128>(static_cast<long long>(X[2][j]));
  return true;
}

// SF = 0: the slice count, pair schedule and epilogue variant are chosen at run time.  SF > 0:
// an instance for S = SF with the triangular pair set only, whose MMA issuer and epilogue
// contain just that schedule and group count -- the tensor pipe is fed markedly faster from
// the compact code (about 67 instead of 100 cycles per 128 x 64 x 16 MMA in a probe of the
// same issue loop) and the epilogue warps run a fraction of the instructions' footprint.
template <int BN, int SF, bool KS>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
slice_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const __grid_constant__ GemmParams p) {
  // Persistent: CTA b handles tiles b, b + gridDim.x, ... (column tile fastest, then row
  // tile, then problem).  The tile warp enumerates them; the other roles follow its ring.
  constexpr int COLS = BN / 4;            // stacked columns per epilogue thread
  const bool single = p.m == nullptr;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int S = SF > 0 ? SF : p.S;
  const int G = SF > 0 ? SF : p.ngroups;
  const uint32_t a_bytes = static_cast<uint32_t>(S) * GEMM_BM * 32;
  const uint32_t b_bytes = static_cast<uint32_t>(S) * BN * 32;
  const uint32_t stage_bytes = a_bytes + b_bytes;
  const int nstage = p.nstage;
  TileInfo<BN>* ring = reinterpret_cast<TileInfo<BN>*>(smem + nstage * stage_bytes);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + GEMM_TILE_SLOTS);
  uint64_t* empty = full + nstage;
  uint64_t* acc_full = empty + nstage;         // the first and the second part of the groups
  uint64_t* acc_empty = acc_full + 2;          // one per group accumulator
  uint64_t* done_bar = acc_empty + 16;
  uint64_t* stall_bar = done_bar + 1;          // the test hook's barrier: no thread arrives at it
  uint64_t* tile_full = stall_bar + 1;
  uint64_t* tile_empty = tile_full + GEMM_TILE_SLOTS;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(tile_empty + GEMM_TILE_SLOTS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < nstage; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(&acc_full[0], 1);
    mbar_init(&acc_full[1], 1);
    for (int i = 0; i < 16; ++i) mbar_init(&acc_empty[i], GEMM_EPI_WARPS);
    mbar_init(done_bar, 1);
    mbar_init(stall_bar, 1);
    // a slot's readers: the TMA and MMA threads and the epilogue warps
    for (int i = 0; i < GEMM_TILE_SLOTS; ++i) { mbar_init(&tile_full[i], 1); mbar_init(&tile_empty[i], 2 + GEMM_EPI_WARPS); }
    *abort_flag = 0;
    mbar_fence_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
  }
  if (warp == 1) tmem_alloc(tmem_holder, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  grid_dependency_wait();                      // the operands' split; C, exponents and tables of kernels before it
  if (p.stall_cycles > 0) {
    // failure-path test: one thread's bounded wait runs out (OZK_ERR_TIMEOUT, abort flag set)
    // before any TMA copy or MMA has been issued; every role then skips its loop
    if (threadIdx.x == 32) mbar_wait(stall_bar, 0, p.status, abort_flag, p.stall_cycles);
    __syncthreads();
  }
  const bool stalled = *abort_flag != 0;
  // the i-th tile's slot, once the tile warp has written it (null: a wait gave up)
  auto tile_at = [&](uint32_t i) -> const TileInfo<BN>* {
    const uint32_t slot = i % GEMM_TILE_SLOTS;
    return mbar_wait(&tile_full[slot], (i / GEMM_TILE_SLOTS) & 1, p.status, abort_flag) ? ring + slot : nullptr;
  };
  auto tile_done = [&](uint32_t i) { mbar_arrive(&tile_empty[i % GEMM_TILE_SLOTS]); };

  // the 20 warps start with 96 registers each (61440 for the CTA); warpgroup 0 keeps 64 and the
  // epilogue warpgroups take 104 (128 x 64 + 512 x 104 = 61440)
  if (warp < GEMM_CTRL_WARPS) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(GEMM_CTRL_REGS));
    if (warp == 0) {
      if (lane == 0) {
        // ---------------- TMA producer: one ring of stages across all tiles
        uint32_t kbc = 0;
        bool ok = !stalled;
        for (uint32_t i = 0; ok; ++i) {
          const TileInfo<BN>* ti = tile_at(i);
          if (!ti) { ok = false; break; }
          if (ti->end) break;
          const int za = ti->za, ra = ti->ra, n0 = ti->n0, kb0 = ti->kb0, kb1 = ti->kb1;
          tile_done(i);
          for (int kb = kb0; kb < kb1; ++kb, ++kbc) {
            const int stage = kbc % nstage;
            const uint32_t ph = kbc / nstage;
            if (kbc >= static_cast<uint32_t>(nstage) && !mbar_wait(&empty[stage], (ph - 1) & 1, p.status, abort_flag)) {
              ok = false;
              break;
            }
            uint8_t* sa = smem + stage * stage_bytes;
            mbar_arrive_expect_tx(&full[stage], stage_bytes);
            tma_load_4d(&tmA, sa, &full[stage], 2 * ra, 0, 2 * kb, za);
            tma_load_4d(&tmB, sa + a_bytes, &full[stage], 2 * n0, 0, 2 * kb, za);
          }
        }
        if (!ok || *abort_flag) {
          // another role gave up: let the copies this thread issued land before the CTA exits
          for (uint32_t k = kbc > static_cast<uint32_t>(nstage) ? kbc - nstage : 0u; k < kbc; ++k) {
            const long long t0 = clock64();
            while (!mbar_try_wait(&full[k % nstage], (k / nstage) & 1) && clock64() - t0 < kWaitBudget) {
            }
          }
        }
      }
    } else if (warp == 1) {
      // ---------------- MMA issuer.  Group g's accumulator of chunk cc may be overwritten once the
      // epilogue released it for chunk cc - 1 (per-group barrier).  The groups are two parts: over
      // the first and over the last K-blocks of a chunk (as many as the stages hold, less one), the
      // MMAs of all those K-blocks on the first part come before those on the second.  So the first
      // part is complete, and drained, while the second part's last MMAs run, and overwritten by the
      // next chunk or tile while the second part is drained: issued K-block by K-block, the tensor
      // pipe stood still for about 2000 cycles at each boundary (completion, wake-up of the
      // epilogue, its reads, release) even with an epilogue that read nothing -- 1.06 us next to
      // 0.55 us per K-block of a 128 x 64 tile at S = 7.
      if (elect_one()) {
        const bool parts = SF > 0 || in_parts<BN>(p, S);
        const int hold = parts ? max(1, nstage - 1) : 0;
        const int ga = parts ? split_group(S) : G;             // groups of the first part
        const uint64_t da = smem_desc_halves(smem_u32(smem), a_bytes / 2);
        const uint64_t db = smem_desc_halves(smem_u32(smem) + a_bytes, b_bytes / 2);
        const uint32_t a_lo = static_cast<uint32_t>(da), b_lo = static_cast<uint32_t>(db), hi = static_cast<uint32_t>(da >> 32);
        const uint32_t stage_units = stage_bytes / 16;
        uint32_t cc = 0, phase = 0;                            // chunk counter; parity of the ring's round
        int stage = 0;
        bool ok = !stalled;
        auto released = [&](int g0, int g1) -> bool {
          if (cc > 0)
            for (int g = g0; g < g1; ++g)
              if (!mbar_wait(&acc_empty[g], (cc - 1) & 1, p.status, abort_flag)) return false;
          tc_fence_after();
          return true;
        };
        auto issue = [&](auto part, int st, bool first) {
          constexpr int PART = decltype(part)::value;
          const uint32_t al = a_lo + st * stage_units, bl = b_lo + st * stage_units;
          if constexpr (SF > 0) issue_tri<SF, BN, PART>(first, tmem, al, bl, hi);
          else issue_dispatch<BN, PART>(p, S, first, tmem, al, bl, hi);
          if (PART != PART_FIRST) mma_commit(&empty[st]);
        };
        using First = std::integral_constant<int, PART_FIRST>;
        using Second = std::integral_constant<int, PART_SECOND>;
        using All = std::integral_constant<int, PART_ALL>;
        auto next = [&](int& st, uint32_t& ph) {
          if (++st == nstage) { st = 0; ph ^= 1; }
        };
        // `run` K-blocks from the ring's position on, the first part's MMAs of all of them first
        auto run_parts = [&](int run, bool opens, bool closes) -> bool {
          int st = stage;
          uint32_t ph = phase;
          if (opens && !released(0, ga)) return false;
          for (int q = 0; q < run; ++q) {
            if (!mbar_wait(&full[st], ph, p.status, abort_flag)) return false;
            tc_fence_after();
            issue(First{}, st, opens && q == 0);
            next(st, ph);
          }
          if (closes) mma_commit(&acc_full[0]);
          if (opens && !released(ga, G)) return false;
          for (int q = 0; q < run; ++q) {
            issue(Second{}, stage, opens && q == 0);
            next(stage, phase);
          }
          return true;
        };
        for (uint32_t i = 0; ok; ++i) {
          const TileInfo<BN>* ti = tile_at(i);
          if (!ti || ti->end) break;
          int left = ti->kb1 - ti->kb0;
          tile_done(i);
          for (; left > 0 && ok; left -= p.chunk_kb, ++cc) {
            const int n = min(left, p.chunk_kb);
            // K-blocks [0, nf) and [n - nl, n) in parts, those between whole
            const int nf = min(hold, (n + 1) / 2), nl = min(hold, n - nf);
            if (nf > 0) ok = run_parts(nf, true, nl == 0);
            else ok = released(0, G);
            for (int j = nf; j < n - nl && ok; ++j) {
              ok = mbar_wait(&full[stage], phase, p.status, abort_flag);
              if (!ok) break;
              tc_fence_after();
              issue(All{}, stage, j == 0);
              next(stage, phase);
            }
            if (ok && nl > 0) ok = run_parts(nl, false, true);
            if (!ok) break;
            if (!parts) mma_commit(&acc_full[0]);
            mma_commit(&acc_full[1]);
          }
        }
        // make sure no MMA is still in flight before TMEM is released
        mma_commit(done_bar);
        const long long t0 = clock64();
        while (!mbar_try_wait(done_bar, 0)) {
          if (clock64() - t0 > kWaitBudget) { flag_error(p.status, OZK_ERR_TIMEOUT); break; }
        }
      }
    } else if (warp == 2) {
      // ---------------- tile warp: finds the CTA's tiles and fills the ring.  With exact
      // enumeration (tile_prefix), problem z owns tiles [prefix[z], prefix[z + 1]) laid out by
      // box_tiles.  Otherwise problem z owns tiles [z tpp, (z + 1) tpp) of the largest problem's
      // grid: the tile rows below its skip box (all columns, column tile fastest), then the tiles
      // right of the box in the rows beside it; tiles wholly inside the box are never enumerated,
      // and indices past the problem's own tiles or outside its extent are passed over.
      const int ntx = p.ntx, nty = p.nty;
      // KS instances run split K (p.ksplit units per tile); the others one unit per tile
      const int ks = KS ? (p.ksplit > 1 ? p.ksplit : 1) : 1;
      const int ntiles = (p.tile_prefix ? p.tile_prefix[p.batch] : p.tpp * p.batch) * ks;
      int zcur = 0;
      auto tile_of = [&](int t, int& z, int& m0, int& n0, int& m_z, int& n2_z) -> bool {
        if (p.tile_prefix) {
          // a CTA's tiles come in order, so the search gallops on from its last problem
          int lo = zcur, step = 1;
          while (lo + step < p.batch && p.tile_prefix[lo + step] <= t) { lo += step; step <<= 1; }
          int hi = min(lo + step, p.batch);
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (p.tile_prefix[mid] <= t) lo = mid; else hi = mid;
          }
          z = zcur = lo;
          const int r = t - p.tile_prefix[z];
          m_z = p.m[z];
          n2_z = 2 * p.n[z];
          const BoxTiles bt = box_tiles(m_z, n2_z, p.skm ? p.skm[z] : 0, p.skn ? p.skn[z] : 0, BN);
          if (r < bt.ku * bt.xu) {                  // beside the box (rows clipped at its edge)
            const int y = r / bt.xu;
            m0 = y * GEMM_BM;
            n0 = bt.n0u + (r - y * bt.xu) * BN;
            m_z = bt.mu;
          } else {                                  // below the box, or the whole grid
            const int r2 = r - bt.ku * bt.xu, y = r2 / bt.ntx;
            m0 = bt.m0l + y * GEMM_BM;
            n0 = (r2 - y * bt.ntx) * BN;
          }
          return true;
        }
        z = t / p.tpp;
        const int r = t - z * p.tpp;
        m_z = single ? p.m1 : p.m[z];
        n2_z = 2 * (single ? p.n1 : p.n[z]);
        const int km = single ? p.skm1 : (p.skm ? p.skm[z] : 0);
        const int kn = single ? p.skn1 : (p.skn ? p.skn[z] : 0);
        const int ky = min(km / GEMM_BM, nty), kx = min((2 * kn) / BN, ntx);
        const int count1 = (nty - ky) * ntx;
        int x, y;
        if (r < count1) {
          y = ky + r / ntx;
          x = r - (y - ky) * ntx;
        } else {
          const int w = ntx - kx, r2 = r - count1;
          if (w <= 0 || r2 >= ky * w) return false;
          y = r2 / w;
          x = kx + (r2 - y * w);
        }
        m0 = y * GEMM_BM;
        n0 = x * BN;
        return m0 < m_z && n0 < n2_z;
      };
      const bool outputs = p.mode != EPI_GROUPS && p.mode != EPI_RESIDUES;
      uint32_t i = 0;
      for (int t = blockIdx.x; !stalled; t += gridDim.x) {
        int z = 0, m0 = 0, n0 = 0, m_z = 0, n2_z = 0;
        const bool end = t >= ntiles;
        if (!end && !tile_of(t / ks, z, m0, n0, m_z, n2_z)) continue;
        const uint32_t slot = i % GEMM_TILE_SLOTS;
        if (i >= GEMM_TILE_SLOTS) {
          int got = lane == 0 ? mbar_wait(&tile_empty[slot], ((i / GEMM_TILE_SLOTS) - 1) & 1, p.status, abort_flag) : 0;
          if (!__shfl_sync(0xffffffffu, got, 0)) break;
        }
        TileInfo<BN>& ti = ring[slot];
        if (!end) {
          int za = z, ra = 0;
          if (p.remap) { const int2 rm = p.remap[z]; za = rm.x; ra = rm.y; }
          const int rows = min(m_z - m0, GEMM_BM);
          if (lane == 0) {
            const int nkb = p.k ? (p.k[z] + 7) >> 3 : p.kblocks;          // the problem's own K
            const int sp = t - (t / ks) * ks, nch = (nkb + p.chunk_kb - 1) / p.chunk_kb;
            ti.za = za; ti.ra = ra + m0; ti.n0 = n0;
            ti.kb0 = sp * nch / ks * p.chunk_kb;
            ti.kb1 = min(nkb, (sp + 1) * nch / ks * p.chunk_kb);
            ti.sp = sp; ti.z = z; ti.row0 = m0; ti.rows = rows; ti.n2 = n2_z;
            ti.skip_rows = (single ? p.skm1 : (p.skm ? p.skm[z] : 0)) - m0;
            ti.skip_cols = single ? p.skn1 : (p.skn ? p.skn[z] : 0);
          }
          if (outputs) {
#pragma unroll
            for (int q = 0; q < GEMM_BM / 32; ++q) {
              const int r = lane + 32 * q;
              RowInfo o{nullptr, 0, 0};
              int e = 0;
              if (r < rows) {
                o = out_row(p, single, z, m0 + r, za, ra + m0 + r);
                e = p.e[za * p.e_stride + ra + m0 + r] + p.base_exp;
              }
              ti.row[r] = o;
              ti.e[r] = e;
            }
            if (lane < BN / 2) ti.f[lane] = n0 / 2 + lane < n2_z / 2 ? p.f[za * p.f_stride + n0 / 2 + lane] : 0;
          }
        }
        if (lane == 0) ti.end = end;
        __syncwarp();
        if (lane == 0) mbar_arrive(&tile_full[slot]);
        ++i;
        if (end) break;
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(GEMM_EPI_REGS));
    // ---------------- epilogue: 16 warps = 4 TMEM lane quadrants x 4 column slabs
    const int quad = warp & 3;
    const int slab = (warp - GEMM_CTRL_WARPS) >> 2;
    const int c0 = slab * COLS;                  // first local stacked column of this thread
    const uint32_t tbase = tmem + (static_cast<uint32_t>(quad * 32) << 16) + c0;
    const bool magic = p.magic != 0;
    const bool update = p.mode == EPI_LU || p.mode == EPI_GENERAL;
    const uint32_t magic_mask = magic ? 0xFFFFFFFFu : static_cast<uint32_t>(p.magic_mask);
    uint32_t cc = 0;
    bool ok = !stalled;
    for (uint32_t i = 0; ok; ++i) {
      const TileInfo<BN>* ti = tile_at(i);
      if (!ti) { ok = false; break; }
      if (ti->end) break;
      const int rl = quad * 32 + lane;           // row in the tile
      const int unch = (ti->kb1 - ti->kb0 + p.chunk_kb - 1) / p.chunk_kb;    // exactness chunks of this unit
      if constexpr (COLS == 16) {
        if (G <= 8 && (SF > 0 || !p.wide) && p.mode != EPI_GROUPS && p.mode != EPI_RESIDUES) {
          EpiCtx x;
          const RowInfo o = ti->row[rl];
          x.row = ti->row0 + rl; x.n2 = ti->n2; x.n0 = ti->n0; x.c0 = c0; x.tbase = tbase; x.sp = ti->sp;
          x.skip_n = rl < ti->skip_rows ? ti->skip_cols : 0;
          x.C = o.C; x.ld = o.ld; x.grow = o.grow;
          x.rowok = o.C != nullptr;
          x.jlim = (p.crow && p.crow_n) ? o.ld : 0x7FFFFFFF;
          x.er = ti->e[rl];
          x.f = ti->f;
          ChunkWait cw{acc_full, unch, &cc, p.status, abort_flag};
          bool e_ok;
          if constexpr (KS) {
            // (a split K's sums are combined by the finishing kernel)
#define OZK_EPI(GG) case GG: e_ok = epilogue_fast<GG, false, true, false>(p, x, acc_empty, magic_mask, lane, cw); break
            if constexpr (SF > 0) {
              switch (SF) { OZK_EPI(SF); default: e_ok = false; }
            } else {
              switch (G) { OZK_EPI(1); OZK_EPI(2); OZK_EPI(3); OZK_EPI(4); OZK_EPI(5); OZK_EPI(6); OZK_EPI(7); OZK_EPI(8); default: e_ok = false; }
            }
#undef OZK_EPI
          } else {
#define OZK_EPI(GG) \
  case GG: \
    if (GG <= 5 && p.fit64) \
      e_ok = update ? epilogue_fast<GG, (GG <= 5), false, true>(p, x, acc_empty, magic_mask, lane, cw) \
                    : epilogue_fast<GG, (GG <= 5), false, false>(p, x, acc_empty, magic_mask, lane, cw); \
    else \
      e_ok = update ? epilogue_fast<GG, false, false, true>(p, x, acc_empty, magic_mask, lane, cw) \
                    : epilogue_fast<GG, false, false, false>(p, x, acc_empty, magic_mask, lane, cw); \
    break
            if constexpr (SF > 0) {
              switch (SF) { OZK_EPI(SF); default: e_ok = false; }
            } else {
              switch (G) { OZK_EPI(1); OZK_EPI(2); OZK_EPI(3); OZK_EPI(4); OZK_EPI(5); OZK_EPI(6); OZK_EPI(7); OZK_EPI(8); default: e_ok = false; }
            }
#undef OZK_EPI
          }
          if (!e_ok) { ok = false; break; }
          __syncwarp();
          if (lane == 0) tile_done(i);
          continue;
        }
      }
      if constexpr (SF == 0 || BN == 32) {       // 64-column compile-time instances take only the fast epilogues
        const bool horner = unch == 1;
        const int row = ti->row0 + rl, n0 = ti->n0, n2_z = ti->n2, z = ti->z;
        const bool rowok = rl < ti->rows;
        __int128 T[COLS];
#pragma unroll
        for (int j = 0; j < COLS; ++j) T[j] = 0;
        if constexpr (SF > 0 && BN == 32) {
          ChunkWait cw{acc_full, unch, &cc, p.status, abort_flag};
          if (!wide_sums<SF>(tbase, acc_empty, lane, magic_mask, cw, T)) ok = false;
        }
        for (int c = 0; SF == 0 && c < unch; ++c, ++cc) {
          // (every group after the second part: these forms are not bound by the boundary)
          if (!mbar_wait(&acc_full[0], cc & 1, p.status, abort_flag) ||
              !mbar_wait(&acc_full[1], cc & 1, p.status, abort_flag)) { ok = false; break; }
          tc_fence_after();
          for (int gi = 0; gi < G; ++gi) {
            uint32_t v[COLS];
            if constexpr (COLS == 16) tmem_ld16(tbase + gi * BN, v); else tmem_ld8(tbase + gi * BN, v);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[gi]);       // group gi may be overwritten now
            if (p.mode == EPI_RESIDUES) {
              // this chunk's exact integer value of group gi (|v| <= 2^24), added to the product
              if (rowok) {
                int* dst = p.resid + ((static_cast<long long>(z) * G + gi) * p.m1 + row) * p.ldres;
#pragma unroll
                for (int j = 0; j < COLS; ++j) {
                  const int col = n0 + c0 + j;
                  if (col < n2_z) atomicAdd(&dst[col], __float2int_rn(__uint_as_float(v[j])));
                }
              }
            } else if (p.mode == EPI_GROUPS) {
              if (z == 0 && rowok) {
#pragma unroll
                for (int j = 0; j < COLS; ++j) {
                  const int col = n0 + c0 + j;
                  if (col < n2_z) {
                    const long long iv = __float2int_rn(__uint_as_float(v[j]));
                    atomicAdd(reinterpret_cast<unsigned long long*>(&p.groups[(static_cast<long long>(gi) * p.m1 + row) * n2_z + col]),
                              static_cast<unsigned long long>(iv));
                  }
                }
              }
            } else if (horner) {
              // one chunk: Horner over the groups, highest weight first, 8-bit steps
#pragma unroll
              for (int j = 0; j < COLS; ++j) T[j] = (T[j] << 8) + static_cast<__int128>(acc_to_int(v[j], magic));
            } else {
              const int w = 8 * (G - 1 - gi);
#pragma unroll
              for (int j = 0; j < COLS; ++j) T[j] += static_cast<__int128>(__float2int_rn(__uint_as_float(v[j]))) << w;
            }
          }
        }
        if (!ok) break;
        if (p.mode != EPI_GROUPS && p.mode != EPI_RESIDUES && ti->row[rl].C) {
          const RowInfo o = ti->row[rl];
          const int jlim = (p.crow && p.crow_n) ? o.ld : 0x7FFFFFFF;
          const int skip_n = rl < ti->skip_rows ? ti->skip_cols : 0;
          const bool needC = p.mode == EPI_LU || p.mode == EPI_GENERAL;
          const bool neg = p.mode == EPI_IMINUS;
#pragma unroll
          for (int j = 0; j < COLS; j += 2) {
            const int jc = (n0 + c0 + j) >> 1;          // complex column
            if (2 * jc < n2_z && jc >= skip_n && jc < jlim) {
              const int E = ti->e[rl] + ti->f[(c0 + j) >> 1];
              double2* dst = o.C + static_cast<long long>(jc) * o.ld;
              double zr = round_scaled_dev(neg ? -T[j] : T[j], E), zi = round_scaled_dev(neg ? -T[j + 1] : T[j + 1], E);
              if (needC) combine<true>(p, zr, zi, *dst, false);
              else combine<false>(p, zr, zi, make_double2(0.0, 0.0), jc == o.grow);
              *dst = make_double2(zr, zi);
            }
          }
        }
        __syncwarp();
        if (lane == 0) tile_done(i);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int BN, int SF, bool KS>
inline void launch_instance(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, int grid, size_t smem,
                            cudaStream_t st) {
  // the limit is the kernel's, not the launch's: the same value from every call, so that a thread whose
  // launch needs less cannot lower it between another's setting and launch
  cudaFuncSetAttribute(slice_gemm_kernel<BN, SF, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM_MAX);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(GEMM_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1] = {pdl_attribute(st)};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, slice_gemm_kernel<BN, SF, KS>, ta, tb, p);
}
// the instances of S = 3..5, of S = 6..8 (split K: S = 7) and of S = 9, 10, each in its own
// translation unit
void launch_slice_gemm_s345(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, int grid, size_t smem,
                            cudaStream_t st);
void launch_slice_gemm_s910(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, int grid, size_t smem,
                            cudaStream_t st);
void launch_slice_gemm_s678(const CUtensorMap& ta, const CUtensorMap& tb, const GemmParams& p, int grid, size_t smem,
                            cudaStream_t st);

}  // namespace ozk
