// Exponent scan and slice split (paper Sec. 2.2: slices by significant bits with exponent
// alignment).  The S balanced int8 digits of every real scalar of an operand are written as fp16
// values in the K-major layout the tensor-core kernel loads with TMA:
//   out[z][h][s][row][8]   (8 fp16 = 16 bytes: one row of a tensor-core core matrix)
// K-block kb covers the elements l = 8 kb .. 8 kb + 7 of a row; half h = 2 kb holds the digits of
// their first scalar, h = 2 kb + 1 those of the second:
//   left operand  (side 0): row r       first Re x_rl, second Im x_rl
//   right operand (side 1): row 2r      first Re,      second -Im (digit-wise)
//                           row 2r + 1  first Im,      second Re
// (sums over K run over all the halves, so their order is free).  A last K-block of at most 4
// elements is packed into half 2 kb alone: 4 values of the first scalar, then 4 of the second;
// the half after it is zero where the plane has one.  Rows follow each other at 16 bytes for a
// fixed (h, s), so the 32 lanes of a warp, one row each, store 512 (left) or 1024 (right)
// contiguous bytes, and a 128-row operand tile is 2 S runs of 2 KB for the TMA (with the digits of
// a row K-contiguous instead, the tile's runs are the 32 bytes of a K-block and row: 1344 of them
// for S = 7, which the TMA fetches at about one per clock, 656 ns per K-block measured with the
// tensor work left out).  All integer work, no FP64 arithmetic.
#include <algorithm>
#include <type_traits>

#include "ozk_params.cuh"

namespace ozk {

constexpr int SPLIT_ROWS = 32;               // rows of a CTA: one per lane
constexpr int SPLIT_MAX_WARPS = 8;           // a warp takes one K-block (8 elements) at a time
constexpr int SPLIT_MAX_KG = 8;              // CTAs of a cluster that share a row block's K-blocks
constexpr int SPLIT_GMAX_KG = 16, SPLIT_GMAX_KB = 384;   // row maxima by a launch of their own: launch_split

// Digits of 8 elements for a compile-time slice count SF <= 10 (nbits = 8 SF - 1; 64-bit images, 96-bit
// ones for SF = 9 and 10), with no dependent chain per digit.  With C = 128 (1 + 256 + ... + 256^(SF-2)), Y = X + C holds
// the balanced digits d_s + 128 of the SF - 1 lower places as its low bytes and the top digit
// as Y >> 8 (SF - 1): X = sum_s d_s 256^s with every lower d_s in [-128, 127], so adding 128
// at each lower place lifts it into [0, 255] without carries, and base-256 digits are unique.
// Plane SF - 1 - s takes byte s of Y.  Two elements' bytes go into the halves of one word,
// offset by 0x6580 = (bit pattern of 1536 in binary16) - 128, which makes each half the bit
// pattern of 1536 + d (the binade [1024, 2048) has unit spacing); one packed subtraction of
// 1536 leaves d, and subtracting the word from 1536 leaves -d, both exact (+0 for d = 0, as
// the int -> half conversion gives).  The top digit (|d| <= 128) takes the offset 0x6600; for
// SF = 8 (|X| < 2^63, so X + C may pass 2^63) it is taken from floor((X + C) / 2), C being even.
__host__ __device__ constexpr long long digit_bias(int S) {
  long long c = 0;
  for (int s = 0; s < S - 1; ++s) c = c * 256 + 128;
  return c;
}

__device__ __forceinline__ uint32_t half2_bits(__half2 h) {
  return static_cast<uint32_t>(__half_as_ushort(__low2half(h))) |
         (static_cast<uint32_t>(__half_as_ushort(__high2half(h))) << 16);
}
__device__ __forceinline__ __half2 bits_half2(uint32_t w) {
  return __halves2half2(__ushort_as_half(static_cast<unsigned short>(w & 0xFFFFu)),
                        __ushort_as_half(static_cast<unsigned short>(w >> 16)));
}
// d (NEG: -d) of both halves of a biased pair
template <bool NEG>
__device__ __forceinline__ uint32_t pair_digits(uint32_t biased) {
  const __half2 k1536 = __half2half2(__ushort_as_half(0x6600));
  return half2_bits(NEG ? __hsub2(k1536, bits_half2(biased)) : __hsub2(bits_half2(biased), k1536));
}

// the biased pair of the top digits (SF < 8) of two images Y, given by their words
template <int SF>
__device__ __forceinline__ uint32_t top_pair(uint32_t al, uint32_t ah, uint32_t bl, uint32_t bh) {
  constexpr int sh = 8 * (SF - 1);
  uint32_t ta, tb;
  if constexpr (sh >= 32) {
    ta = static_cast<uint32_t>((static_cast<int>(ah) >> (sh - 32)) + 0x6600);
    tb = static_cast<uint32_t>((static_cast<int>(bh) >> (sh - 32)) + 0x6600);
  } else {                                       // the top digit fits in 9 bits: low word after the shift
    ta = __funnelshift_r(al, ah, sh) + 0x6600u;
    tb = __funnelshift_r(bl, bh, sh) + 0x6600u;
  }
  return __byte_perm(ta, tb, 0x5410);
}

// where the digits of one row and K-block go: uint4 words of the planes (see the layout above)
template <int SIDE>
struct SplitDst {
  uint4* out;                // plane (h = 2 kb, s = 0), row r (left) or 2 r (right)
  int splane;                // uint4 words from slice s to s + 1 (= out_rows)
  long long hplane;          // from half h to h + 1 (= S out_rows)
  bool tail4;                // at most 4 elements: packed into the first half
  bool has2;                 // the plane has the second half
};

// the 4 words (8 fp16) of each scalar of one slice: r first scalar, i the second, n = -i
template <int SIDE>
__device__ __forceinline__ void store_slice(const SplitDst<SIDE>& d, int s, const uint32_t (&r)[4], const uint32_t (&i)[4],
                                            const uint32_t (&n)[4]) {
  uint4* o = d.out + static_cast<long long>(s) * d.splane;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  if (!d.tail4) {
    if constexpr (SIDE == 0) {
      o[0] = make_uint4(r[0], r[1], r[2], r[3]);
      o[d.hplane] = make_uint4(i[0], i[1], i[2], i[3]);
    } else {
      o[0] = make_uint4(r[0], r[1], r[2], r[3]);
      o[1] = make_uint4(i[0], i[1], i[2], i[3]);
      o[d.hplane] = make_uint4(n[0], n[1], n[2], n[3]);
      o[d.hplane + 1] = make_uint4(r[0], r[1], r[2], r[3]);
    }
  } else {
    if constexpr (SIDE == 0) {
      o[0] = make_uint4(r[0], r[1], i[0], i[1]);
    } else {
      o[0] = make_uint4(r[0], r[1], n[0], n[1]);
      o[1] = make_uint4(i[0], i[1], r[0], r[1]);
      if (d.has2) o[d.hplane + 1] = zero;
    }
    if (d.has2) o[d.hplane] = zero;
  }
}

// The integer image X = trunc(x 2^(nbits - e)) of |x| < 2^e, e >= -1021, nbits =
// 8 SF - 1: the 53-bit significand, shifted left by the constant max(0, nbits - 53) that no element
// exceeds, then right.  (Rows flagged non-finite have e = 0, which does not bound their finite
// elements: those are cut to the significand's range.)
template <int SF>
__device__ __forceinline__ long long image_fixed(long long bits, int e) {
  constexpr int nbits = 8 * SF - 1, left = nbits > 53 ? (nbits - 53) % 64 : 0;
  const int ex = static_cast<int>(bits >> 52) & 0x7FF;
  const unsigned long long man = static_cast<unsigned long long>(bits) & ((1ull << 52) - 1ull);
  const unsigned long long M = ex == 0 ? man : (man | (1ull << 52));
  const int right = e + (left + 1075 - nbits) - max(ex, 1);
  const long long mag = static_cast<long long>((M << left) >> min(max(right, 0), 63));
  return bits < 0 ? -mag : mag;
}

// the same for SF = 9, 10 plus the bias: Y = C + X in three words (the significand shifted left by up
// to 18 or 26 bits)
template <int SF>
__device__ __forceinline__ void image_wide(long long bits, int e, uint32_t& w0, uint32_t& w1, uint32_t& w2) {
  constexpr int nbits = 8 * SF - 1, left = nbits - 53;
  const int ex = static_cast<int>(bits >> 52) & 0x7FF;
  const unsigned long long man = static_cast<unsigned long long>(bits) & ((1ull << 52) - 1ull);
  const unsigned long long M = ex == 0 ? man : (man | (1ull << 52));
  const int right = max(e + (left + 1075 - nbits) - max(ex, 1), 0);
  const int up = max(left - right, 0);
  unsigned long long lo = (M << up) >> min(max(right - left, 0), 63);
  uint32_t hi = up > 11 ? static_cast<uint32_t>(M >> (64 - up)) : 0u;
  if (bits < 0) {
    hi = ~hi + (lo == 0ull ? 1u : 0u);
    lo = 0ull - lo;
  }
  constexpr unsigned long long Clo = 0x8080808080808080ull;             // bytes 0..7
  constexpr uint32_t Chi = SF == 9 ? 0u : 0x80u;                         // byte 8 (SF = 10)
  const unsigned long long s = lo + Clo;
  hi += Chi + (s < lo ? 1u : 0u);
  w0 = static_cast<uint32_t>(s);
  w1 = static_cast<uint32_t>(s >> 32);
  w2 = hi;
}

template <int SF, int SIDE>
__device__ __forceinline__ void emit_fixed(const SplitDst<SIDE>& d, const longlong2 (&v)[8], int e) {
  constexpr long long C = SF <= 8 ? digit_bias(SF <= 8 ? SF : 8) : 0;
  uint32_t rl[8], rh[8], il[8], ih[8];                    // low and high words of Y
  uint32_t tr[4], ti[4];                                  // SF = 8: the top digits, two a word
  uint32_t rx[8], ix[8];                                  // SF > 8: third words
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if constexpr (SF > 8) {
      image_wide<SF>(v[q].x, e, rl[q], rh[q], rx[q]);
      image_wide<SF>(v[q].y, e, il[q], ih[q], ix[q]);
      continue;
    }
    const long long xr = image_fixed<SF>(v[q].x, e), xi = image_fixed<SF>(v[q].y, e);
    const unsigned long long a = static_cast<unsigned long long>(xr) + C, b = static_cast<unsigned long long>(xi) + C;
    rl[q] = static_cast<uint32_t>(a); rh[q] = static_cast<uint32_t>(a >> 32);
    il[q] = static_cast<uint32_t>(b); ih[q] = static_cast<uint32_t>(b >> 32);
    if constexpr (SF == 8) {
      const uint32_t ta = static_cast<uint32_t>(static_cast<int>(((xr >> 1) + C / 2) >> 55) + 0x6600);
      const uint32_t tb = static_cast<uint32_t>(static_cast<int>(((xi >> 1) + C / 2) >> 55) + 0x6600);
      tr[q / 2] = q & 1 ? __byte_perm(tr[q / 2], ta, 0x5410) : ta;
      ti[q / 2] = q & 1 ? __byte_perm(ti[q / 2], tb, 0x5410) : tb;
    }
  }
#pragma unroll
  for (int s = SF - 1; s >= 0; --s) {
    const int k = SF - 1 - s;                               // byte of Y (s > 0)
    uint32_t r[4], i[4], n[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      uint32_t br, bi;
      if (s > 0) {
        const uint32_t sel = static_cast<uint32_t>(k & 3) | (static_cast<uint32_t>((k & 3) + 4) << 8);
        br = (__byte_perm(k < 4 ? rl[2 * h] : (k < 8 ? rh[2 * h] : rx[2 * h]),
                          k < 4 ? rl[2 * h + 1] : (k < 8 ? rh[2 * h + 1] : rx[2 * h + 1]), sel) & 0x00FF00FFu) +
             0x65806580u;
        bi = (__byte_perm(k < 4 ? il[2 * h] : (k < 8 ? ih[2 * h] : ix[2 * h]),
                          k < 4 ? il[2 * h + 1] : (k < 8 ? ih[2 * h + 1] : ix[2 * h + 1]), sel) & 0x00FF00FFu) +
             0x65806580u;
      } else if constexpr (SF == 8) {
        br = tr[h];
        bi = ti[h];
      } else if constexpr (SF > 8) {                        // the top digit: third word from byte SF - 9 on
        constexpr int sh = 8 * (SF - 9);
        br = __byte_perm(static_cast<uint32_t>((static_cast<int>(rx[2 * h]) >> sh) + 0x6600),
                         static_cast<uint32_t>((static_cast<int>(rx[2 * h + 1]) >> sh) + 0x6600), 0x5410);
        bi = __byte_perm(static_cast<uint32_t>((static_cast<int>(ix[2 * h]) >> sh) + 0x6600),
                         static_cast<uint32_t>((static_cast<int>(ix[2 * h + 1]) >> sh) + 0x6600), 0x5410);
      } else {
        br = top_pair<SF>(rl[2 * h], rh[2 * h], rl[2 * h + 1], rh[2 * h + 1]);
        bi = top_pair<SF>(il[2 * h], ih[2 * h], il[2 * h + 1], ih[2 * h + 1]);
      }
      r[h] = pair_digits<false>(br);
      i[h] = pair_digits<false>(bi);
      n[h] = pair_digits<true>(bi);
    }
    store_slice(d, s, r, i, n);
  }
}

// Any S (run time): digits one at a time from 64-bit (nbits <= 62) or 128-bit images.  dbg: the
// int16 copy of the test hook, [S][out_rows][2 K].
template <bool W64, int SIDE>
__device__ __forceinline__ void emit_generic(const SplitParams& p, const SplitDst<SIDE>& d, const longlong2 (&v)[8], int e,
                                             int row, int l0, int K, int16_t* dbg) {
  using Int = typename std::conditional<W64, long long, __int128>::type;
  Int Xr[8], Xi[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if constexpr (W64) {
      Xr[q] = integer_image64(__longlong_as_double(v[q].x), e, p.nbits);
      Xi[q] = integer_image64(__longlong_as_double(v[q].y), e, p.nbits);
    } else {
      Xr[q] = integer_image(__longlong_as_double(v[q].x), e, p.nbits);
      Xi[q] = integer_image(__longlong_as_double(v[q].y), e, p.nbits);
    }
  }
  for (int s = p.S - 1; s >= 0; --s) {
    uint32_t r[4], i[4], n[4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      int dr, di;
      if constexpr (W64) {
        dr = s ? next_digit64(Xr[q]) : static_cast<int>(Xr[q]);
        di = s ? next_digit64(Xi[q]) : static_cast<int>(Xi[q]);
      } else {
        dr = s ? next_digit(Xr[q]) : static_cast<int>(Xr[q]);
        di = s ? next_digit(Xi[q]) : static_cast<int>(Xi[q]);
      }
      const uint32_t hr = __half_as_ushort(__int2half_rn(dr)), hi = __half_as_ushort(__int2half_rn(di)),
                     hn = __half_as_ushort(__int2half_rn(-di));
      if (q & 1) { r[q / 2] |= hr << 16; i[q / 2] |= hi << 16; n[q / 2] |= hn << 16; }
      else { r[q / 2] = hr; i[q / 2] = hi; n[q / 2] = hn; }
      if (dbg && l0 + q < K) {
        const int l = l0 + q;
        if (SIDE == 0) {
          int16_t* o = dbg + (static_cast<long long>(s) * p.out_rows + row) * 2LL * K;
          o[l] = static_cast<int16_t>(dr);
          o[K + l] = static_cast<int16_t>(di);
        } else {
          int16_t* o = dbg + (static_cast<long long>(s) * p.out_rows + 2LL * row) * 2LL * K;
          o[l] = static_cast<int16_t>(dr);
          o[K + l] = static_cast<int16_t>(-di);
          o[2LL * K + l] = static_cast<int16_t>(di);
          o[3LL * K + l] = static_cast<int16_t>(dr);
        }
      }
    }
    store_slice(d, s, r, i, n);
  }
}

__device__ __forceinline__ unsigned long long abs_bits(long long x) {
  return static_cast<unsigned long long>(x) & 0x7FFFFFFFFFFFFFFFull;
}

// 8 elements (zero past K) of logical row r from element l0 on; trans: they are contiguous
__device__ __forceinline__ void load_block(const SplitParams& p, const longlong2* __restrict__ P, long long ld, int r,
                                           int l0, int K, longlong2 (&v)[8]) {
  const longlong2* s = P + (p.trans ? l0 + r * ld : r + l0 * ld);
  const long long step = p.trans ? 1 : ld;
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = l0 + q < K ? s[q * step] : make_longlong2(0, 0);
}

// largest |Re|, |Im| bit pattern (non-finite values compare above every finite one)
__device__ __forceinline__ unsigned long long block_max(const longlong2 (&v)[8]) {
  unsigned long long mx = 0ull;
#pragma unroll
  for (int q = 0; q < 8; ++q) mx = max(mx, max(abs_bits(v[q].x), abs_bits(v[q].y)));
  return mx;
}

// Both operands of one emulated GEMM in one launch: blockIdx.z selects the side.  A CTA owns 32
// rows, one per lane; warp w takes the K-blocks w, w + nwarps, ... of its share.  With kgroups > 1
// the CTAs of a cluster share a row block's K-blocks and exchange their row maxima through
// distributed shared memory; GIVEN: the row maxima are there already (gmax: split_rowmax_kernel) and
// the CTAs, no cluster then, have nothing to exchange.  A share of at most one K-block per warp is read from memory once
// and kept in registers between the maximum and the digits; longer shares are read twice.  Non-finite
// scalars flag OZK_ERR_NONFINITE, make their row's exponent 0 and are split as zero.
template <int SF, bool W64, int SIDE, bool GIVEN>
__device__ __forceinline__ void split_rows(const SplitParams& p, unsigned long long (&wmax)[SPLIT_MAX_WARPS][SPLIT_ROWS],
                                           unsigned long long (&cmax)[SPLIT_MAX_KG][SPLIT_ROWS]) {
  const int z = blockIdx.y;
  const bool single = p.X == nullptr;
  const int R = single ? p.rows1 : p.rows[z];
  const int K = single ? p.k1 : p.kdim[z];
  const int kgs = p.kgroups;
  const int rank = static_cast<int>(blockIdx.x) % kgs;
  const int r0 = (static_cast<int>(blockIdx.x) / kgs) * SPLIT_ROWS;
  if (r0 >= R) return;                                 // the same for every CTA of the cluster
  if (!GIVEN && kgs > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const longlong2* __restrict__ P = reinterpret_cast<const longlong2*>(single ? p.X1 + z * p.zstride1 : p.X[z]);
  const long long ld = single ? p.ld1 : p.ld[z];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int r = r0 + lane;
  const bool rok = r < R;
  const int nkb = (K + 7) >> 3, share = (nkb + kgs - 1) / kgs;
  const int kb0 = rank * share, kb1 = min(nkb, kb0 + share);
  const bool resident = !GIVEN && share <= nw;

  longlong2 v[8];
  unsigned long long mx = 0ull;
  if (rok && GIVEN) {
    mx = p.gmax[z * p.exp_stride + r];
  } else if (rok) {
    if (resident) {
      if (kb0 + warp < kb1) {
        load_block(p, P, ld, r, 8 * (kb0 + warp), K, v);
        mx = block_max(v);
      }
    } else {
      for (int kb = kb0 + warp; kb < kb1; kb += nw) {
        load_block(p, P, ld, r, 8 * kb, K, v);
        mx = max(mx, block_max(v));
      }
    }
  }
  if constexpr (!GIVEN) {
    wmax[warp][lane] = mx;
    __syncthreads();
    for (int w = 0; w < nw; ++w) mx = max(mx, wmax[w][lane]);
  }
  if (!GIVEN && kgs > 1) {
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");      // every peer has started
    if (warp < kgs) {
      uint32_t dst;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(smem_u32(&cmax[rank][lane])), "r"(warp));
      asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(dst), "l"(mx) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    for (int c = 0; c < kgs; ++c) mx = max(mx, cmax[c][lane]);
  }
  const bool bad = mx >= 0x7FF0000000000000ull;
  const int e = bad ? 0 : frexp_exponent_from_bits(mx);
  if (warp == 0 && rank == 0 && rok) {
    if (bad) flag_error(p.status, OZK_ERR_NONFINITE);
    p.exps[z * p.exp_stride + r] = e;
  }
  if (!rok) return;

  const int halves = static_cast<int>(p.kpad >> 3);    // halves of a plane
  SplitDst<SIDE> d;
  d.splane = static_cast<int>(p.out_rows);
  d.hplane = static_cast<long long>(p.S) * p.out_rows;
  uint4* outz = reinterpret_cast<uint4*>(p.out) + static_cast<long long>(z) * halves * d.hplane;
  for (int kb = kb0 + warp; kb < kb1; kb += nw) {
    if (!resident) load_block(p, P, ld, r, 8 * kb, K, v);
    if (p.conj) {
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q].y ^= static_cast<long long>(0x8000000000000000ull);
    }
    if (bad) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (abs_bits(v[q].x) >= 0x7FF0000000000000ull) v[q].x = 0;
        if (abs_bits(v[q].y) >= 0x7FF0000000000000ull) v[q].y = 0;
      }
    }
    // rows of subnormal numbers: their significands are shorter than their exponent says, so they are
    // scaled (exactly) into the normal range, and the exponent with them
    int ei = e;
    if (SF > 0 && e < -1000) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        v[q].x = __double_as_longlong(__longlong_as_double(v[q].x) * 0x1.0p100);
        v[q].y = __double_as_longlong(__longlong_as_double(v[q].y) * 0x1.0p100);
      }
      ei += 100;
    }
    d.out = outz + 2LL * kb * d.hplane + (SIDE == 0 ? r : 2 * r);
    d.tail4 = K - 8 * kb <= 4;
    d.has2 = 2 * kb + 1 < halves;
    if constexpr (SF > 0) emit_fixed<SF, SIDE>(d, v, ei);
    else emit_generic<W64, SIDE>(p, d, v, e, r, 8 * kb, K, z == 0 ? p.dbg_digits : nullptr);
  }
}

template <int SF, bool W64, bool GIVEN>
__global__ void __launch_bounds__(SPLIT_MAX_WARPS * 32, 2) split_kernel(const __grid_constant__ SplitPair pp) {
  __shared__ unsigned long long wmax[SPLIT_MAX_WARPS][SPLIT_ROWS];     // row maxima of the warps
  __shared__ unsigned long long cmax[SPLIT_MAX_KG][SPLIT_ROWS];        // and of the cluster's CTAs
  grid_dependency_wait();
  launch_dependents();
  if (pp.s[blockIdx.z].side == 0) split_rows<SF, W64, 0, GIVEN>(pp.s[blockIdx.z], wmax, cmax);
  else split_rows<SF, W64, 1, GIVEN>(pp.s[blockIdx.z], wmax, cmax);
}

// Row maxima ahead of the split: the same CTAs (kgroups per row block), each over its share of the
// K-blocks; one 64-bit atomicMax per row and CTA into gmax, which the launcher clears.
__global__ void __launch_bounds__(SPLIT_MAX_WARPS * 32, 2) split_rowmax_kernel(const __grid_constant__ SplitPair pp) {
  __shared__ unsigned long long wmax[SPLIT_MAX_WARPS][SPLIT_ROWS];
  grid_dependency_wait();
  launch_dependents();
  const SplitParams& p = pp.s[blockIdx.z];
  const int z = blockIdx.y;
  const bool single = p.X == nullptr;
  const int R = single ? p.rows1 : p.rows[z];
  const int K = single ? p.k1 : p.kdim[z];
  const int rank = static_cast<int>(blockIdx.x) % p.kgroups;
  const int r0 = (static_cast<int>(blockIdx.x) / p.kgroups) * SPLIT_ROWS;
  if (r0 >= R) return;
  const longlong2* __restrict__ P = reinterpret_cast<const longlong2*>(single ? p.X1 + z * p.zstride1 : p.X[z]);
  const long long ld = single ? p.ld1 : p.ld[z];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int r = r0 + lane;
  const int nkb = (K + 7) >> 3, share = (nkb + p.kgroups - 1) / p.kgroups;
  const int kb0 = rank * share, kb1 = min(nkb, kb0 + share);
  unsigned long long mx = 0ull;
  if (r < R)
    for (int kb = kb0 + warp; kb < kb1; kb += nw) {
      longlong2 v[8];
      load_block(p, P, ld, r, 8 * kb, K, v);
      mx = max(mx, block_max(v));
    }
  wmax[warp][lane] = mx;
  __syncthreads();
  if (warp != 0 || r >= R) return;
  for (int w = 1; w < nw; ++w) mx = max(mx, wmax[w][lane]);
  if (mx) atomicMax(&p.gmax[z * p.exp_stride + r], mx);
}

// compile-time slice counts 3..10 (nbits = 8 S - 1 on every side); the test hook's digit copy and
// other slice counts take the run-time form
template <bool GIVEN>
static void launch_instances(const cudaLaunchConfig_t& cfg, const SplitPair& pp) {
  int sf = pp.s[0].S;
  for (int sd = 0; sd < pp.nsides; ++sd)
    if (pp.s[sd].S != sf || pp.s[sd].nbits != 8 * sf - 1 || pp.s[sd].dbg_digits) sf = 0;
  switch (sf) {
    case 3: cudaLaunchKernelEx(&cfg, split_kernel<3, true, GIVEN>, pp); break;
    case 4: cudaLaunchKernelEx(&cfg, split_kernel<4, true, GIVEN>, pp); break;
    case 5: cudaLaunchKernelEx(&cfg, split_kernel<5, true, GIVEN>, pp); break;
    case 6: cudaLaunchKernelEx(&cfg, split_kernel<6, true, GIVEN>, pp); break;
    case 7: cudaLaunchKernelEx(&cfg, split_kernel<7, true, GIVEN>, pp); break;
    case 8: cudaLaunchKernelEx(&cfg, split_kernel<8, true, GIVEN>, pp); break;
    case 9: cudaLaunchKernelEx(&cfg, split_kernel<9, false, GIVEN>, pp); break;
    case 10: cudaLaunchKernelEx(&cfg, split_kernel<10, false, GIVEN>, pp); break;
    default:
      if (pp.s[0].nbits <= 62 && (pp.nsides < 2 || pp.s[1].nbits <= 62))
        cudaLaunchKernelEx(&cfg, split_kernel<0, true, GIVEN>, pp);
      else
        cudaLaunchKernelEx(&cfg, split_kernel<0, false, GIVEN>, pp);
  }
}

void launch_split(const SplitParams& a, int rows_a, const SplitParams* b, int rows_b, int kmax, int batch,
                  cudaStream_t st) {
  SplitPair pp;
  pp.s[0] = a;
  pp.nsides = b ? 2 : 1;
  if (b) pp.s[1] = *b;
  const int rows = std::max(rows_a, b ? rows_b : 0);
  const int rblocks = (rows + SPLIT_ROWS - 1) / SPLIT_ROWS;
  const int nkb = (kmax + 7) / 8;
  // a cluster of up to 8 CTAs shares a row block's K-blocks when its rows are longer than the 8
  // K-blocks that a CTA reads once (K > 64), or while the launch has fewer than two CTAs per SM
  // and a CTA would keep at least 8 K-blocks
  const long long ctas = static_cast<long long>(rblocks) * batch * pp.nsides;
  int kg = 1;
  while (kg < SPLIT_MAX_KG && ((nkb + kg - 1) / kg > SPLIT_MAX_WARPS ||
                               (ctas * kg < 2LL * gpu_sm_count() && nkb / (2 * kg) >= 8)))
    kg *= 2;
  // Clusters of 8 over few row blocks leave most of a GPU idle that holds 2 CTAs an SM, and read a long
  // share twice.  Where at least 16 CTAs a row block find room, the row maxima of 384 K-blocks (K = 3072)
  // or more are taken by a launch of their own, and every row block's K-blocks are dealt to all those CTAs,
  // at least 8 to each.  Products at S = 7 with clusters and so: 32 x 32 x 2048 51 and 44 us, x 4096 88 and
  // 63, x 32768 578 and 318; 256 x 256 (19 CTAs a row block) x 1024 39 and 44, x 4096 105 and 94; at S = 5
  // 16 x 16 x 2048 103 and 105, x 3072 148 and 145; 500 x 500 (9 CTAs a row block) x 4096 225 and 241.
  const long long fill = std::min<long long>(2LL * gpu_sm_count() / std::max(1LL, ctas), nkb / SPLIT_MAX_WARPS);
  const bool given = a.gmax && (!b || b->gmax) && fill >= SPLIT_GMAX_KG && nkb >= SPLIT_GMAX_KB;
  if (given) kg = static_cast<int>(fill);
  const int share = (nkb + kg - 1) / kg;
  for (int sd = 0; sd < pp.nsides; ++sd) {
    pp.s[sd].kgroups = kg;
    if (!given) pp.s[sd].gmax = nullptr;
    else cudaMemsetAsync(pp.s[sd].gmax, 0, sizeof(unsigned long long) * pp.s[sd].exp_stride * batch, st);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(rblocks * kg), static_cast<unsigned>(batch), static_cast<unsigned>(pp.nsides));
  cfg.blockDim = dim3(32u * static_cast<unsigned>(given ? SPLIT_MAX_WARPS : std::max(std::min(share, SPLIT_MAX_WARPS), kg)));
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = static_cast<unsigned>(kg);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1] = pdl_attribute(st);
  const bool cluster = kg > 1 && !given;
  cfg.attrs = cluster ? at : at + 1;
  cfg.numAttrs = cluster ? 2 : 1;
  if (given) {
    cudaLaunchKernelEx(&cfg, split_rowmax_kernel, pp);
    record_launch();
  }
  if (given) launch_instances<true>(cfg, pp);
  else launch_instances<false>(cfg, pp);
  record_launch();
}

}  // namespace ozk
