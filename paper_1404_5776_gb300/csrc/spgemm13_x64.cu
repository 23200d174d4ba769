// FP64 block products on the tensor cores: 13-function atoms, and 4-function atoms
// in quads.
//
// Same contraction as spgemm.cu (C_ij = sum_k op(A)_ik op(B)_kj over the triple
// list of the output block).  GB300 does two FP64 fused multiply-adds per clock
// and SM, and the CUDA-core kernel ran at 87 % of that (a real triple: 1,099
// clocks); the tensor cores do about a thousand FP16 ones through mma.sync.  So
// every operand is written in 72-bit fixed point and multiplied digit by digit,
// exactly (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012):
//   * each row of op(A) (each column of op(B)) takes one power-of-two scale,
//     the first power 2^e above its magnitudes over the whole block row
//     (column); each block takes off it the whole digits that its own largest
//     value leaves at zero (z of them): x = X 2^(e - 9 z - 70), X an integer
//     rounded to nearest, |X| < 2^70;
//   * X in radix 512 with digits -256..255: the 9-bit groups of X + 256 (1 + 512 +
//     ... + 512^7) are the digits plus 256, so the split is one addition;
//   * a pair of digits (p, q) has the weight p + q + z_A + z_B; weights count from
//     the first one that any triple of the item reaches, and the pairs of weights
//     0..8 from there on are multiplied as FP16 integers (one m16n8k16 per pair and
//     8-column half: 43 pairs for a triple that starts at the first, 28 two
//     weights further, 15 four), each weight in its own FP32 accumulators.  These
//     stay integers below 2^24 for CARRY products, and so exact; then multiples of
//     512 move up one weight, exactly as well;
//   * at the end the weights meet as two 64-bit integers, and these in FP64 with
//     one rounding.
// An entry keeps its 53 bits down to 2^-17 of the largest of its row (column) in a
// near block, and is rounded to 2^-71 of the block's share of the scale below that;
// what the pairs left out add is smaller still.  So the error of an element is
// bounded by the scales of its row and column, not by its own terms as that of
// multiply-adds is (n 2^-53 of |A||B|); on the library's matrices it is the smaller
// of the two element by element, as the blocks' entries spread over far less than
// the 2^18 between 2^-53 and 2^-71.  Measured over 64-bit-mantissa sums (64 and 216
// atoms x 13, 512 x 4, r = 6..10 A), S^-1 H and U K U^dagger: relative 2-norm error 4e-17 to
// 8e-17 (multiply-adds 4e-16 to 3e-15), the largest error of a single element over |A||B|
// 6e-17 to 6e-16 (9e-16 to 8e-15).  (64 bits in radix 256, with the weights of an item
// counted from its row's scale, are 10 % faster and leave up to 4e-13 there.)
//
// Layout: a split block is stored in the order in which an m16n8k16 operand
// lies in a warp's registers (lane = 4 (row mod 8) + (k mod 8)/2), 16 bytes a
// lane and load: one digit of op(A), two digits of one 8-column half of op(B).
// Operands go from L2 straight into registers, without shared memory.  Rows and
// k of 13..15 are padding.
//
// One warp owns an 8-column half of a real output (a complex item: four warps,
// halves x real and imaginary part, reading the same blocks through L1): 36
// accumulators, 32 registers of A's digits and 16 of B's fit 128 registers, so
// 16 warps a SM; a warp with both halves (168 registers, 12 warps) measured 1.3
// times slower.  What bounds it: the tensor pipe, with the wait for the next blocks'
// first digits and the carries beside it.  216 atoms x 13, r = 8 A: a Taylor power
// 1.15 ms with its splits 1.20, M = U K 3.9 ms, 2.8 for a real K (the CUDA-core kernel: 8.9 and 21.7 ms);
// FP64 EM step at 512 atoms 22 ms (126).  The time follows the warps in flight: A's
// digits in two sets of registers (12 warps) took 27 % longer, five CTAs of 96
// registers (spills) 65 %.
//
// 4-function atoms take the same kernel in quads: the blocks between two groups of
// four consecutive atoms as one 16 x 16 block, absent ones zero (a 4 x 4 triple
// alone would fill an eighth of a product).  FP64 EM step of 1728 atoms x 4 at 8 A:
// 7.7 ms (one lane group a block on the CUDA cores: 12.4); of 64 atoms x 4: 0.16 ms (0.41).
#include <algorithm>

#include "rt_internal.cuh"

namespace rt {

namespace x64 {

// A block of the product: a 13-function block as stored, or a quad: the 4-function
// blocks between two groups of four consecutive atoms as one 16 x 16 block (absent
// ones are zero).
template <bool QUAD>
struct Shape {
  static constexpr int BS = QUAD ? 16 : 13;
  static constexpr int NE = BS * BS;
};
constexpr int BLK = 4096;      // bytes of one split real block: 8 digits x 32 lanes x 8 elements in FP16
constexpr int WARPS = 4;
constexpr int MINB = 4;
// warps of a CTA: an item takes 2 (real) or 4 (complex) for each share of its triples
template <bool CPLX, int KS>
constexpr int CTA_WARPS = (CPLX ? 4 : 2) * KS > WARPS ? (CPLX ? 4 : 2) * KS : WARPS;
constexpr int NW = 9;          // weights of the digit pairs that are multiplied
// real products between two carries: a weight has at most seven pairs of digits, of which the
// first is at most 128, so that a product adds at most 16 * 7 * 2^16 to weights 4..8 and, with
// up to four pairs, 16 * 3 * 2^16 to weights 0..3; with what the carries leave and bring in,
// CARRY and 2 CARRY of them stay below 2^24
constexpr int CARRY = 2;
constexpr int HIGH = 4;        // weights below this one carry at every second turn
constexpr int DIGIT = 9;       // bits of a digit
constexpr int EXP_NAN = 2047;  // scale of a row that holds a NaN or an infinity: its products are NaN
constexpr int MAX_LEAD = 120;  // leading zero digits that a block's shift takes off at most
constexpr int ZERO_LEAD = 255; // a block of zeros (above 2 MAX_LEAD + NW: no product of it has a weight)
constexpr int SPLIT_WARPS = 16;

// ---------------------------------------------------------------------------
// split: one CTA per atom; its block row (by_col: its block column, reached
// through the transposes) is read for the scales, then again (from L2) for the
// digits.  Bound by the integer pipe that builds the digits: 52 us for the 31 MB
// of a real matrix at 216 atoms, 5 % of the product that it serves.
// ---------------------------------------------------------------------------
// x in 72-bit fixed point, 256 added to each digit: hi and lo hold four digits each.
__device__ __forceinline__ void fixed_biased(double x, int ex_row, unsigned long long& hi, unsigned long long& lo) {
  constexpr long long BIAS = 256ll * (1 + (1ll << 9) + (1ll << 18) + (1ll << 27)), MASK = (1ll << 36) - 1;
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = b & 0xfffffffffffffull;
  if (ex) m |= 1ull << 52;
  // |x| < 2^(ex_row - 1022); X = x 2^(70 - (ex_row - 1022)) = m 2^(max(ex,1) - ex_row + 17)
  int s = max(ex, 1) - ex_row + 17;
  if (s < 0) {
    m = s > -64 ? (m + (1ull << (-s - 1))) >> -s : 0ull;
    s = 0;
  }
  long long h = (long long)(m >> (36 - s)), l = (long long)((m << s) & MASK);
  if (b >> 63) {
    h = -h;
    l = -l;
  }
  l += BIAS;
  hi = (unsigned long long)(h + BIAS + (l >> 36));
  lo = (unsigned long long)(l & MASK);
}

// Two biased digits (18 bits) as the FP16 numbers 1024 + u in the lower and upper half.
__device__ __forceinline__ unsigned two_digits(unsigned w) {
  return (w & 0x1ffu) | ((w << 7) & 0x1ff0000u) | 0x64006400u;
}
__device__ __forceinline__ unsigned less_1280(unsigned h) {
  unsigned r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0x65006500u));
  return r;
}

// Element (x, y) of block q: in the stored blocks, or (quads) in the 4-function
// block that the map names for its two atoms (-1: none, zero).
template <bool QUAD>
__device__ __forceinline__ int64_t element(const int32_t* __restrict__ map, int64_t q, int x, int y) {
  if constexpr (QUAD) {
    const int blk = map[q * 16 + (x >> 2) * 4 + (y >> 2)];
    return blk < 0 ? -1 : (int64_t)blk * 16 + (x & 3) * 4 + (y & 3);
  } else {
    return q * 169 + x * 13 + y;
  }
}

struct SplitArgs {  // one operand; a launch takes one or two (blockIdx.y)
  const double* vals;
  const int32_t* map;
  const int32_t* rowptr;
  const int32_t* tmap;
  int by_col, right;
  unsigned char* dig;
  unsigned char* lead;
  int32_t* exps;
};
struct SplitPair {
  SplitArgs s[2];
};

template <bool CPLX, bool QUAD>
__global__ void __launch_bounds__(SPLIT_WARPS * 32, 2) k_split13(const __grid_constant__ SplitPair pair) {
  const SplitArgs& s = pair.s[blockIdx.y];
  const double* __restrict__ vals = s.vals;
  const int32_t* __restrict__ map = s.map;
  const int32_t* __restrict__ rowptr = s.rowptr;
  const int32_t* __restrict__ tmap = s.tmap;
  const int by_col = s.by_col, right = s.right;
  unsigned char* __restrict__ dig = s.dig;
  unsigned char* __restrict__ lead = s.lead;
  int32_t* __restrict__ exps = s.exps;
  constexpr int NC = CPLX ? 2 : 1;
  constexpr int BS = Shape<QUAD>::BS, NE = Shape<QUAD>::NE;
  __shared__ int smax[16];
  const int atom = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q0 = rowptr[atom], q1 = rowptr[atom + 1];
  if (threadIdx.x < 16) smax[threadIdx.x] = 1;
  __syncthreads();
  constexpr int EPT = (NE + 31) / 32;  // 13: elements e = lane + 32 k keep their row and column from block to block
  int mx[EPT];
#pragma unroll
  for (int k = 0; k < EPT; ++k) mx[k] = 1;
  for (int q = q0 + warp; q < q1; q += SPLIT_WARPS) {
    const int qb = by_col ? tmap[q] : q;
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
      const int e = lane + 32 * k;
      const int64_t at = e < NE ? element<QUAD>(map, qb, e / BS, e % BS) : -1;
      if (at >= 0) {
        int m;
        if constexpr (CPLX) {
          const double2 z = reinterpret_cast<const double2*>(vals)[at];
          m = max(__double2hiint(z.x) & 0x7fffffff, __double2hiint(z.y) & 0x7fffffff);
        } else {
          m = __double2hiint(vals[at]) & 0x7fffffff;
        }
        mx[k] = max(mx[k], m >> 20);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < EPT; ++k) {
    const int e = lane + 32 * k;
    if (e < NE) atomicMax(&smax[by_col ? e % BS : e / BS], mx[k]);
  }
  __syncthreads();
  if (threadIdx.x < 16) exps[atom * 16 + threadIdx.x] = smax[threadIdx.x];

  const int g = lane >> 2, t = lane & 3;
  for (int q = q0 + warp; q < q1; q += SPLIT_WARPS) {
    const int qb = by_col ? tmap[q] : q;
    double val[NC][8];
#pragma unroll
    for (int f = 0; f < 8; ++f) {
      const int m = g + ((f >> 1) & 1) * 8;               // scaled index
      const int k = 2 * t + (f & 1) + (f >> 2) * 8;       // summed index
      const bool in = m < BS && k < BS && smax[m] != EXP_NAN;
      const int64_t at = in ? element<QUAD>(map, qb, by_col ? k : m, by_col ? m : k) : -1;
      if constexpr (CPLX) {
        const double2 z = at >= 0 ? reinterpret_cast<const double2*>(vals)[at] : make_double2(0.0, 0.0);
        val[0][f] = z.x;
        val[1][f] = z.y;
      } else {
        val[0][f] = at >= 0 ? vals[at] : 0.0;
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      // the block's own shift: whole digits that its largest value leaves at zero, from the
      // exponents alone (|x| < 2^(ex - 1022) and 2^70 is the row's bound)
      int gap = DIGIT * ZERO_LEAD;
#pragma unroll
      for (int f = 0; f < 8; ++f) {
        const int ex = (__double2hiint(val[c][f]) >> 20) & 0x7ff;
        if (val[c][f] != 0.0) gap = min(gap, smax[g + ((f >> 1) & 1) * 8] - max(ex, 1));
      }
      gap = __reduce_min_sync(0xffffffffu, gap);
      const int z = gap == DIGIT * ZERO_LEAD ? ZERO_LEAD : min(gap / DIGIT, MAX_LEAD);
      if (lane == 0) lead[(int64_t)qb * NC + c] = (unsigned char)z;
      unsigned long long X[8][2];  // digits 0..3 and 4..7
#pragma unroll
      for (int f = 0; f < 8; ++f)
        fixed_biased(val[c][f], smax[g + ((f >> 1) & 1) * 8] - DIGIT * z, X[f][0], X[f][1]);
      uint4* out = reinterpret_cast<uint4*>(dig + ((int64_t)qb * NC + c) * BLK) + lane;
#pragma unroll
      for (int p2 = 0; p2 < 4; ++p2) {  // digits 2 p2 and 2 p2 + 1, most significant first
        unsigned w[2][4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const unsigned a = (unsigned)(X[2 * r][p2 >> 1] >> (p2 & 1 ? 0 : 18)) & 0x3ffffu;
          const unsigned b = (unsigned)(X[2 * r + 1][p2 >> 1] >> (p2 & 1 ? 0 : 18)) & 0x3ffffu;
          const unsigned ta = two_digits(a), tb = two_digits(b);
          w[0][r] = less_1280(__byte_perm(ta, tb, 0x7632));
          w[1][r] = less_1280(__byte_perm(ta, tb, 0x5410));
        }
        if (right) {
          // op(B): the 8-column halves apart, two digits of one half together
          out[32 * p2] = make_uint4(w[0][0], w[0][2], w[1][0], w[1][2]);
          out[32 * (4 + p2)] = make_uint4(w[0][1], w[0][3], w[1][1], w[1][3]);
        } else {
          out[32 * (2 * p2)] = make_uint4(w[0][0], w[0][1], w[0][2], w[0][3]);
          out[32 * (2 * p2 + 1)] = make_uint4(w[1][0], w[1][1], w[1][2], w[1][3]);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// product
// ---------------------------------------------------------------------------
struct Args {
  GemmArgs g;
  const unsigned char* dA;
  const unsigned char* dB;
  const unsigned char* lA;
  const unsigned char* lB;
  const int32_t* eA;
  const int32_t* eB;
  const int32_t* cmap;  // quads: the output's 4-function blocks
};

__device__ __forceinline__ void mma16816(float (&c)[4], const uint4& a, unsigned b0, unsigned b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
// v 2^(ea - 1022) 2^(eb - 1022) 2^-shift, a normal result by its exponent field
// alone; a row with a NaN or an infinity gives NaN
__device__ __forceinline__ double pow2_scaled(double v, int ea, int eb, int shift) {
  if (ea == EXP_NAN || eb == EXP_NAN) return __longlong_as_double(0x7ff8000000000000ll);
  const int k = ea + eb - 2044 - shift, h = __double2hiint(v), ex = ((h >> 20) & 0x7ff) + k;
  if (v == 0.0) return 0.0;
  return ex > 0 && ex < 2047 ? __hiloint2double(h + k * (1 << 20), __double2loint(v)) : ldexp(v, k);
}
// pairs of FP32 numbers in one register pair
__device__ __forceinline__ unsigned long long pair_of(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpair(unsigned long long v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// an FP32 integer below 2^22 in magnitude
__device__ __forceinline__ int small_int(float v) { return __float_as_int(v + 12582912.f) - 0x4b400000; }

// The digit pairs of one real product whose blocks leave the first Z weights
// at zero.  A digit's registers take the next product's digit (na, nb; weights
// from znext on) right after their last use here, so that the loads are in
// flight under the multiplications that follow.
// ALL: every digit is loaded, also those below the last weight (a real product's
// warp is bound by its instructions: 3 % faster; a complex one's by its loads:
// 7 % slower).
template <int Z, bool ALL>
__device__ __forceinline__ void multiply(float (&acc)[NW][4], uint4 (&a)[8], uint4 (&b)[4],
                                         const uint4* __restrict__ na, const uint4* __restrict__ nb, int znext) {
  constexpr int LAST = NW - 1 - Z;  // p + q <= LAST
#pragma unroll
  for (int p = 7; p >= 0; --p)
    if (p > LAST && (ALL || p + znext < NW)) a[p] = na[32 * p];
#pragma unroll
  for (int q2 = 3; q2 >= 0; --q2)
    if (2 * q2 > LAST && (ALL || 2 * q2 + znext < NW)) b[q2] = nb[32 * q2];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    if (q <= LAST) {
      const unsigned b0 = (q & 1) ? b[q >> 1].z : b[q >> 1].x, b1 = (q & 1) ? b[q >> 1].w : b[q >> 1].y;
#pragma unroll
      for (int p = 7; p >= 0; --p)  // the digits of A that the last product left first come first
        if (p + q <= LAST) mma16816(acc[p + q + Z], a[p], b0, b1);
      if (((q & 1) || q == LAST) && (ALL || (q & ~1) + znext < NW)) b[q >> 1] = nb[32 * (q >> 1)];
#pragma unroll
      for (int p = 7; p >= 0; --p)
        if (p <= LAST && (LAST - p < 7 ? LAST - p : 7) == q && (ALL || p + znext < NW)) a[p] = na[32 * p];
    }
  }
}

template <bool CPLX, bool ADAG, bool BDAG, int EPI, bool QUAD, int KS>
__global__ void __launch_bounds__(CTA_WARPS<CPLX, KS> * 32, MINB * WARPS / CTA_WARPS<CPLX, KS>) k_gemm13_x64(const __grid_constant__ Args x) {
  constexpr int NP = CPLX ? 2 : 1;  // real products per triple and warp; parts of a complex output
  constexpr int WPB = 2 * NP;       // warps of one share of an item: 8-column halves x parts
  constexpr int WPI = WPB * KS;     // warps per item
  constexpr int NWARP = CTA_WARPS<CPLX, KS>;
  constexpr int BS = Shape<QUAD>::BS, NE = Shape<QUAD>::NE;
  const GemmArgs& g = x.g;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int half = warp & 1;                      // output columns 8 half .. 8 half + 7
  const int part = CPLX ? ((warp >> 1) & 1) : 0;  // 0: real part, 1: imaginary part
  const int slot = warp / WPI, ks = KS > 1 ? (warp % WPI) / WPB : 0;
  const int64_t item = (int64_t)blockIdx.x * (NWARP / WPI) + slot;
  if (item >= g.n_items) return;  // the warps of one item leave together

  __shared__ double sC[NWARP / WPI][NE * NP];
  __shared__ long long shares[KS > 1 ? (KS - 1) * WPB : 1][KS > 1 ? 8 : 1][32];  // integer sums of the shares after the first (one item a CTA)

  // signs of the two real products of this part (op(A) = Ar + i sa Ai, op(B) = Br + i sb Bi):
  //   real part:       Ar Br - sa sb Ai Bi;   imaginary part: sb Ar Bi + sa Ai Br
  const bool neg0 = CPLX && part && BDAG;
  const bool neg1 = CPLX && (part ? ADAG : (ADAG == BDAG));

  float acc[NW][4], top[4];  // sums of each weight; the carry out of the first
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    top[r] = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) acc[w][r] = 0.f;
  }
  // moves multiples of 512 up one weight, from the last weight to `first` (FP32 integers below
  // 2^24: every operation is exact; two at a time, a third of the warp's issue slots otherwise)
  auto carry = [&](int first, int last) {
    constexpr float MAGIC = 12582912.f;  // 1.5 * 2^23: adding it rounds to an integer
    const unsigned long long part512 = pair_of(1.f / 512.f, 1.f / 512.f), minus512 = pair_of(-512.f, -512.f);
    const unsigned long long plus = pair_of(MAGIC, MAGIC), minus = pair_of(-MAGIC, -MAGIC);
#pragma unroll
    for (int w = NW - 1; w >= 0; --w)
      if (w >= first && w <= last) {
        float(&up)[4] = w > 0 ? acc[w > 0 ? w - 1 : 0] : top;
#pragma unroll
        for (int r = 0; r < 4; r += 2) {
          const unsigned long long v = pair_of(acc[w][r], acc[w][r + 1]);
          const unsigned long long c = add2(fma2(v, part512, plus), minus);
          unpair(fma2(c, minus512, v), acc[w][r], acc[w][r + 1]);
          unpair(add2(pair_of(up[r], up[r + 1]), c), up[r], up[r + 1]);
        }
      }
  };

  const int64_t t0 = g.ptr[item];
  int nt = (int)(g.ptr[item + 1] - t0);
  const int2* __restrict__ ab = g.ab + t0;
  const unsigned char* __restrict__ dA = x.dA + lane * 16;
  const unsigned char* __restrict__ dB = x.dB + lane * 16 + half * (BLK / 2);
  // leading zero digits of a triple's blocks: bytes 0, 1: A's parts, bytes 2, 3: B's
  auto leads = [&](int2 p) {
    if constexpr (CPLX)
      return (unsigned)reinterpret_cast<const unsigned short*>(x.lA)[p.x] |
             (unsigned)reinterpret_cast<const unsigned short*>(x.lB)[p.y] << 16;
    else
      return (unsigned)x.lA[p.x] | (unsigned)x.lB[p.y] << 16;
  };
  auto lead_a = [&](unsigned z, int sub) { return (int)((z >> (8 * sub)) & 0xff); };
  auto lead_b = [&](unsigned z, int sub) { return (int)((z >> (16 + 8 * (CPLX ? (sub ^ part) : 0))) & 0xff); };
  // weights count from the first that any triple of the item (of all its shares) reaches:
  // a far block keeps as many digits of its own as a near one
  int z0 = ZERO_LEAD;
  for (int t = lane; t < nt; t += 32) {
    const unsigned z = leads(ab[t]);
#pragma unroll
    for (int sub = 0; sub < NP; ++sub) z0 = min(z0, lead_a(z, sub) + lead_b(z, sub));
  }
  z0 = __reduce_min_sync(0xffffffffu, z0);
  if constexpr (KS > 1) {  // this warp's share of the triples
    const int share = (nt + KS - 1) / KS, first = min(nt, share * ks);
    ab += first;
    nt = min(share, nt - first);
  }
  if (nt > 0) {
    // triples t, t + 1 and t + 2 of the list; the digits to skip of the first two
    int2 cur = ab[0], nxt = 1 < nt ? ab[1] : cur, nxt2 = 2 < nt ? ab[2] : nxt;
    unsigned zc = leads(cur), zn = leads(nxt);
    uint4 a[8], b[4];
    {
      const uint4* pa = reinterpret_cast<const uint4*>(dA + (int64_t)cur.x * (BLK * NP));
      const uint4* pb = reinterpret_cast<const uint4*>(dB + ((int64_t)cur.y * NP + part) * BLK);
#pragma unroll
      for (int p = 0; p < 8; ++p) a[p] = pa[32 * p];
#pragma unroll
      for (int p = 0; p < 4; ++p) b[p] = pb[32 * p];
    }
    int since = 0;
    for (int t = 0; t < nt; ++t) {
      const int2 nxt3 = t + 3 < nt ? ab[t + 3] : nxt2;
      const unsigned zn2 = leads(nxt2);
#pragma unroll
      for (int sub = 0; sub < NP; ++sub) {
        // the blocks of the next real product (after the last one: this triple's again, unused)
        const bool last = sub + 1 == NP;
        const int2 nb = last ? nxt : cur;
        const unsigned z = last ? zn : zc;
        const int ns = CPLX ? (sub ^ 1) : 0;  // its part of A; of B: ns ^ part
        const uint4* na = reinterpret_cast<const uint4*>(dA + ((int64_t)nb.x * NP + ns) * BLK);
        const uint4* nbp = reinterpret_cast<const uint4*>(dB + ((int64_t)nb.y * NP + (CPLX ? (ns ^ part) : 0)) * BLK);
        // weights below the first that can be non-zero, of this product and the next
        const int zz = lead_a(zc, sub) + lead_b(zc, sub) - z0, znext = lead_a(z, ns) + lead_b(z, ns) - z0;
        if (CPLX && (sub ? neg1 : neg0)) {
#pragma unroll
          for (int p = 0; p < 8; ++p) {
            a[p].x ^= 0x80008000u;
            a[p].y ^= 0x80008000u;
            a[p].z ^= 0x80008000u;
            a[p].w ^= 0x80008000u;
          }
        }
        // the digits of A that this product needs longest are loaded last and needed first: into L1
#pragma unroll
        for (int p = 0; p < 4; ++p)
          if (p + znext < NW) asm volatile("prefetch.global.L1 [%0];" ::"l"(na + 32 * p));
        switch (zz) {
          case 0: multiply<0, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 1: multiply<1, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 2: multiply<2, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 3: multiply<3, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 4: multiply<4, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 5: multiply<5, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 6: multiply<6, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 7: multiply<7, !CPLX>(acc, a, b, na, nbp, znext); break;
          case 8: multiply<8, !CPLX>(acc, a, b, na, nbp, znext); break;
          default: multiply<NW, !CPLX>(acc, a, b, na, nbp, znext); break;  // below every weight: nothing but the loads
        }
        ++since;
        if (since % CARRY == 0) carry(HIGH, NW - 1);
        if (since == 2 * CARRY) {
          carry(0, HIGH - 1);
          since = 0;
        }
      }
      cur = nxt;
      nxt = nxt2;
      nxt2 = nxt3;
      zc = zn;
      zn = zn2;
    }
    carry(0, NW - 1);
  }

  const int q = g.item_blk[item];
  const int i = g.rowidx[q], j = g.colidx[q];
  // the weights as two integers, hi 2^54 + lo in units of 512^6 2^-140
  long long hi[4], lo[4];
#pragma unroll
  for (int rr = 0; rr < 4; ++rr) {
    const int lo1 = (small_int(acc[3][rr]) * 512 + small_int(acc[4][rr])) * 512 + small_int(acc[5][rr]);
    const int lo0 = (small_int(acc[6][rr]) * 512 + small_int(acc[7][rr])) * 512 + small_int(acc[8][rr]);
    const int hi1 = __float2int_rn(top[rr]);
    const int hi0 = (small_int(acc[0][rr]) * 512 + small_int(acc[1][rr])) * 512 + small_int(acc[2][rr]);
    lo[rr] = (long long)lo1 * (1 << 27) + lo0;
    hi[rr] = (long long)hi1 * (1 << 27) + hi0;
  }
  if constexpr (KS > 1) {
    const int base = warp % WPB;
    if (ks > 0)
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) {
        shares[(ks - 1) * WPB + base][rr][lane] = hi[rr];
        shares[(ks - 1) * WPB + base][4 + rr][lane] = lo[rr];
      }
    asm volatile("bar.sync %0, %1;" ::"r"(slot + 1), "n"(32 * WPI) : "memory");
    if (ks == 0)
#pragma unroll
      for (int k = 1; k < KS; ++k)
#pragma unroll
        for (int rr = 0; rr < 4; ++rr) {
          hi[rr] += shares[(k - 1) * WPB + base][rr][lane];
          lo[rr] += shares[(k - 1) * WPB + base][4 + rr][lane];
        }
  }
  if (ks == 0) {
    const int gr = lane >> 2, tc = lane & 3;
#pragma unroll
    for (int rr = 0; rr < 4; ++rr) {
      const int r = gr + (rr >> 1) * 8, c = 8 * half + 2 * tc + (rr & 1);
      if (r < BS && c < BS) {
        // lo within 2^53, so that it is exact in FP64; the integers enter as mantissas of 1.5 2^20,
        // 1.5 2^-7 and 1.5 2^-34 (exact), and the two halves of lo, then hi and lo meet: one rounding
        const long long up = (lo[rr] + (1ll << 53)) >> 54;
        const long long l = lo[rr] - (up << 54), l0 = ((l + (1ll << 26)) & ((1ll << 27) - 1)) - (1ll << 26);
        constexpr double MH = 0x1.8p20, M1 = 0x1.8p-7, M0 = 0x1.8p-34;
        const double vh = __longlong_as_double(__double_as_longlong(MH) + hi[rr] + up) - MH;
        const double v1 = __longlong_as_double(__double_as_longlong(M1) + ((l - l0) >> 27)) - M1;
        const double v0 = __longlong_as_double(__double_as_longlong(M0) + l0) - M0;
        sC[slot][(r * BS + c) * NP + part] =
            pow2_scaled(vh + (v1 + v0), x.eA[i * 16 + r], x.eB[j * 16 + c], DIGIT * z0);
      }
    }
  }
  asm volatile("bar.sync %0, %1;" ::"r"(slot + 1), "n"(32 * WPI) : "memory");

  using V = typename std::conditional<CPLX, double2, double>::type;
  const V* val = reinterpret_cast<const V*>(sC[slot]);
  const int el = lane + 32 * (warp % WPI);  // this thread's first element
  constexpr int STEP = 32 * WPI;
  V* __restrict__ C = static_cast<V*>(g.C);
  if constexpr (EPI == EPI_STORE || EPI == EPI_ADD || EPI == EPI_STORE_ACC) {
    for (int e = el; e < NE; e += STEP) {
      const int r = e / BS, c = e - r * BS;
      const int64_t at = element<QUAD>(x.cmap, q, r, c);
      if (QUAD && at < 0) continue;
      if constexpr (EPI == EPI_STORE) {
        C[at] = val[e];
      } else if constexpr (EPI == EPI_ADD) {
        if constexpr (CPLX) {
          const double2 o = C[at];
          C[at] = make_double2(o.x + val[e].x, o.y + val[e].y);
        } else {
          C[at] += val[e];
        }
      } else {
        // real power T^n stored (unless C is null); coef * T^n added to complex U (on the same pattern)
        if (C) C[at] = val[e];
        double2* __restrict__ U = static_cast<double2*>(g.U);
        double2 u = U[at];
        if (g.coef_imag) u.y += g.coef * val[e];
        else u.x += g.coef * val[e];
        U[at] = u;
      }
    }
  } else if constexpr (EPI == EPI_TWO_I) {
    double part_sum = 0.0;
    for (int e = el; e < NE; e += STEP) {
      const int r = e / BS, c = e - r * BS;
      const int64_t at = element<QUAD>(x.cmap, q, r, c);
      if (QUAD && at < 0) continue;
      double re, im = 0.0;
      if constexpr (CPLX) {
        re = val[e].x;
        im = val[e].y;
      } else {
        re = val[e];
      }
      const bool on = i == j && r == c;
      const double dre = (on ? 1.0 : 0.0) - re;
      const int bi = QUAD ? g.bsize[4 * i + (r >> 2)] : g.bsize[i], bj = QUAD ? g.bsize[4 * j + (c >> 2)] : g.bsize[j];
      if ((QUAD ? (r & 3) : r) < bi && (QUAD ? (c & 3) : c) < bj) part_sum += dre * dre + im * im;
      if constexpr (CPLX) C[at] = make_double2((on ? 2.0 : 0.0) - re, -im);
      else C[at] = (on ? 2.0 : 0.0) - re;
    }
    for (int off = 16; off > 0; off >>= 1) part_sum += __shfl_down_sync(0xffffffffu, part_sum, off);
    __shared__ double partial[NWARP];
    if (lane == 0) partial[warp] = part_sum;
    asm volatile("bar.sync %0, %1;" ::"r"(slot + 1), "n"(32 * WPI) : "memory");
    if (lane == 0 && warp % WPI == 0) {
      double sum = 0.0;
      for (int w = 0; w < WPI; ++w) sum += partial[warp + w];
      g.red[item] = sum;
    }
  } else if constexpr (EPI == EPI_SANDWICH) {
    // K'_ij for j >= i; mirror K'_ji = K'_ij^dagger; hermitian diagonal blocks (atoms i, j: a
    // quad of two different groups lies above the diagonal as a whole)
    if (i != j) {
      for (int e = el; e < NE; e += STEP) {
        const int r = e / BS, c = e - r * BS;
        const int64_t at = element<QUAD>(x.cmap, q, r, c);
        if (QUAD && at < 0) continue;
        C[at] = val[e];
        if constexpr (QUAD) {
          C[(int64_t)g.tmap[at >> 4] * 16 + (c & 3) * 4 + (r & 3)] = make_double2(val[e].x, -val[e].y);
        } else {
          // the mirror, written in its own order: element (r,c) of block (j,i)
          const double2 m = val[c * BS + r];
          C[(int64_t)g.tmap[q] * NE + e] = make_double2(m.x, -m.y);
        }
      }
    } else {
      double herm = 0.0;
      for (int e = el; e < NE; e += STEP) {
        const int r = e / BS, c = e - r * BS;
        const int64_t at = element<QUAD>(x.cmap, q, r, c);
        if (QUAD && (at < 0 || (r >> 2) > (c >> 2))) continue;
        const double2 v = val[e];
        if (QUAD && (r >> 2) < (c >> 2)) {
          C[at] = v;
          C[(int64_t)g.tmap[at >> 4] * 16 + (c & 3) * 4 + (r & 3)] = make_double2(v.x, -v.y);
          continue;
        }
        const double2 tv = val[c * BS + r];
        const double dr = v.x - tv.x, di = v.y + tv.y;  // K - K^dagger
        herm = fmax(herm, sqrt(dr * dr + di * di));
        C[at] = make_double2(0.5 * (v.x + tv.x), 0.5 * (v.y - tv.y));
      }
      for (int off = 16; off > 0; off >>= 1) herm = fmax(herm, __shfl_xor_sync(0xffffffffu, herm, off));
      if (lane == 0 && g.herm_max) atomicMax(g.herm_max, (unsigned long long)__double_as_longlong(herm));
    }
  }
}

template <bool CPLX, bool ADAG, bool BDAG, int EPI, int KS>
static void launch_ks(const Args& x, cudaStream_t st) {
  constexpr int W = CTA_WARPS<CPLX, KS>;
  const int64_t per = W / ((CPLX ? 4 : 2) * KS);
  const int64_t grid = (x.g.n_items + per - 1) / per;
  RT_REQUIRE(grid < (1ll << 31), RT_EINTERNAL, "grid too large");
  if (x.cmap) k_gemm13_x64<CPLX, ADAG, BDAG, EPI, true, KS><<<(unsigned)grid, W * 32, 0, st>>>(x);
  else k_gemm13_x64<CPLX, ADAG, BDAG, EPI, false, KS><<<(unsigned)grid, W * 32, 0, st>>>(x);
  RT_CUDA_CHECK(cudaGetLastError());
}

// A product whose warps leave most of the chip idle shares each item's triples
// between KS times the warps (the integer sums of the shares add up exactly, so
// the result does not depend on KS): as long as all of them are resident at once,
// 16 warps on each of 152 SMs.
template <bool CPLX, bool ADAG, bool BDAG, int EPI>
static void launch(const Args& x, cudaStream_t st) {
  const int64_t warps = x.g.n_items * (CPLX ? 4 : 2);
  if (4 * warps <= 152 * 16) return launch_ks<CPLX, ADAG, BDAG, EPI, 4>(x, st);
  if (2 * warps <= 152 * 16) return launch_ks<CPLX, ADAG, BDAG, EPI, 2>(x, st);
  launch_ks<CPLX, ADAG, BDAG, EPI, 1>(x, st);
}

}  // namespace x64

size_t x64_block_bytes(bool cplx) { return (size_t)x64::BLK * (cplx ? 2 : 1); }

void launch_split13(const X64Split* ops, int n, bool cplx, cudaStream_t st) {
  using namespace x64;
  SplitPair pair{};
  for (int k = 0; k < n; ++k) {
    const X64Split& o = ops[k];
    pair.s[k] = {static_cast<const double*>(o.vals), o.quad_map,   o.P->rowptr, o.P->tmap, o.by_col, o.right,
                 o.out.dig,                          o.out.lead, o.out.exps};
  }
  const int atoms = ops[0].P->n_atoms;  // both operands: the same system
  if (n == 0 || atoms == 0) return;
  auto go = [&](auto kernel) { kernel<<<dim3(atoms, n), SPLIT_WARPS * 32, 0, st>>>(pair); };
  if (ops[0].quad_map) cplx ? go(k_split13<true, true>) : go(k_split13<false, true>);
  else cplx ? go(k_split13<true, false>) : go(k_split13<false, false>);
  RT_CUDA_CHECK(cudaGetLastError());
}

void launch_gemm13_x64(bool cplx, bool a_dag, bool b_dag, Epilogue epi, const GemmArgs& g, const X64Operand& A,
                       const X64Operand& B, const int32_t* quad_cmap, cudaStream_t st) {
  using namespace x64;
  if (g.n_items == 0) return;
  RT_REQUIRE(epi != EPI_STORE_ACC || (!g.umap && g.U), RT_EINTERNAL, "the Taylor accumulator lies on the output pattern");
  const Args x{g, A.dig, B.dig, A.lead, B.lead, A.exps, B.exps, quad_cmap};
  if (!cplx && !a_dag && !b_dag) {
    if (epi == EPI_STORE) return launch<false, false, false, EPI_STORE>(x, st);
    if (epi == EPI_STORE_ACC) return launch<false, false, false, EPI_STORE_ACC>(x, st);
    if (epi == EPI_TWO_I) return launch<false, false, false, EPI_TWO_I>(x, st);
    if (epi == EPI_ADD) return launch<false, false, false, EPI_ADD>(x, st);
  } else if (cplx && !a_dag && !b_dag) {
    if (epi == EPI_STORE) return launch<true, false, false, EPI_STORE>(x, st);
    if (epi == EPI_TWO_I) return launch<true, false, false, EPI_TWO_I>(x, st);
    if (epi == EPI_ADD) return launch<true, false, false, EPI_ADD>(x, st);
  } else if (cplx && !a_dag && b_dag) {
    if (epi == EPI_STORE) return launch<true, false, true, EPI_STORE>(x, st);
    if (epi == EPI_SANDWICH) return launch<true, false, true, EPI_SANDWICH>(x, st);
  } else if (cplx && a_dag && !b_dag) {
    if (epi == EPI_STORE) return launch<true, true, false, EPI_STORE>(x, st);
  }
  throw Error{RT_EINTERNAL, "unsupported product variant"};
}

}  // namespace rt
