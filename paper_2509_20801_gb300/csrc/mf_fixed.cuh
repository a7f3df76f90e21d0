// complex128 substitution products on the tensor cores.
//
// A preconditioner application reads every factor entry once per right-hand
// side and needs four FP64 multiply-adds for it.  GB300's FP64 pipe does two
// multiply-adds per clock and SM, so the pipe, not the memory, set the pace
// (0.5 entries per clock and SM against the 1.4 that HBM delivers).  Here the
// products run as exact integer arithmetic on the FP16 tensor cores instead,
// by splitting both operands into digits (the scheme of Ozaki, Ogita, Oishi
// and Rump, Numer. Algorithms 59, 2012):
//
//  * After a front is eliminated its factor blocks are rewritten in place as
//    64-bit fixed-point numbers: row r of a chain of FX_COLS columns shares
//    one exponent e, |x| < 2^e, and each real or imaginary part becomes
//    Y = x 2^(63 - e), stored as Y + 2^63.  Sixteen bytes an entry as before,
//    63 bits below the row's largest entry where FP64 has 53 below each.
//    Finv's columns are scaled by a power of two near the operator's diagonal
//    first (and the values they meet by its inverse), so that they and H12's
//    columns, and sources and fields, are of one magnitude within a chain.
//  * The bytes of Y are its digits in radix 256, and a byte b in the low half
//    of a 16-bit word *is* the FP16 subnormal b 2^-24: splitting an entry
//    costs one mask or byte permutation per pair of digits (and one addition
//    that takes the 2^63 back off the leading digit), no conversion.
//  * The vector values of a chain share one exponent likewise and are held as
//    X = x 2^(62 - e) + 0x80..80, whose bytes are balanced digits plus 128,
//    picked out with byte permutations as well.
//  * One mma.m16n8k16 multiplies four digits of 16 rows x 4 columns by the
//    vector's digits arranged so that accumulator column g collects the digit
//    products of order g, i + j = g: the eight accumulator columns are the
//    eight orders 0..7, nothing of the MMA is padding.  (tcgen05 has M = 128
//    and operands in shared memory; a matrix-vector product would stage every
//    entry there only to use it once.  mma.sync takes the entries straight
//    from the registers they were loaded into, and its measured rate, 0.41
//    m16n8k16 per clock and SM, is 3.3 entries per clock and SM.)
//
// Exactness: a digit of Y is in [-128, 255], one of X in [-128, 127]; a chain
// of 32 columns gives an accumulator at most 32 x 2 x 8 products of at most
// 255 x 128, less than 2^24 in all, so every partial sum is an integer FP32
// holds (measured: exact up to 255^2 x 256).  The orders of a chain are
// combined in 64-bit integers and rounded to FP64 once.  Dropped are the
// orders above 7, below 2^-59 of the row's and the vector's scale: the
// chain's result is closer to the exact one than a chain of FP64
// multiply-adds, which rounds each product at 2^-53.  Chains are added in
// FP64 in column order, the association of the complex64 products.
//
// Measured against FP64 multiply-adds, one application: 4096 x 1024 nodes in
// 16 strips 7.89 -> 4.89 ms, 2048 x 512 one strip after another (8 strips)
// 10.6 -> 5.4 ms, 200 x 200 in 2 strips 479 -> 205 us (there the overlapped
// launches of consecutive levels count as much as the products).  What bounds
// it now is the latency of the dependent loads ahead of a warp's products
// (long-scoreboard stalls at 16 warps an SM), not a pipe.
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace stdd {

constexpr int FX_COLS = MF_SUB;          // columns that share a row's exponent: one chain
constexpr int FX_EMPTY = -4000;          // exponent of a row or vector without a nonzero value
constexpr int FX_BAD = 4000;             // and of one with an infinity or NaN
static_assert(FX_COLS == 32, "one lane gathers one column of a chain");

// exponent e of x 2^sh, |x 2^sh| < 2^e: zero and subnormals FX_EMPTY, inf and NaN FX_BAD
__device__ __forceinline__ int fx_exp(double x, int sh) {
  const int ef = (int)((__double_as_longlong(x) >> 52) & 0x7ff);
  return ef == 0 ? FX_EMPTY : ef == 0x7ff ? FX_BAD : ef - 1022 + sh;
}

// |x| 2^(63 - e) for |x| < 2^e, bits below the last one dropped
__device__ __forceinline__ unsigned long long fx_magnitude(double x, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)((u >> 52) & 0x7ff);
  if (ef == 0 || ef == 0x7ff) return 0ull;
  const unsigned long long m = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);   // |x| = m 2^(ef - 1075)
  const int sh = e - (ef - 1022) - 10;                                   // m 2^(10 - (e - (ef - 1022)))
  return sh <= 0 ? m << -sh : (sh < 64 ? m >> sh : 0ull);
}

// a factor entry's stored form, and a vector value's
__device__ __forceinline__ unsigned long long fx_matrix_word(double x, int e) {
  const unsigned long long m = fx_magnitude(x, e);
  return (x < 0.0 ? 0ull - m : m) ^ (1ull << 63);
}
__device__ __forceinline__ unsigned long long fx_vector_word(double x, int e) {
  const unsigned long long m = fx_magnitude(x, e) >> 1;   // balanced digits reach 0x7f7f..7f only
  return (x < 0.0 ? 0ull - m : m) + 0x8080808080808080ull;
}

__device__ __forceinline__ void fx_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                       uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// the two digit pairs of a 32-bit word: bytes 0 and 2, bytes 1 and 3
__device__ __forceinline__ uint32_t fx_even(uint32_t w) { return w & 0x00ff00ffu; }
__device__ __forceinline__ uint32_t fx_odd(uint32_t w) { return __byte_perm(w, 0u, 0x4341); }
// FP16 subnormals -128 2^-24, added where a digit was stored plus 128
__device__ __forceinline__ uint32_t fx_add(uint32_t w, uint32_t v) {
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;\n" : "=r"(r) : "r"(w), "r"(v));
  return r;
}
// bytes 1 and 3 of a high word, the 2^63 taken off byte 3
__device__ __forceinline__ uint32_t fx_odd_top(uint32_t w) { return fx_add(fx_odd(w), 0x80800000u); }

// What a lane needs to pick the digits X[g - m], m = 0..7, of its order g =
// lane / 4 out of a vector word: the byte selector of m = 0, the masks of
// the valid ones (digits of negative index are zero) and their -128s.
// Pair order as in the matrix words: high word bytes 3, 2, 1, 0 = digits 0..3.
struct FxLane {
  uint32_t sel, mask[4], off[4];   // high even, high odd, low even, low odd
  __device__ __forceinline__ explicit FxLane(int lane) {
    const int g = lane >> 2;
    sel = (uint32_t)(7 - g) * 0x101u;   // bytes 1 and 3 of a pick are masked off
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int m = pair(w);
      mask[w] = (m <= g ? 0xffu : 0u) | (m - 2 <= g ? 0xff0000u : 0u);
      off[w] = (m <= g ? 0x8080u : 0u) | (m - 2 <= g ? 0x80800000u : 0u);
    }
  }
  // digit offset of the low half of pair w (the high half is two less)
  __device__ static __forceinline__ constexpr int pair(int w) { return w == 0 ? 3 : w == 1 ? 2 : w == 2 ? 7 : 6; }
  __device__ __forceinline__ uint32_t pick(uint32_t lo, uint32_t hi, int w) const {
    return fx_add(__byte_perm(lo, hi, sel + (uint32_t)(pair(w) | ((pair(w) - 2) << 8))) & mask[w], off[w]);
  }
};

// The exponents of a front's rows: down block (p rows, n columns) first, then
// the up block (b rows, p columns), chain by chain.
__host__ __device__ __forceinline__ int64_t fx_exps_down(int p, int b) {
  return (int64_t)p * ((p + b + FX_COLS - 1) / FX_COLS);
}
__host__ __device__ __forceinline__ int64_t fx_exps(int p, int b) {
  return fx_exps_down(p, b) + (int64_t)b * ((p + FX_COLS - 1) / FX_COLS);
}

// A warp's walk over the columns of MT x 16 rows, 32 columns (a chain) at a
// time: of the fixed-point block M (leading dimension `rows`, row r0 + i of
// column c at M[c rows + r0 + i]) with the rows' exponents E, chain by chain.
// The matrix loads run AHEAD groups of four columns in front of the products,
// across chains and before the chain's vector values have arrived.
template <int MT, int NR> struct FxRows {
  // (two right-hand sides: their accumulators take the registers)
  static constexpr int AHEAD = (MT == 2 ? 2 : 4) / NR;
  const uint4 *row[2 * MT];
  int64_t ld;
  const short *E;
  int rows, cend;        // rows of the block, last column + 1 of the walk
  uint4 m[AHEAD][2 * MT];

  __device__ __forceinline__ void load(int col, int slot, int lane) {
    const int64_t at = (int64_t)min(col + (lane & 3), cend - 1) * ld;   // columns past the end meet zeros
#pragma unroll
    for (int t = 0; t < 2 * MT; ++t) m[slot][t] = row[t][at];
  }
  __device__ __forceinline__ void start(const double2 *M, const short *E_, int r0, int rows_, int c0, int c1,
                                        int lane) {
    rows = rows_;
    ld = rows_;
    E = E_;
    cend = c1;
    if (rows <= 0) return;      // a root's empty border
    // rows past the block repeat its last one: read, never used
#pragma unroll
    for (int t = 0; t < 2 * MT; ++t)
      row[t] = reinterpret_cast<const uint4 *>(M) + min(r0 + 8 * t + (lane >> 2), rows - 1);
#pragma unroll
    for (int a = 0; a < AHEAD; ++a)
      if (c0 + 4 * a < c1) load(c0 + 4 * a, a, lane);
  }
};

// (hi 2^32 + lo) 2^e rounded to FP64 once; |hi|, |lo| < 2^50.  One conversion
// is all that runs on the FP64 pipe.
__device__ __forceinline__ double fx_value(long long hi, long long lo, int e) {
  hi += lo >> 32;
  const unsigned low = (unsigned)lo;
  // up to 62 leading bits of hi 2^32 + low
  const int sh = min(32, max(0, __clzll(hi < 0 ? ~hi : hi) - 2));
  const long long T = (long long)(((unsigned long long)hi << sh) | (((unsigned long long)low << sh) >> 32));
  e += 32 - sh;
  const double d = __ll2double_rn(T);
  const long long b = __double_as_longlong(d);
  const int ef = (int)((b >> 52) & 0x7ff) + e;
  if (T != 0 && ef > 0 && ef < 2047) return __longlong_as_double(b + ((long long)e << 52));
  return T == 0 ? 0.0 : scalbn(d, e);
}

// One chain for NR right-hand sides: columns [c0, c0 + 32) of the walk.
// xs[q]: the warp's shared copy of the chain's vector words, two per column,
// zero past the end; ex[q]: their exponent.  out[q][t]: of row 16 t + lane /
// 4 + 8 (lane / 2 % 2), component lane % 2.
template <int MT, int NR>
__device__ __forceinline__ void fx_chain(FxRows<MT, NR> &f, int r0, int c0, int lane, const FxLane &fl,
                                         const ulonglong2 (*xs)[FX_COLS], const int (&ex)[NR],
                                         double (&out)[NR][MT]) {
  const int g = lane >> 2, c = lane & 3;
  const int dr = 8 * ((lane >> 1) & 1) + g;
  int er[MT];
#pragma unroll
  for (int t = 0; t < MT; ++t)
    er[t] = f.E[(int64_t)(c0 / FX_COLS) * f.rows + min(r0 + 16 * t + dr, f.rows - 1)];
  const int groups = (min(FX_COLS, f.cend - c0) + 3) >> 2;
  float d[NR][MT][2][4];        // [component][accumulator]: integers of 2^-48
#pragma unroll
  for (int q = 0; q < NR; ++q)
#pragma unroll
    for (int t = 0; t < MT; ++t)
#pragma unroll
      for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i) d[q][t][k][i] = 0.f;
#pragma unroll
  for (int k = 0; k < FX_COLS / 4; ++k) {
    if (k >= groups) break;
    uint32_t br[NR][4], bi[NR][4];
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      const uint4 x = *reinterpret_cast<const uint4 *>(&xs[q][4 * k + c]);
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        br[q][w] = fl.pick(x.x, x.y, w);
        bi[q][w] = fl.pick(x.z, x.w, w);
      }
    }
#pragma unroll
    for (int t = 0; t < MT; ++t) {
      const uint4 u = f.m[k % f.AHEAD][2 * t], v = f.m[k % f.AHEAD][2 * t + 1];
#pragma unroll
      for (int w = 0; w < 2; ++w) {   // high words, low words
        const uint32_t ur = w ? u.x : u.y, vr = w ? v.x : v.y, ui = w ? u.z : u.w, vi = w ? v.z : v.w;
        const uint32_t ure = fx_even(ur), vre = fx_even(vr), uie = fx_even(ui), vie = fx_even(vi);
        const uint32_t uro = w ? fx_odd(ur) : fx_odd_top(ur), vro = w ? fx_odd(vr) : fx_odd_top(vr);
        const uint32_t uio = w ? fx_odd(ui) : fx_odd_top(ui), vio = w ? fx_odd(vi) : fx_odd_top(vi);
#pragma unroll
        for (int q = 0; q < NR; ++q) {
          fx_mma(d[q][t][0], ure, vre, uro, vro, br[q][2 * w], br[q][2 * w + 1]);
          fx_mma(d[q][t][1], ure, vre, uro, vro, bi[q][2 * w], bi[q][2 * w + 1]);
          fx_mma(d[q][t][1], uie, vie, uio, vio, br[q][2 * w], br[q][2 * w + 1]);
          fx_mma(d[q][t][0], uie, vie, uio, vio, bi[q][2 * w] ^ 0x80008000u, bi[q][2 * w + 1] ^ 0x80008000u);
        }
      }
    }
    if (c0 + 4 * (k + f.AHEAD) < f.cend) f.load(c0 + 4 * (k + f.AHEAD), k % f.AHEAD, lane);
  }
  // The four lanes of a row hold orders 2 c, 2 c + 1 of (row g, re), (g, im),
  // (g + 8, re), (g + 8, im); each lane ends with the sum of one of the four:
  //   sum_g D_g 256^(7 - g) = A 2^32 + B,  A = V_0 2^16 + V_1,  B = V_2 2^16 + V_3,
  // V_c = D_2c 256 + D_2c+1, |D| < 2^24: A and B are below 2^49.
#pragma unroll
  for (int q = 0; q < NR; ++q)
#pragma unroll
    for (int t = 0; t < MT; ++t) {
      long long v[4];   // (g, re), (g, im), (g + 8, re), (g + 8, im)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float *D = &d[q][t][i & 1][2 * (i >> 1)];
        v[i] = (long long)__float2int_rn(D[0] * 281474976710656.0f) * 256 + __float2int_rn(D[1] * 281474976710656.0f);
      }
      const bool odd = c & 1, up = c & 2;
      long long w[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // keep (re if even, im if odd) of row g + 8 h
        const long long keep = odd ? v[2 * h + 1] : v[2 * h], send = odd ? v[2 * h] : v[2 * h + 1];
        const long long got = __shfl_xor_sync(0xffffffffu, send, 1);
        w[h] = odd ? got * 65536 + keep : keep * 65536 + got;
      }
      const long long mine = up ? w[1] : w[0], other = up ? w[0] : w[1];
      const long long got = __shfl_xor_sync(0xffffffffu, other, 2);
      out[q][t] = (er[t] == FX_BAD || ex[q] == FX_BAD)
                      ? __longlong_as_double(0x7ff8000000000000ll)
                      : fx_value(up ? got : mine, up ? mine : got, er[t] + ex[q] - 69);
    }
}

}  // namespace stdd
