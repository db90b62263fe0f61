// The products of the block recurrences (arXiv:0907.3261, Sec. 2, the algorithm box) on the tensor cores in
// exact digits: block times L x L matrix (U = S alpha, P = R + U gamma, V = W + Y gamma) and the L x L Gram
// products R~_0^H R and R~_0^H V, fused with the updates that feed them.
//
// GB300's FP64 pipe issues two lanes per clock per SM, and a complex multiply-add in FP32 pairs takes about 20
// packed instructions, so these products bounded the updates.  Here every factor is an integer of ND
// balanced base-256 digits (ND = 7: 55 bits and the sign, ND = 8: 63), and a digit is an FP16 number: the
// products of digits and their sums, below 2^22, are exact in mma.sync's FP32 accumulators.  One accumulator
// per order (the sum of the two digits' positions) for the orders 0 .. ND - 1, started at 1.5 2^23, whose
// bits are then the sum as an integer; what is dropped is below 2^-8ND of the largest product.  mma.sync and
// not tcgen05: a tile is 16 rows by at most 32 columns, and the thread that loads an element also
// owns the element of the same place in the product, so nothing but the digits of alpha and gamma passes
// through shared memory.  (Exact products of split factors on matrix units: K. Ozaki, T. Ogita, S. Oishi and
// S. M. Rump, Numer. Algorithms 59 (2012) 95.)
//
// Scales: in block times matrix, a power of two per row of the block, per row and per column of the
// matrix (its entries are first divided by their row's scale, which goes to the block's column, so that columns
// of very different size lose nothing where the matrix makes up for them, as alpha and gamma do).  In a Gram
// product, a power of two per column of either block, held by a warp from tile to tile while the columns'
// largest elements stay within 2^-GR_WINDOW of it; the warp's sums are 64-bit integers and go to FP64 when a scale
// changes or after GR_TILES tiles.
//
// What the common scales would lose is computed in FP64: an element of a product none of whose terms comes
// within DG_SPAN bits of them (a nearly diagonal matrix and a factor that much below the largest of its row), a
// tile of a Gram product one of whose columns' products has no row near both scales (add_in_fp64), and whatever
// has subnormals among its factors.  So every element keeps its own accuracy, whatever the others are.
// An infinity or a NaN makes its row of a product, and its row or column of a Gram product, infinite or NaN.
//
// A warp takes 16 rows at a time: thread (g, t) = (lane / 4, lane % 4) holds rows g, g + 8 and columns
// t + 4 i, i < NI = ceil(L / 4).  That is the layout of an mma A fragment with (re, im) as its pairs, and of
// the accumulators, so products need no exchange; a Gram product contracts over the rows, and movmatrix
// transposes the digits of both blocks.  Partial sums are added in a fixed order, bitwise reproducible.
//
// Measured on a GB300, 16^3x32, L = 12, with the call's 50 us, seven digits (double-float mode): U 0.30 ms against
// 0.62 in FP32 pairs; P and V 1.04 against 1.81; X and R 0.73 against 0.95; eight digits (FP64 mode): 0.37, 1.27
// and 0.81 against 1.76, 4.90 and 2.66 on the FP64 pipe.  L = 1: 0.11, 0.28 and 0.26 ms against 0.10, 0.36 and 0.46
// (FP32 pairs); 4^4, L = 4: as before, 35 to 60 us.  Looking for what has to be computed in FP64 takes 0.01 of
// U's time, 0.07 of P and V's and 0.04 of X and R's.  Bytes alone would take 0.14, 0.32 and 0.41 ms.  X and R is
// bound by the FP64 pipe (its updates stay FP64); the others
// are bound by the latency of a tile's chain at 12 to 16 warps per SM (tensor pipe 33 to 44%, integer pipe
// 35 to 42% before the looking).  P and V in three blocks of 168 registers; two copies of the product's code for
// U and Y overflow the instruction cache.  Scales without a bit to spare, more flushes: slower by 0.18 ms.
#include <type_traits>

#include "fixed.cuh"
#include "internal.h"

namespace {

using fx::i64;
using fx::u64;

constexpr int DG_TPB = 128;                // 4 warps
constexpr int DG_WARPS = DG_TPB / 32;
static_assert(DG_WARPS == 4, "Gram::write adds four warps' sums in pairs");
constexpr int GR_TILES = 8;                // |tile sum| <= 2^59.1: 8 of them stay below 2^63
constexpr int GR_WINDOW = 3;               // bits by which a tile's column may fall below its scale
constexpr int GR_SPAN = 4;                 // bits by which the factors of a tile's largest product may (GR_WINDOW at least)
constexpr int DG_BAD = 1 << 20;            // an exponent that marks an infinity or a NaN
// Bits by which the factor of a sum's largest term may fall below its row's scale: the digits then keep 2^-44 of
// the term (seven) or 2^-54 (eight).  Each bit less takes four times as many elements to be computed again: of a
// diagonal matrix and Gaussian columns 2.5e-4 at 7 bits, where P and V took 1.07 ms, 1.6e-5 at 9 (0.98).
template <int ND>
constexpr int DG_SPAN = ND == 8 ? 7 : 9;
constexpr int DG_TINY = 64;                // exponent fields up to this one: subnormals beside them count
constexpr unsigned DG_MAGIC = 0x4B400000u;   // 1.5 2^23

WD_DEV void mma16(float c[4], const unsigned a[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
WD_DEV void mma8(float c[4], unsigned a0, unsigned a1, unsigned b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5},{%6},{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}
WD_DEV unsigned transposed(unsigned a) {
  unsigned d;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(d) : "r"(a));
  return d;
}
WD_DEV unsigned hfma2(unsigned a, unsigned b, unsigned c) {
  unsigned d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;\n" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
WD_DEV int raw_exponent(double v) { return (__double2hiint(v) >> 20) & 0x7FF; }
// v is not zero (v with an exponent field of at most DG_TINY).
WD_DEV bool nonzero(double2 v) {
  return ((__double2hiint(v.x) | __double2hiint(v.y)) & 0x7FFFFFFF) | __double2loint(v.x) | __double2loint(v.y);
}

// |v| >> sh as an integer of 8 ND - 1 bits for a v in [1, 2) 2^e at sh = 0, plus 128 in every byte below the
// top digit's.  FP64 subnormals count as zero.
template <int ND>
WD_DEV u64 biased(double v, int e_minus_scale) {
  const int h = __double2hiint(v);
  const int sh = (h & 0x7FF00000) ? -e_minus_scale : 64;
  const u64 m = ((u64)(unsigned)((h & 0xFFFFF) | 0x100000) << 32 | (unsigned)__double2loint(v))
                << (ND == 8 ? 10 : 2);
  return fx::shr_u(m, sh) + (ND == 8 ? 0x0080808080808080ull : 0x0000808080808080ull);
}
// v as a digit integer for the scale E: |v| < 2^(E - 1022), e added to v's exponent.
template <int ND>
WD_DEV u64 biased_at(double v, int e, int E) {
  return biased<ND>(v, raw_exponent(v) + e - E);
}
// The ND digits of x and y (biased magnitudes, signs from the words hx, hy) as FP16 pairs, most significant
// first: the bytes b become 1024 + b, and (1024 + b) s - 1152 s is the digit (the top one has no bias).
template <int ND>
WD_DEV void digits(u64 x, u64 y, int hx, int hy, unsigned d[ND]) {
  const unsigned p = __byte_perm(hx, hy, 0x7030) & 0x80008000u;
  const unsigned s = p | 0x3C003C00u, c = p ^ 0xE480E480u, ct = p ^ 0xE400E400u;
  const unsigned xl = (unsigned)x, yl = (unsigned)y, xh = (unsigned)(x >> 32), yh = (unsigned)(y >> 32);
  const unsigned w[4] = {__byte_perm(xl, yl, 0x5140), __byte_perm(xl, yl, 0x7362),
                         __byte_perm(xh, yh, 0x5140), __byte_perm(xh, yh, 0x7362)};
#pragma unroll
  for (int j = 0; j < ND; ++j)
    d[ND - 1 - j] = hfma2(__byte_perm(w[j >> 1], 0x64646464u, (j & 1) ? 0x4342 : 0x4140), s,
                          j == ND - 1 ? ct : c);
}

// v 2^k, rounded once.  The FP64 pipe's conversions would take 130 cycles of it per warp.
WD_DEV double scaled(i64 v, int k) {
  const i64 sg = v >> 63;
  const u64 m = (u64)((v ^ sg) - sg);
  const int n = __clzll((i64)m);
  const u64 q = (((m << (n & 63)) >> 10) + 1) >> 1;
  const int h = (int)(q >> 32) + ((1085 - n + k) << 20);
  return m ? __hiloint2double(h | ((int)(sg) & 0x80000000), (int)q) : 0.0;
}
__device__ __noinline__ double scaled_any(i64 v, int k) { return ldexp(scaled(v, 0), k); }
// re 2^(k + kr), im 2^(k + ki) for small kr, ki.
WD_DEV double2 scaled2(i64 re, i64 im, int k, int kr = 0, int ki = 0) {
  if ((unsigned)(k + 900) < 1700u) return make_double2(scaled(re, k + kr), scaled(im, k + ki));
  if (k < DG_BAD / 2) return make_double2(scaled_any(re, k + kr), scaled_any(im, k + ki));
  const double nan = __longlong_as_double(0x7FF8000000000000LL);
  return make_double2(nan, nan);
}

// Sums of the orders as an integer (j: accumulator bits, b: the bits that stand for zero), the order 0 in
// units of 2^(40 + UP); the orders 6 and 7 are rounded (a floor's bias would grow with the rows of a Gram
// product).
template <int ND, int UP>
WD_DEV i64 joined(const unsigned j[ND], unsigned b) {
  const int A = (int)((j[0] << 8) + j[1] - 257u * b), B = (int)((j[2] << 8) + j[3] - 257u * b);
  const int C = (int)((j[4] << 8) + j[5] - 257u * b);
  int D;
  if constexpr (ND == 8) D = (int)((j[6] << 8) + j[7] - 257u * b + (1u << (15 - UP))) >> (16 - UP);
  else D = (int)(j[6] - b + (1u << (7 - UP))) >> (8 - UP);
  return (i64)B * (1 << (16 + UP)) + ((i64)C * (1 << UP) + D) + (i64)((u64)(i64)A << (32 + UP));
}
// The same for one sum of a product, in the units of UP = 3 times 2^k: with eight digits the sum moves up by
// its own leading zeros, so that a small one loses nothing in the 64 bits.
template <int ND>
WD_DEV i64 product_sum(const unsigned j[ND], unsigned b, int& k) {
  k = 0;
  if constexpr (ND == 7) return joined<ND, 3>(j, b);
  const int A = (int)((j[0] << 8) + j[1] - 257u * b), B = (int)((j[2] << 8) + j[3] - 257u * b);
  const int C = (int)((j[4] << 8) + j[5] - 257u * b), D = (int)((j[6] << 8) + j[7] - 257u * b);
  const i64 hi = (i64)A * 65536 + B, lo = (i64)C * 65536 + D;    // below 2^45; hi counts 2^32
  const int up = min(__clzll((i64)fx::absbits(hi)) - 2, 32);
  k = 19 - up;
  return (i64)((u64)hi << up) + fx::shr_s(lo + (i64)((1ull << (32 - up)) >> 1), 32 - up);
}

// t + z f
WD_DEV double2 axpy(double2 t, double2 z, double2 f) {
  return make_double2(fma(-z.y, f.y, fma(z.x, f.x, t.x)), fma(z.y, f.x, fma(z.x, f.y, t.y)));
}

// ---------------------------------------------------------------- block times matrix
// The digits of an L x L matrix as mma B fragments, and its scales.
template <int NI, int ND>
struct Coef {
  unsigned d[NI * NI * ND * 32];           // [column tile][entry group][digit][lane]
  int rmax[4 * NI], cmax[4 * NI];          // largest exponent field of a row; 4096 + of a column less its row's scale
  unsigned tops[4 * NI];                   // bits a: entry (a, b) has column b's scale; LOST: subnormals
  int lost;                                // some column has them
  static constexpr unsigned LOST = 1u << 31;
  // |m_ab| < 2^(row + col - 1022); a row or column of zeros has any scale
  WD_DEV int row(int a) const { return rmax[a] ? rmax[a] - 1023 : 0; }
  WD_DEV int col(int b) const { return cmax[b] == 0 ? 1023 : cmax[b] == DG_BAD ? DG_BAD : cmax[b] - 4096; }
  // which factors of a row of the block make a term of the column's scale
  WD_DEV unsigned top(int b) const { return tops[b] & LOST ? 0 : cmax[b] == 0 ? 0xFFFFu : tops[b]; }
};

// Fills `t` from the matrix m, staged in `st` (L^2 entries); ends with a barrier.
template <int NI, int ND>
WD_DEV void load_coef(Coef<NI, ND>& t, double2* st, const double2* __restrict__ m, int L) {
  const int tid = threadIdx.x;
  if (tid < 4 * NI) t.rmax[tid] = t.cmax[tid] = t.tops[tid] = 0;
  if (!tid) t.lost = 0;
  __syncthreads();
  // exponent fields: 0 for zero, 2047 for an infinity or a NaN, which do not count for a row's scale
  for (int e = tid; e < L * L; e += DG_TPB) {
    const double2 v = st[e] = m[e];
    const int x = fx::exponent_of(v);
    if (x && x < 2047) atomicMax(&t.rmax[e / L], x);
  }
  __syncthreads();
  for (int e = tid; e < L * L; e += DG_TPB) {
    const int x = fx::exponent_of(st[e]), a = e / L;
    if (x) atomicMax(&t.cmax[e - a * L], x == 2047 ? DG_BAD : 4096 + x - t.row(a));
  }
  __syncthreads();
  for (int e = tid; e < L * L; e += DG_TPB) {
    const int x = fx::exponent_of(st[e]), a = e / L, b = e - a * L;
    if (x <= DG_TINY) {
      if (nonzero(st[e])) {
        atomicOr(&t.tops[b], t.LOST);
        t.lost = 1;
      }
    } else if (4096 + x - t.row(a) == t.cmax[b]) {
      atomicOr(&t.tops[b], 1u << a);
    }
  }
  for (int q = tid; q < NI * NI * 32; q += DG_TPB) {
    const int lane = q & 31, ni = q >> 5, i = ni % NI, nt = ni / NI;
    const int a = (lane & 3) + 4 * i, b = (lane >> 3) + 4 * nt, ra = t.row(a), cb = t.col(b);
    double2 v = make_double2(0.0, 0.0);
    if (a < L && b < L) v = st[a * L + b];
    // column 2b of the real matrix has (re, -im) in rows 2a, 2a + 1, column 2b + 1 (im, re)
    const double x = (lane & 4) ? v.y : v.x, y = (lane & 4) ? v.x : -v.y;
    unsigned d[ND];
    digits<ND>(biased_at<ND>(x, -ra, cb), biased_at<ND>(y, -ra, cb), __double2hiint(x), __double2hiint(y), d);
#pragma unroll
    for (int k = 0; k < ND; ++k) t.d[(ni * ND + k) * 32 + lane] = d[k];
  }
  __syncthreads();
}

// This lane's element (row of A + zeta V, column t of the four columns at m) in FP64 arithmetic; V may be null.
// `who`: the lanes that ask.  Each row's four lanes share the sum over the factors.  Rare, and so kept small: fetching
// cold code costs more than the arithmetic.
__device__ __noinline__ double2 exact_product(const double2* A, const double2* V, double2 zeta, const double2* m,
                                              int L, unsigned who) {
  const int t = threadIdx.x & 3;
  double2 mine = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    if (!(who & 0x11111111u << c)) continue;
    double2 v = make_double2(0.0, 0.0);
    if (who >> (threadIdx.x & 28) >> c & 1) {
#pragma unroll 1
      for (int a = t; a < L; a += 4) {
        double2 x = A[a];
        if (V) x = axpy(x, zeta, V[a]);
        v = axpy(v, x, m[a * L + c]);
      }
    }
#pragma unroll 1
    for (int k = 1; k < 4; k <<= 1) {
      v.x += __shfl_xor_sync(0xFFFFFFFFu, v.x, k);
      v.y += __shfl_xor_sync(0xFFFFFFFFu, v.y, k);
    }
    if (t == c) mine = v;
  }
  return mine;
}

// The product of the warp's 16 rows with the matrix: put(h, nt, base, v) gets element (row g + 8 h, column
// t + 4 nt), base from get(h, nt).  `ok`: the thread's elements (bits h * NI + i).  Where the digits hold too
// few bits of a sum's terms -- none has a factor within DG_SPAN of its row's scale and an entry of its column's --
// exact(h, nt, who) gives it in the end, when the digits' registers are free (who: the lanes that ask).
template <int NI, int ND, class G, class X, class F>
WD_DEV void row_product(const double2 in[2][NI], const Coef<NI, ND>& t, unsigned ok, const G& get, const X& exact,
                        const F& put) {
  const int lane = threadIdx.x & 31;
  unsigned a[ND][2][NI];
  constexpr int ZERO = -4000, LOST = DG_BAD - 100;   // exponents of zeros and of what the digits lose
  int E[2];
  unsigned within = 0;                     // the thread's factors within DG_SPAN of their row's scale
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    int ra[NI], ex[NI];
    E[h] = ZERO;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      ra[i] = t.row((lane & 3) + 4 * i);
      const int e = fx::exponent_of(in[h][i]);
      ex[i] = e == 2047 ? DG_BAD : e ? e + ra[i] : ZERO;
      if (e <= DG_TINY && nonzero(in[h][i])) ex[i] = LOST;
      E[h] = max(E[h], ex[i]);
    }
    E[h] = max(E[h], __shfl_xor_sync(0xFFFFFFFFu, E[h], 1));
    E[h] = max(E[h], __shfl_xor_sync(0xFFFFFFFFu, E[h], 2));
    const int lim = E[h] == LOST ? DG_BAD : E[h] - DG_SPAN<ND>;
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (ex[i] >= lim) within |= 1u << (h * NI + i);
    if (E[h] == ZERO) E[h] = 1023;         // a row of zeros
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const double2 v = in[h][i];
      unsigned d[ND];
      digits<ND>(biased_at<ND>(v.x, ra[i], E[h]), biased_at<ND>(v.y, ra[i], E[h]), __double2hiint(v.x),
                 __double2hiint(v.y), d);
#pragma unroll
      for (int k = 0; k < ND; ++k) a[k][h][i] = d[k];
    }
  }
#pragma unroll 1
  for (int nt = 0; nt < NI; ++nt) {
    const double2 base[2] = {get(0, nt), get(1, nt)};
    float acc[ND][4];
#pragma unroll
    for (int o = 0; o < ND; ++o)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[o][q] = __uint_as_float(DG_MAGIC);
    const unsigned* bd = t.d + nt * NI * ND * 32 + lane;
#pragma unroll
    for (int i = 0; i + 1 < NI; i += 2) {
#pragma unroll
      for (int k2 = 0; k2 < ND; ++k2) {
        const unsigned b0 = bd[(i * ND + k2) * 32], b1 = bd[((i + 1) * ND + k2) * 32];
#pragma unroll
        for (int k1 = 0; k1 + k2 < ND; ++k1) {
          const unsigned f[4] = {a[k1][0][i], a[k1][1][i], a[k1][0][i + 1], a[k1][1][i + 1]};
          mma16(acc[k1 + k2], f, b0, b1);
        }
      }
    }
    if constexpr (NI & 1) {
#pragma unroll
      for (int k2 = 0; k2 < ND; ++k2) {
        const unsigned b0 = bd[((NI - 1) * ND + k2) * 32];
#pragma unroll
        for (int k1 = 0; k1 + k2 < ND; ++k1)
          mma8(acc[k1 + k2], a[k1][0][NI - 1], a[k1][1][NI - 1], b0);
      }
    }
    const int C = t.col((lane & 3) + 4 * nt);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      unsigned re[ND], im[ND];
#pragma unroll
      for (int o = 0; o < ND; ++o) {
        re[o] = __float_as_uint(acc[o][2 * h]);
        im[o] = __float_as_uint(acc[o][2 * h + 1]);
      }
      int kr, ki;
      const i64 sr = product_sum<ND>(re, DG_MAGIC, kr), si = product_sum<ND>(im, DG_MAGIC, ki);
      put(h, nt, base[h], scaled2(sr, si, E[h] + C - 2101, kr, ki));
    }
  }
  if (__any_sync(0xFFFFFFFFu, (~within & ok) || t.lost)) {
    unsigned large = 0;                    // bits a (h = 0) and 16 + a: the row's factors within the span
#pragma unroll
    for (int q = 0; q < 2 * NI; ++q)
      if (within >> q & 1) large |= 1u << ((lane & 3) + (q < NI ? 4 * q : 16 + 4 * (q - NI)));
    large |= __shfl_xor_sync(0xFFFFFFFFu, large, 1);
    large |= __shfl_xor_sync(0xFFFFFFFFu, large, 2);
#pragma unroll 1
    for (int nt = 0; nt < NI; ++nt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool lossy = (ok >> (h * NI + nt) & 1) && !(large >> 16 * h & t.top((lane & 3) + 4 * nt));
        const unsigned who = __ballot_sync(0xFFFFFFFFu, lossy);
        if (who) {
          const double2 v = exact(h, nt, who);
          if (lossy) put(h, nt, get(h, nt), v);
        }
      }
  }
}

// ---------------------------------------------------------------- Gram product
// The larger part's high word without its sign (its exponent above 20 bits), at least 1 for what is not zero.
WD_DEV unsigned word(double2 v) {
  const unsigned x = (__double2hiint(v.x) & 0x7FFFFFFF) | min((unsigned)__double2loint(v.x), 1u);
  const unsigned y = (__double2hiint(v.y) & 0x7FFFFFFF) | min((unsigned)__double2loint(v.y), 1u);
  return max(x, y);
}
// The least word of an element within `span` of a scale.
WD_DEV unsigned span_word(int E, int span) { return (unsigned)max(E - span, DG_TINY + 1) << 20; }

// A tile of `n` rows without one whose elements are all within GR_SPAN.  A product loses nothing if some row has
// both factors within `span`, or if no row has both; if one does lose, adds A^H B to this thread's elements of
// `out` in FP64 arithmetic and returns true.  ea, eb: the scales of columns t + 4 i.  Rare (see exact_product).
__device__ __noinline__ bool add_in_fp64(double2* out, int ld, const double2* A, const double2* B, int n, int L,
                                         int4 ea, int4 eb, int span) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  // Of this quad's columns (of A, << 16: of B): the rows within the span, the rows that are not zero.
  unsigned within[4], some[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int c = t + 4 * i;
    const unsigned la = span_word(i == 0 ? ea.x : i == 1 ? ea.y : i == 2 ? ea.z : ea.w, span);
    const unsigned lb = span_word(i == 0 ? eb.x : i == 1 ? eb.y : i == 2 ? eb.z : eb.w, span);
    within[i] = some[i] = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = g + 8 * h;
      if (c >= L || r >= n) continue;
      const unsigned x = word(A[(size_t)r * L + c]), y = word(B[(size_t)r * L + c]);
      within[i] |= (x >= la ? 1u << r : 0) | (y >= lb ? 65536u << r : 0);
      some[i] |= (x ? 1u << r : 0) | (y ? 65536u << r : 0);
    }
#pragma unroll
    for (int k = 4; k < 32; k <<= 1) {
      within[i] |= __shfl_xor_sync(0xFFFFFFFFu, within[i], k);
      some[i] |= __shfl_xor_sync(0xFFFFFFFFu, some[i], k);
    }
  }
  unsigned short rows[8];                  // of this thread's products: the rows with both factors
  bool lossy = false;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    const unsigned w0 = __shfl_sync(0xFFFFFFFFu, within[2 * mt], g >> 1);
    const unsigned w1 = __shfl_sync(0xFFFFFFFFu, within[2 * mt + 1], g >> 1);
    const unsigned s0 = __shfl_sync(0xFFFFFFFFu, some[2 * mt], g >> 1);
    const unsigned s1 = __shfl_sync(0xFFFFFFFFu, some[2 * mt + 1], g >> 1);
    const unsigned w = (g & 1) ? w1 : w0, s = (g & 1) ? s1 : s0;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const unsigned both = s & some[nt] >> 16;
      rows[4 * mt + nt] = (unsigned short)both;
      lossy = lossy || ((both & 0xFFFFu) && !(w & within[nt] >> 16));
    }
  }
  if (!__any_sync(0xFFFFFFFFu, lossy)) return false;
#pragma unroll 1
  for (int q = 0; q < 8; ++q) {
    const int a = 8 * (q >> 2) + 4 * (g & 1) + (g >> 1), b = t + 4 * (q & 3);
    if (!rows[q]) continue;                // also columns beyond L
    double2 v = out[a * ld + b];
#pragma unroll 1
    for (unsigned m = rows[q]; m; m &= m - 1) {
      const size_t r = (size_t)(__ffs((int)m) - 1) * L;
      const double2 x = A[r + a];
      v = axpy(v, make_double2(x.x, -x.y), B[r + b]);
    }
    out[a * ld + b] = v;
  }
  return true;
}

// One warp's A^H B: element (a, b), a = 8 mt + 4 (g % 2) + g / 2 and b = t + 4 nt, belongs to thread (g, t).
template <int NI, int ND>
struct Gram {
  static constexpr int MT = (NI + 1) / 2, NV = MT * NI * 2, LD = 4 * NI;
  i64* sum;                                // [NV][DG_TPB], this thread's slots
  double2* out;                            // [LD][LD] of this warp
  int ea[NI], eb[NI], tiles;
  unsigned bad;                            // bits i: column t + 4 i of A, 8 + i: of B holds an infinity or a NaN

  WD_DEV void init(i64* s, double2* o) {
    sum = s;
    out = o;
    tiles = 0;
    bad = 0;
#pragma unroll
    for (int i = 0; i < NI; ++i) ea[i] = eb[i] = -1;
#pragma unroll
    for (int q = 0; q < NV; ++q) sum[q * DG_TPB] = 0;
    for (int e = threadIdx.x & 31; e < LD * LD; e += 32) out[e] = make_double2(0.0, 0.0);
    __syncwarp();
  }
  WD_DEV void flush() {
    const int lane = threadIdx.x & 31, g = lane >> 2, tt = lane & 3;
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      const int e0 = __shfl_sync(0xFFFFFFFFu, ea[2 * mt], g >> 1);
      const int e1 = 2 * mt + 1 < NI ? __shfl_sync(0xFFFFFFFFu, ea[2 * mt + 1 < NI ? 2 * mt + 1 : 0], g >> 1) : 0;
      const int E = (g & 1) ? e1 : e0, a = 8 * mt + 4 * (g & 1) + (g >> 1);
#pragma unroll
      for (int nt = 0; nt < NI; ++nt) {
        i64* s = sum + (mt * NI + nt) * 2 * DG_TPB;
        const double2 v = scaled2(s[0], s[DG_TPB], E + eb[nt] - 2098);
        if (a < LD) {
          double2& o = out[a * LD + tt + 4 * nt];
          o = make_double2(o.x + v.x, o.y + v.y);
        }
        s[0] = 0;
        s[DG_TPB] = 0;
      }
    }
    tiles = 0;
  }
  // The largest word of a tile's column from this thread's two; an infinity or a NaN sets `bit` of `bad`.
  WD_DEV static unsigned column(unsigned w0, unsigned w1, unsigned& bad, int bit) {
    unsigned w = max(w0, w1);
    if (w >= 0x7FF00000u) {
      bad |= 1u << bit;
      w = 0x7FE00000u;
    }
    w = max(w, __shfl_xor_sync(0xFFFFFFFFu, w, 4));
    w = max(w, __shfl_xor_sync(0xFFFFFFFFu, w, 8));
    return max(w, __shfl_xor_sync(0xFFFFFFFFu, w, 16));
  }
  // A tile of the rows from n0 on.  `pa`, `pb`: the blocks, whose rows the warp may have just written.
  WD_DEV void tile(const double2 A[2][NI], const double2 B[2][NI], const double* pa, const double* pb, long long n0,
                   long long n1, int L) {
    {
      unsigned wa[2][NI], wb[2][NI], ca[NI], cb[NI];
      bool moved = tiles == GR_TILES;      // some column left its window
#pragma unroll
      for (int i = 0; i < NI; ++i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          wa[h][i] = word(A[h][i]);
          wb[h][i] = word(B[h][i]);
        }
        ca[i] = column(wa[0][i], wa[1][i], bad, i);
        cb[i] = column(wb[0][i], wb[1][i], bad, 8 + i);
        const int na = ca[i] >> 20, nb = cb[i] >> 20;
        moved = moved || na > ea[i] || nb > eb[i] || (na && na < ea[i] - GR_WINDOW) ||
                (nb && nb < eb[i] - GR_WINDOW);
      }
      if (__any_sync(0xFFFFFFFFu, moved)) {
        if (tiles) flush();
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int na = ca[i] >> 20, nb = cb[i] >> 20;
          if (na || ea[i] < 0) ea[i] = na + (ea[i] >= 0);   // from the second time on with a bit to spare
          if (nb || eb[i] < 0) eb[i] = nb + (eb[i] >= 0);
        }
      }
      ++tiles;
      // A row whose elements are all within the span makes products that are.
      bool in0 = true, in1 = true;         // this quad's elements of rows g and g + 8 (a column of zeros loses nothing)
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const unsigned la = ca[i] ? span_word(ea[i], GR_SPAN) : 0, lb = cb[i] ? span_word(eb[i], GR_SPAN) : 0;
        in0 = in0 && wa[0][i] >= la && wb[0][i] >= lb;
        in1 = in1 && wa[1][i] >= la && wb[1][i] >= lb;
      }
      const unsigned r0 = __ballot_sync(0xFFFFFFFFu, in0), r1 = __ballot_sync(0xFFFFFFFFu, in1);
      const unsigned p0 = r0 & r0 >> 1, p1 = r1 & r1 >> 1;
      if (!((p0 & p0 >> 2 | p1 & p1 >> 2) & 0x11111111u)) {
        auto four = [](const int e[NI]) {
          return make_int4(e[0], e[NI > 1 ? 1 : 0], e[NI > 2 ? 2 : 0], e[NI > 3 ? 3 : 0]);
        };
        __syncwarp();                      // the warp may have just written the rows
        const double2 *ra = reinterpret_cast<const double2*>(pa), *rb = reinterpret_cast<const double2*>(pb);
        if (add_in_fp64(out, LD, ra + n0 * L, rb + n0 * L, (int)min(16LL, n1 - n0), L, four(ea), four(eb),
                        ND == 8 ? 1 : GR_SPAN))
          return;
      }
    }
    unsigned b[NI][2][ND];
#pragma unroll
    for (int nt = 0; nt < NI; ++nt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const double2 v = B[h][nt];
        digits<ND>(biased_at<ND>(v.x, 0, eb[nt]), biased_at<ND>(v.y, 0, eb[nt]), __double2hiint(v.x),
                   __double2hiint(v.y), b[nt][h]);
#pragma unroll
        for (int k = 0; k < ND; ++k) b[nt][h][k] = transposed(b[nt][h][k]);
      }
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
      unsigned a[ND][4];                   // rows g: real parts, rows g + 8: imaginary parts
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        double2 v[2];
        int e[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {      // columns 2 mt + c
          const bool lo = MT == 1 || mt == 0;
          v[c] = lo ? (c < NI ? A[h][c < NI ? c : 0] : make_double2(0.0, 0.0))
                    : (2 + c < NI ? A[h][2 + c < NI ? 2 + c : 0] : make_double2(0.0, 0.0));
          e[c] = lo ? ea[c < NI ? c : 0] : ea[2 + c < NI ? 2 + c : 0];
        }
        unsigned d[ND];
        digits<ND>(biased_at<ND>(v[0].x, 0, e[0]), biased_at<ND>(v[1].x, 0, e[1]), __double2hiint(v[0].x),
                   __double2hiint(v[1].x), d);
#pragma unroll
        for (int k = 0; k < ND; ++k) a[k][2 * h] = transposed(d[k]);
        digits<ND>(biased_at<ND>(v[0].y, 0, e[0]), biased_at<ND>(v[1].y, 0, e[1]), __double2hiint(v[0].y),
                   __double2hiint(v[1].y), d);
#pragma unroll
        for (int k = 0; k < ND; ++k) a[k][2 * h + 1] = transposed(d[k]);
      }
#pragma unroll
      for (int nt = 0; nt < NI; ++nt) {
        float acc[ND][4];
#pragma unroll
        for (int o = 0; o < ND; ++o)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[o][q] = __uint_as_float(DG_MAGIC);
#pragma unroll
        for (int k2 = 0; k2 < ND; ++k2)
#pragma unroll
          for (int k1 = 0; k1 + k2 < ND; ++k1) mma16(acc[k1 + k2], a[k1], b[nt][0][k2], b[nt][1][k2]);
        unsigned re[ND], im[ND];
#pragma unroll
        for (int o = 0; o < ND; ++o) {
          re[o] = __float_as_uint(acc[o][0]) + __float_as_uint(acc[o][3]);
          im[o] = __float_as_uint(acc[o][1]) - __float_as_uint(acc[o][2]);
        }
        i64* s = sum + (mt * NI + nt) * 2 * DG_TPB;
        s[0] += joined<ND, 0>(re, 2u * DG_MAGIC);
        s[DG_TPB] += joined<ND, 0>(im, 0u);
      }
    }
  }
  // The block's sums into its slot of the partial sums; `nacc`: this thread's column norms, or null.
  WD_DEV void write(double2* __restrict__ part, const double2* all, double* nred, int L, const double* nacc) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    flush();
    unsigned m = bad;
#pragma unroll
    for (int k = 4; k < 32; k <<= 1) m |= __shfl_xor_sync(0xFFFFFFFFu, m, k);
    const double nan = __longlong_as_double(0x7FF8000000000000LL);
    __syncwarp();
    if (lane < 4) {
#pragma unroll
      for (int i = 0; i < NI; ++i)
        for (int q = 0; q < LD; ++q) {
          if (m >> i & 1) out[(lane + 4 * i) * LD + q] = make_double2(nan, nan);
          if (m >> (8 + i) & 1) out[q * LD + lane + 4 * i] = make_double2(nan, nan);
        }
    }
    if (nacc) {
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        double v = nacc[i];
#pragma unroll
        for (int k = 4; k < 32; k <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, k);
        if (lane < 4) nred[w * 16 + lane + 4 * i] = v;
      }
    }
    __syncthreads();
    double2* p = part + (size_t)blockIdx.x * PART_STRIDE;
    for (int e = threadIdx.x; e < L * L; e += DG_TPB) {
      const int a = e / L, b = e - a * L;
      const double2* w = all + a * LD + b;
      const double2 u = w[0], v = w[LD * LD], x = w[2 * LD * LD], y = w[3 * LD * LD];
      p[e] = make_double2((u.x + v.x) + (x.x + y.x), (u.y + v.y) + (x.y + y.y));
    }
    if (nacc && threadIdx.x < L) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < DG_WARPS; ++k) v += nred[k * 16 + threadIdx.x];
      p[WD_LMAX * WD_LMAX + threadIdx.x] = make_double2(v, 0.0);
    }
  }
};

// This thread's elements of a tile's rows; `e` and `ok` from Place.
template <int NI>
struct Place {
  size_t e[2];                             // element (row g + 8 h, column t)
  bool row[2];
  int left;                                // columns left from t on
  WD_DEV Place(long long tile, int L, long long rows) {
    const int lane = threadIdx.x & 31;
    left = L - (lane & 3);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long long n = tile * 16 + (lane >> 2) + 8 * h;
      row[h] = n < rows;
      e[h] = (size_t)n * L + (lane & 3);
    }
  }
  WD_DEV bool ok(int h, int i) const { return row[h] && 4 * i < left; }
  WD_DEV unsigned mask() const {           // bits h * NI + i of the elements that are ok
    const unsigned m = (1u << max(0, (left + 3) / 4)) - 1;
    return (row[0] ? m : 0) | (row[1] ? m << NI : 0);
  }
  WD_DEV void load(const double* __restrict__ p, double2 v[2][NI]) const {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < NI; ++i)
        v[h][i] = ok(h, i) ? reinterpret_cast<const double2*>(p)[e[h] + 4 * i] : make_double2(0.0, 0.0);
  }
};
// A tile's elements on their way to the thread that asked for them: its own slots of shared memory, so a
// wait of the thread is all that a read needs.
template <int NI>
struct Staged {
  double2 slot[2 * NI][DG_TPB];
  WD_DEV void ask(const Place<NI>& pl, const double* __restrict__ p) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const bool ok = pl.ok(h, i);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                         (unsigned)__cvta_generic_to_shared(&slot[h * NI + i][threadIdx.x])),
                     "l"(ok ? p + 2 * (pl.e[h] + 4 * i) : p), "r"(ok ? 16 : 0)
                     : "memory");
      }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  WD_DEV void take(double2 v[2][NI]) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < NI; ++i) v[h][i] = slot[h * NI + i][threadIdx.x];
  }
};
WD_DEV double2& at(double* p, size_t e) { return reinterpret_cast<double2*>(p)[e]; }
WD_DEV const double2& at(const double* p, size_t e) { return reinterpret_cast<const double2*>(p)[e]; }

// Blocks per SM of the three kinds of kernels; their shared memory beyond 48 KB is dynamic.
constexpr int u_blocks(int NI, int ND) { return ND == 8 && NI >= 3 ? 3 : 4; }
constexpr int gram_blocks(int NI, int ND) { return NI == 4 || (ND == 8 && NI == 3) ? 3 : 4; }
constexpr int pv_blocks(int NI, int) { return NI >= 3 ? 3 : 4; }
extern __shared__ __align__(16) unsigned char dg_smem[];

template <int NI, int ND>
struct ShU {
  Staged<NI> sp, sv;                       // sp is also the matrix's stage
  Coef<NI, ND> al;
};
// U = (P - zeta V) alpha
template <int NI, int ND>
__global__ void __launch_bounds__(DG_TPB, u_blocks(NI, ND))
update_u_dg_kernel(const double* __restrict__ P, const double* __restrict__ V, double* __restrict__ U, int L,
                   long long rows, const SolverState* __restrict__ st) {
  ShU<NI, ND>& sh = *reinterpret_cast<ShU<NI, ND>*>(dg_smem);
  Staged<NI>&sp = sh.sp, &sv = sh.sv;
  Coef<NI, ND>& al = sh.al;
  if (st->status != ST_OK) return;
  const double2 z = st->zeta, mz = make_double2(-z.x, -z.y);
  load_coef(al, &sp.slot[0][0], st->alpha, L);
  const long long tiles = (rows + 15) / 16, step = (long long)gridDim.x * DG_WARPS;
  long long q = (long long)blockIdx.x * DG_WARPS + (threadIdx.x >> 5);
  if (q < tiles) {
    const Place<NI> pl(q, L, rows);
    sp.ask(pl, P);
    sv.ask(pl, V);
  }
  for (; q < tiles; q += step) {
    const Place<NI> pl(q, L, rows);
    double2 s[2][NI], v[2][NI];
    sp.take(s);
    sv.take(v);
    if (q + step < tiles) {
      const Place<NI> next(q + step, L, rows);
      sp.ask(next, P);
      sv.ask(next, V);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < NI; ++i) s[h][i] = axpy(s[h][i], mz, v[h][i]);
    row_product<NI, ND>(
        s, al, pl.mask(), [](int, int) { return make_double2(0.0, 0.0); },
        [&](int h, int nt, unsigned who) {
          const size_t r = pl.e[h] - (threadIdx.x & 3);
          return exact_product(&at(P, r), &at(V, r), mz, st->alpha + 4 * nt, L, who);
        },
        [&](int h, int nt, double2, double2 u) {
          if (pl.ok(h, nt)) at(U, pl.e[h] + 4 * nt) = u;
        });
  }
}

// Partial A^H B, and the column norms of B.
template <int NI, int ND>
__global__ void __launch_bounds__(DG_TPB, gram_blocks(NI, ND))
gram_dg_kernel(const double* __restrict__ A, const double* __restrict__ B, int L, long long rows,
               double2* __restrict__ part, bool norms) {
  using Gr = Gram<NI, ND>;
  __shared__ i64 sums[Gr::NV][DG_TPB];
  __shared__ double2 outs[DG_WARPS][Gr::LD * Gr::LD];
  __shared__ double nred[DG_WARPS * 16];
  Gr gr;
  gr.init(&sums[0][threadIdx.x], outs[threadIdx.x >> 5]);
  double nacc[NI] = {};
  const long long tiles = (rows + 15) / 16;
  for (long long q = (long long)blockIdx.x * DG_WARPS + (threadIdx.x >> 5); q < tiles;
       q += (long long)gridDim.x * DG_WARPS) {
    const Place<NI> pl(q, L, rows);
    double2 a[2][NI], b[2][NI];
    pl.load(A, a);
    pl.load(B, b);
    if (norms) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < NI; ++i) nacc[i] = fma(b[h][i].x, b[h][i].x, fma(b[h][i].y, b[h][i].y, nacc[i]));
    }
    gr.tile(a, b, A, B, q * 16, rows, L);
  }
  gr.write(part, outs[0], nred, L, norms ? nacc : nullptr);
}

// X += zeta F + G;  R -= zeta W + Y;  partial R~_0^H R_{k+1} and ||r_i||^2.
template <int NI, int ND>
__global__ void __launch_bounds__(DG_TPB, gram_blocks(NI, ND))
update_xr_dg_kernel(double* __restrict__ X, const double* __restrict__ F, const double* __restrict__ G,
                    double* __restrict__ R, const double* __restrict__ W, const double* __restrict__ Y,
                    const double* __restrict__ Rt, int L, long long rows, double2* __restrict__ part,
                    const SolverState* __restrict__ st) {
  using Gr = Gram<NI, ND>;
  __shared__ __align__(16) i64 sums[Gr::NV][DG_TPB];
  __shared__ double2 outs[DG_WARPS][Gr::LD * Gr::LD];
  __shared__ double nred[DG_WARPS * 16];
  if (st->status != ST_OK) return;
  const double2 z = st->zeta, mz = make_double2(-z.x, -z.y);
  Gr gr;
  gr.init(&sums[0][threadIdx.x], outs[threadIdx.x >> 5]);
  double nacc[NI] = {};
  const long long tiles = (rows + 15) / 16;
  for (long long q = (long long)blockIdx.x * DG_WARPS + (threadIdx.x >> 5); q < tiles;
       q += (long long)gridDim.x * DG_WARPS) {
    const Place<NI> pl(q, L, rows);
    double2 r[2][NI], rt[2][NI];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const size_t e = pl.e[h] + 4 * i;
        r[h][i] = make_double2(0.0, 0.0);
        if (!pl.ok(h, i)) continue;
        const double2 x = at(X, e), g = at(G, e), y = at(Y, e);
        r[h][i] = at(R, e);
        at(X, e) = axpy(make_double2(x.x + g.x, x.y + g.y), z, at(F, e));
        r[h][i] = axpy(make_double2(r[h][i].x - y.x, r[h][i].y - y.y), mz, at(W, e));
        at(R, e) = r[h][i];
        nacc[i] = fma(r[h][i].x, r[h][i].x, fma(r[h][i].y, r[h][i].y, nacc[i]));
      }
    pl.load(Rt, rt);
    gr.tile(rt, r, Rt, R, q * 16, rows, L);
  }
  gr.write(part, outs[0], nred, L, nacc);
}

template <int NI, int ND>
struct ShPv {
  Staged<NI> sg;
  i64 sums[Gram<NI, ND>::NV][DG_TPB];      // also the matrix's stage
  double2 outs[DG_WARPS][16 * NI * NI];
  Coef<NI, ND> ga;
};
// P = R + U gamma;  V = W + Y gamma;  partial R~_0^H V_{k+1}.
template <int NI, int ND>
__global__ void __launch_bounds__(DG_TPB, pv_blocks(NI, ND))
update_pv_dg_kernel(double* __restrict__ P, double* __restrict__ V, const double* __restrict__ R,
                    const double* __restrict__ W, const double* __restrict__ U, const double* __restrict__ Y,
                    const double* __restrict__ Rt, int L, long long rows, double2* __restrict__ part,
                    const SolverState* __restrict__ st) {
  using Gr = Gram<NI, ND>;
  using Sh = ShPv<NI, ND>;
  Sh& sh = *reinterpret_cast<Sh*>(dg_smem);
  auto& sums = sh.sums;
  auto& outs = sh.outs;
  Coef<NI, ND>& ga = sh.ga;
  Staged<NI>& sg = sh.sg;
  if (st->status != ST_OK) return;
  const long long tiles = (rows + 15) / 16, step = (long long)gridDim.x * DG_WARPS;
  const long long q0 = (long long)blockIdx.x * DG_WARPS + (threadIdx.x >> 5);
  if (q0 < tiles) sg.ask(Place<NI>(q0, L, rows), U);
  load_coef(ga, reinterpret_cast<double2*>(sums), st->gamma, L);
  Gr gr;
  gr.init(&sums[0][threadIdx.x], outs[threadIdx.x >> 5]);
  for (long long q = q0; q < tiles; q += step) {
    const Place<NI> pl(q, L, rows);
    double2 u[2][NI], v[2][NI];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < NI; ++i) v[h][i] = make_double2(0.0, 0.0);
#pragma unroll 1                           // one copy of the product's code: two overflow the instruction cache
    for (int c = 0; c < 2; ++c) {
      const double* base = c ? W : R;
      double* out = c ? V : P;
      sg.take(u);
      sg.ask(pl, c ? Rt : Y);
      row_product<NI, ND>(
          u, ga, pl.mask(),
          [&](int h, int nt) { return pl.ok(h, nt) ? at(base, pl.e[h] + 4 * nt) : make_double2(0.0, 0.0); },
          [&](int h, int nt, unsigned who) {
            return exact_product(&at(c ? Y : U, pl.e[h] - (threadIdx.x & 3)), nullptr, double2(), st->gamma + 4 * nt,
                                 L, who);
          },
          [&](int h, int nt, double2 w, double2 p) {
            if (!pl.ok(h, nt)) return;
            const double2 x = make_double2(w.x + p.x, w.y + p.y);
            at(out, pl.e[h] + 4 * nt) = x;
#pragma unroll
            for (int i = 0; i < NI; ++i)
              if (i == nt) v[h][i] = x;    // V's in the end
          });
    }
    sg.take(u);
    if (q + step < tiles) sg.ask(Place<NI>(q + step, L, rows), U);
    gr.tile(u, v, Rt, V, q * 16, rows, L);
  }
  gr.write(part, outs[0], nullptr, L, nullptr);
}

// Calls f with the kernels' NI and ND.  Seven digits for the double-float updates, of which they are 30 times as
// exact as the FP32 pairs were, and eight for FP64's: a term is then off by less than 2^-58 of the largest factors'
// product, and the error that is left is the result's one rounding (relative to U's rms at L = 1 0.79e-16,
// against 0.93e-16 with seven and 0.83e-16 in FP64; at L = 4 seven had 1.23e-16 against 1.19e-16).
template <class F>
auto with_shape(int L, bool df, const F& f) {
  auto ni = [&](auto nd) {
    using std::integral_constant;
    if (L <= 4) return f(integral_constant<int, 1>(), nd);
    if (L <= 8) return f(integral_constant<int, 2>(), nd);
    if (L <= 12) return f(integral_constant<int, 3>(), nd);
    return f(integral_constant<int, 4>(), nd);
  };
  return df ? ni(std::integral_constant<int, 7>()) : ni(std::integral_constant<int, 8>());
}
template <class K>
cudaError_t allow_smem(K kernel, size_t bytes) {
  return bytes <= 48 * 1024 ? cudaSuccess
                            : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

int update_u_blocks(int L, bool df) {
  return with_shape(L, df, [](auto ni, auto nd) { return u_blocks(ni(), nd()); });
}
int gram_blocks(int L, bool df) {
  return with_shape(L, df, [](auto ni, auto nd) { return gram_blocks(ni(), nd()); });
}
int update_pv_blocks(int L, bool df) {
  return with_shape(L, df, [](auto ni, auto nd) { return pv_blocks(ni(), nd()); });
}

cudaError_t launch_update_u_dg(const double* P, const double* V, double* U, int L, long long rows, int nb,
                               const SolverState* st, cudaStream_t s, bool df) {
  return with_shape(L, df, [&](auto ni, auto nd) {
    constexpr size_t bytes = sizeof(ShU<ni(), nd()>);
    const cudaError_t e = allow_smem(update_u_dg_kernel<ni(), nd()>, bytes);
    if (e != cudaSuccess) return e;
    update_u_dg_kernel<ni(), nd()><<<nb, DG_TPB, bytes, s>>>(P, V, U, L, rows, st);
    return cudaGetLastError();
  });
}

cudaError_t launch_gram_dg(const double* A, const double* B, int L, long long rows, int nb, double2* part,
                           bool norms, cudaStream_t s) {
  return with_shape(L, false, [&](auto ni, auto nd) {
    gram_dg_kernel<ni(), nd()><<<nb, DG_TPB, 0, s>>>(A, B, L, rows, part, norms);
    return cudaGetLastError();
  });
}

cudaError_t launch_update_xr_dg(double* X, const double* F, const double* G, double* R, const double* W,
                                const double* Y, const double* Rt, int L, long long rows, int nb,
                                double2* part, const SolverState* st, cudaStream_t s, bool df) {
  return with_shape(L, df, [&](auto ni, auto nd) {
    update_xr_dg_kernel<ni(), nd()><<<nb, DG_TPB, 0, s>>>(X, F, G, R, W, Y, Rt, L, rows, part, st);
    return cudaGetLastError();
  });
}

cudaError_t launch_update_pv_dg(double* P, double* V, const double* R, const double* W, const double* U,
                                const double* Y, const double* Rt, int L, long long rows, int nb,
                                double2* part, const SolverState* st, cudaStream_t s, bool df) {
  return with_shape(L, df, [&](auto ni, auto nd) {
    constexpr size_t bytes = sizeof(ShPv<ni(), nd()>);
    const cudaError_t e = allow_smem(update_pv_dg_kernel<ni(), nd()>, bytes);
    if (e != cudaSuccess) return e;
    update_pv_dg_kernel<ni(), nd()><<<nb, DG_TPB, bytes, s>>>(P, V, R, W, U, Y, Rt, L, rows, part, st);
    return cudaGetLastError();
  });
}
