// The parts of the fixed-point stencil (dslash_fx.cu) that do not depend on its limbs: 64-bit integer helpers, conversions
// from and to FP64, and the loads of a hop's spinors.  A field is 16 bytes per complex number, site-major
// [site][spin*3+colour][rhs], with one exponent per (site, rhs); two threads of a warp share one
// (site, rhs), thread sp the upper spin sp in the hops and chirality sp in the site blocks.
#pragma once

#include "common.cuh"

namespace fx {

typedef long long i64;
typedef unsigned long long u64;

constexpr int FX_EMIN = 1;                 // smallest exponent of a field made from FP64
constexpr int FX_NONFINITE = 30000;        // the exponent of a spinor with an infinity or a NaN
constexpr int FX_EK = -4;                  // smallest exponent of the links' scale
// Bits by which a site's field may exceed its neighbours' before its block is done in FP64: beyond them the common
// scale would cost its small components more than FP64's rounding of the neighbours' part.
constexpr int FX_APART = 1;
constexpr int TPB = 128;
constexpr unsigned NB_MASK = (1u << 26) - 1u;

WD_DEV u64 shr_u(u64 v, int n) {           // counts above 63 give 0
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
WD_DEV i64 shr_s(i64 v, int n) {
  i64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
WD_DEV i64 shl(i64 v, int n) { return (i64)((u64)v << n); }   // defined for negative v
WD_DEV void mac(i64& a, int x, int y) { a += (i64)x * y; }

// The magnitude of an FP64 number (words h, l) as a 53-bit integer and a power of two: m 2^(ef - 1075).
WD_DEV u64 mantissa(int h, unsigned l, int& ef) {
  const int e = (h >> 20) & 0x7FF;
  ef = max(e, 1);
  return (u64)(unsigned)((h & 0xFFFFF) | (e ? 0x100000 : 0)) << 32 | l;
}
WD_DEV int exponent_of(double2 v) {
  return max((__double2hiint(v.x) >> 20) & 0x7FF, (__double2hiint(v.y) >> 20) & 0x7FF);
}
WD_DEV short field_exponent(int e) { return (short)(e < 2047 ? max(e, FX_EMIN) : FX_NONFINITE); }

WD_DEV void cp16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}

// Three colours of a neighbour's spin sp (u) and of the spin that G_mu brings to it (d).
struct Raw {
  int4 u[3], d[3];
};
// xo: component (3 sp, rhs) of site 0; the partner is `od` bytes from spin sp, colours `cl` bytes apart.
WD_DEV void fetch(Raw& w, const char* __restrict__ xo, unsigned nb, unsigned stride, i64 od, i64 cl) {
  const char* pu = xo + (u64)(nb & NB_MASK) * stride;
  const char* pd = pu + od;
#pragma unroll
  for (int col = 0; col < 3; ++col) {
    w.u[col] = __ldg(reinterpret_cast<const int4*>(pu));
    w.d[col] = __ldg(reinterpret_cast<const int4*>(pd));
    pu += cl;
    pd += cl;
  }
}

// v or -v for a mask m of 0 or -1, without the +1 of the negation (added by the caller as b = m & 1)
WD_DEV i64 flip(i64 v, i64 m) { return v ^ m; }

// v 2^k as FP64, v rounded once: its words become the doubles 2^84 + 2^63 + 2^32 hi and 2^52 + lo.
WD_DEV double fx_to(i64 v, int k) {
  const double dh = __hiloint2double(0x45300000, (int)(v >> 32) ^ 0x80000000);
  const double dl = __hiloint2double(0x43300000, (int)v);
  const double r = (dh - 0x1.00000801p84) + dl;     // 2^84 + 2^63 + 2^52
  const int rh = __double2hiint(r);
  return __hiloint2double(rh + (rh ? (k << 20) : 0), __double2loint(r));
}
// The same for scales at which the exponent field could leave the normal range.
static __device__ __noinline__ double fx_to_any(i64 v, int k) { return ldexp(fx_to(v, 0), k); }
// Both parts in units of 2^k, e the exponent that decides about the range.
WD_DEV double2 fx_out(i64 re, i64 im, int k, int e, bool finite) {
  if (e > 300 && e < 1800) return make_double2(fx_to(re, k), fx_to(im, k));
  if (finite) return make_double2(fx_to_any(re, k), fx_to_any(im, k));
  const double nan = __longlong_as_double(0x7FF8000000000000LL);
  return make_double2(nan, nan);
}

WD_DEV u64 absbits(i64 v) { return (u64)(v ^ (v >> 63)); }
WD_DEV int bit_len(u64 b) { return 64 - __clzll((i64)b); }

// The neighbours of a site with the shifts that align their fields to E, into nbs (one slot of TPB apart per
// direction; xe points at this right-hand side).  E is the largest of their exponents and e0, the site's own, unless
// `apart` finds e0 more than FX_APART above theirs: then the largest of theirs alone.
WD_DEV int neighbours_and_scale(const int4* __restrict__ nbt, const short* __restrict__ xe, int s, int L,
                                int e0, unsigned* nbs, bool* apart) {
  const int4 n0 = __ldg(nbt + 2 * (size_t)s), n1 = __ldg(nbt + 2 * (size_t)s + 1);
  const int nn[8] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w};
  int e[8], E = 0;
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    e[d] = __ldg(xe + (size_t)nn[d] * L);
    E = max(E, e[d]);
  }
  if (apart) *apart = e0 > E + FX_APART && e0 < FX_NONFINITE;
  if (!apart || !*apart) E = max(E, e0);
#pragma unroll
  for (int d = 0; d < 8; ++d) nbs[d * TPB] = (unsigned)nn[d] | ((unsigned)min(E - e[d], 60) << 26);
  return E;
}
// The sums of this thread's chirality from the hops' sums: the even thread of a pair takes the upper
// chirality, so both threads' upper spins; the odd one the lower: for spin 2 its own through mu 0, 1 and
// the other's through mu 2, 3, for spin 3 the reverse.  acc: [2][6][TPB] lower sums through mu 0, 1 and
// mu 2, 3, overwritten by the odd thread; hs: components (spin, colour, re/im).  Begins with a barrier of
// the warp: the other thread's slots are read, and nothing before makes its last sums visible.
template <typename T>
WD_DEV void exchange(T (*acc)[6][TPB], const T au[6], int sp, T hs[12]) {
  const int t = threadIdx.x, o = t ^ 1;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const T a = acc[0][q][t], b = acc[1][q][t], c = acc[1][q][o], d = acc[0][q][o];
    hs[q] = sp ? a + c : au[q];
    hs[6 + q] = b + d;
  }
  __syncwarp();
  if (sp) {
#pragma unroll
    for (int q = 0; q < 6; ++q) acc[0][q][t] = au[q];
  }
  __syncwarp();
  if (!sp) {
#pragma unroll
    for (int q = 0; q < 6; ++q) hs[6 + q] = acc[0][q][o];
  }
  __syncwarp();
}

}  // namespace fx
