// The FP64 stencil Y = A X, R = B - A X and the FP64 Jacobi sweep in 64-bit fixed point on the integer
// pipes (arXiv:0907.3261, Eq. (1); the paper's method is FP64 throughout, Sec. 3.1).
//
// GB300's FP64 pipe issues two lanes per clock per SM, its 32x32+64 -> 64-bit integer multiply-add
// (IMAD.WIDE) about 29, so an FP64-accurate stencil is fastest in exact integers:
//   * a spinor field is kept as 24 integers below 2^58 per (site, right-hand side) with one common
//     exponent (5 more bits than an FP64 significand at the largest entry), each in two signed limbs
//     of 28 and 30 bits; the links and the site blocks as integers of 60 bits in two limbs, scaled
//     by one power of two per context (links, kappa folded in) or per site and chirality (blocks);
//   * a real product takes three IMAD.WIDE: the high limbs' product, and the two mixed ones in a
//     second accumulator 2^-30 lower.  The low limbs' product (below 2^-59 of the bound) is dropped.
//     A complex product takes three real ones (re = k1 - k3, im = k1 + k2 with k1 = hr (ar + ai),
//     k2 = ar (hi - hr), k3 = ai (hr + hi)): 9 IMAD.WIDE instead of 12;
//   * every sum is exact in its 64-bit accumulator.  The hops of a site are aligned to the largest
//     exponent among the eight neighbours and the site itself; each hop's sum is rounded once to
//     2^-59 of that scale (forward and backward hops with opposite ties, so the roundings have no
//     bias, which a Jacobi sweep would amplify), and the result is rounded to FP64 once.
//   * a site whose own spinor is more than 2^FX_APART above all its neighbours' (a point source) has its site
//     block applied in FP64 arithmetic and only the neighbours aligned: its small components would otherwise be
//     held to 2^-59 of its largest, where their hopping sums are much finer.
// Bounds: a field's integers are at most 2^28 in high limbs, so |h| <= 2^29 and |hr +- hi| <= 2^30;
// link rows have norm <= 1 (checked at creation), so a hop's sums stay below 2^62 and the eight hops'
// total, in units of 2^FX_UP, below 2^62.3; a block's sum, shifted left by at most FX_CS, and a sweep's
// right-hand side in these units are below 2^61.  A block's row sum is below 2^30 in high limbs.
//
// Two threads share one (site, right-hand side): each projects and transports one of the two upper
// spins, and then applies one chirality block.  This halves the registers of a thread (128: 16 warps
// per SM) and doubles the parallelism of small lattices.  The links and blocks of the sites of a CTA are
// copied to shared memory with cp.async while the exponents are read; the next hop's six spinor
// components are loaded while the current one is summed.
//
// Measured on a GB300, Y = A X with the copy of X into the field form, 16^3x32, L = 12: 0.72 ms (0.10 of
// it the copy; 0.71 without the sites apart), against 1.51 ms for the same product in exact FP32 sums on
// fixed grids and 3.09 ms on the FP64 pipe; 4^4, L = 1: 17 us against 61 us (a thread's serial chain is a quarter as long); 32^3x64,
// L = 12: 11.3 against 23.4 ms; j = 12 FP64 sweeps on 8^3x16, L = 12: 0.57 against 1.63 ms.  Error
// against quad precision (4^4, Gaussian X): 0.80e-16 of |A X|, against 1.56e-16 in exact FP32 sums with
// FP64 site blocks; 12 sweeps 2.0e-16 against 2.7e-16.  Bound by the multiplier pipe (about 72% of its
// slots, at 4.3 cycles per IMAD.WIDE and 2 per other integer operation on it; DRAM 10% of peak).
// Variants measured at 16^3x32, L = 12: one thread per pair (168 registers) 1.11 ms; complex products of
// four real ones 0.78; hops unrolled in all eight directions (instruction fetch) 1.10; 96 registers and
// 20 warps 0.78.  Two-operand integer additions compile to multiplier-pipe operations; with a third
// operand that is zero at run time (z0) they take the other integer pipe: 0.79 to 0.72 ms.
#include <cmath>

#include "fixed.cuh"
#include "internal.h"

namespace {

using namespace fx;

enum { MODE_APPLY = 0, MODE_RESID = 1, MODE_JACOBI = 2 };

constexpr int FX_S = 30;                   // bits of a low limb
constexpr int FX_HI = 28;                  // bits of a field's high limb
constexpr int FX_OP = 30;                  // bits of an operator entry's high limb
constexpr int FX_UP = 1;                   // a hop's sum is kept in units of 2^FX_UP
constexpr int FX_CS = 3;                   // largest left shift of a site block's sum
constexpr int FX_BIAS = 1022 + FX_HI;      // unit of a field's high limbs with exponent e: 2^(e - FX_BIAS)
// A real as two limbs, h 2^FX_S + l.  z is zero (see the header).
struct Lim {
  int h, l;
};
WD_DEV Lim add3(Lim a, Lim b, int z) { return {a.h + b.h + z, a.l + b.l + z}; }
WD_DEV Lim sub3(Lim a, Lim b, int z) { return {a.h - b.h + z, a.l - b.l + z}; }
// A spinor component as the three reals that a product takes: re, im - re, re + im.
struct Fac {
  Lim r, d, s;
};
WD_DEV Fac fac_of(Lim r, Lim i, int z) { return {r, sub3(i, r, z), add3(r, i, z)}; }
// An operator entry: re, im, re + im.
struct Ent {
  Lim r, i, s;
};
WD_DEV Ent ent_of(int4 a, int z) { return {{a.x, a.y}, {a.z, a.w}, add3({a.x, a.y}, {a.z, a.w}, z)}; }

// v in units of 2^(n - FX_S), rounded, as limbs; n in [FX_S, FX_S + 60].
WD_DEV Lim lim_of(i64 v, int n) {
  const i64 t = shr_s(v + (i64)((1ull << (n - FX_S)) >> 1), n - FX_S);
  const int h = (int)((t + (1ll << (FX_S - 1))) >> FX_S);
  return {h, (int)((unsigned)t - ((unsigned)h << FX_S))};
}
// The same for any n >= -FX_HI with |v| < 2^(n + FX_HI): what is left of v's bits moves up, so that
// a normalised field never loses a bit for a coarse unit (a sweep's losses would add up).
WD_DEV Lim lim_norm(i64 v, int n) {
  return lim_of((i64)((u64)v << max(FX_S - n, 0)), max(n, FX_S));
}
// v as limbs of a field with exponent E (v's exponent field at most E, E >= FX_EMIN), rounded.
WD_DEV Lim fx_of(double v, int E) {
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  // |v| = m 2^(ef - 1075) with a 53-bit m, in units of 2^(E - FX_BIAS - FX_S) and one bit to round
  int ef;
  const u64 m = mantissa(h, l, ef) << (FX_S + FX_BIAS - 1075 + 1);
  const u64 q = (shr_u(m, E - ef) + 1) >> 1;
  const i64 sg = (i64)(h >> 31);
  return lim_of(((i64)q ^ sg) - sg, FX_S);
}
// Sums of products: of the high limbs, and the mixed ones 2^-FX_S lower.
struct Sum {
  i64 h, m;
};
WD_DEV void mul(Sum& K, Lim a, Lim b) {      // the first product; the mixed sums start at half of 2^32
  K.h = (i64)a.h * b.h;
  K.m = (i64)a.h * b.l + (1ll << 31);
  mac(K.m, a.l, b.h);
}
WD_DEV void madd(Sum& K, Lim a, Lim b) {
  mac(K.h, a.h, b.h);
  mac(K.m, a.h, b.l);
  mac(K.m, a.l, b.h);
}
// K += a f: re = K[0] - K[2], im = K[0] + K[1]
WD_DEV void cmul3(Sum K[3], const Ent& a, const Fac& f) {
  mul(K[0], a.s, f.r);
  mul(K[1], a.r, f.d);
  mul(K[2], a.i, f.s);
}
WD_DEV void cmadd3(Sum K[3], const Ent& a, const Fac& f) {
  madd(K[0], a.s, f.r);
  madd(K[1], a.r, f.d);
  madd(K[2], a.i, f.s);
}
// The two parts plus c; the mixed sums enter in units of 4 of the high ones (2^32 / 2^FX_S), rounded.
WD_DEV void csum(const Sum K[3], i64 c, int z, i64& re, i64& im) {
  const int m1 = (int)(K[0].m >> 32), m2 = (int)(K[1].m >> 32), m3 = (int)(K[2].m >> 32);
  re = K[0].h - K[2].h + shl((i64)(m1 - m3 + z), 2) + c;
  im = K[0].h + K[1].h + shl((i64)(m1 + m2 + z), 2) + c;
}

// Operator tables are read from shared memory (staged) or through the read-only cache.
template <bool ST>
WD_DEV int4 ldt(const int4* p) {
  if constexpr (ST) return *p;
  else return __ldg(p);
}
// Two hops of one direction mu, forward then backward, for the upper spin of this thread:
// h = u +- s d (SW: +- s i d), au += W h, and the lower spin's sum takes s i Z (SW, the first of two
// contributions) or -s Z, Z the backward minus the forward hop.  m = 0 for s = 1, -1 for s = -1.
// nbs: this thread's slots of neighbour and shift, forward, backward, and the next direction's
// forward one; w holds the forward neighbour's components on entry and the next direction's on exit.
template <bool SW, bool ST>
WD_DEV void hop_pair(const char* __restrict__ xo, const unsigned* nbs, bool more, unsigned stride, int m,
                     i64 od, i64 cl, const int4* U, Raw& w, i64 au[6], i64* ad, int z0) {
  const int b = m & 1;
  i64 z[6];
#pragma unroll
  for (int dir = 0; dir < 2; ++dir) {         // 0 forward, 1 backward
    const int sh = (int)(nbs[dir * TPB] >> 26) + FX_UP;
    Fac f[3];
#pragma unroll
    for (int col = 0; col < 3; ++col) {
      const int4 u = w.u[col], d = w.d[col];
      // SW: s i d = (-s d.im, s d.re)
      const Lim dr = SW ? Lim{d.z, d.w} : Lim{d.x, d.y}, di = SW ? Lim{d.x, d.y} : Lim{d.z, d.w};
      const bool mr = SW ? dir == 0 : dir == 1, mi = dir == 1;
      const Lim hr = mr ? Lim{u.x - (dr.h ^ m) - b, u.y - (dr.l ^ m) - b}
                        : Lim{u.x + (dr.h ^ m) + b, u.y + (dr.l ^ m) + b};
      const Lim hi = mi ? Lim{u.z - (di.h ^ m) - b, u.w - (di.l ^ m) - b}
                        : Lim{u.z + (di.h ^ m) + b, u.w + (di.l ^ m) + b};
      f[col] = fac_of(hr, hi, z0);
    }
    if (dir == 0 || more) fetch(w, xo, nbs[(dir + 1) * TPB], stride, od, cl);
    // half a unit: ties go up for the backward hop, down for the forward one
    const i64 half = dir ? (i64)(1ull << (sh - 1)) : (i64)~(~0ull << (sh - 1));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Sum K[3];
      cmul3(K, ent_of(ldt<ST>(U + dir * 9 + a * 3), z0), f[0]);
      cmadd3(K, ent_of(ldt<ST>(U + dir * 9 + a * 3 + 1), z0), f[1]);
      cmadd3(K, ent_of(ldt<ST>(U + dir * 9 + a * 3 + 2), z0), f[2]);
      i64 wr, wi;
      csum(K, half, z0, wr, wi);
      wr = shr_s(wr, sh);
      wi = shr_s(wi, sh);
      au[2 * a] += wr;
      au[2 * a + 1] += wi;
      if (dir == 0) {
        z[2 * a] = wr;
        z[2 * a + 1] = wi;
      } else {
        const i64 zr = wr - z[2 * a], zi = wi - z[2 * a + 1];
        i64 *pr = ad + (2 * a) * TPB, *pi = ad + (2 * a + 1) * TPB;
        if constexpr (SW) {            // s i Z = (-s Z.im, s Z.re)
          *pr = (i64)0 - flip(zi, m) - b;
          *pi = flip(zr, m) + b;
        } else {
          *pr = (*pr - flip(zr, m)) - b;
          *pi = (*pi - flip(zi, m)) - b;
        }
      }
    }
  }
}

// One row of a chirality block (six entries at D) times v.
template <bool ST>
WD_DEV void block_row(const int4* D, const Fac v[6], i64& re, i64& im, int z0) {
  Sum K[3];
  cmul3(K, ent_of(ldt<ST>(D), z0), v[0]);
#pragma unroll
  for (int j = 1; j < 6; ++j) cmadd3(K, ent_of(ldt<ST>(D + j), z0), v[j]);
  csum(K, 0, z0, re, im);
}

// Six results of this thread (re, im at slots 2 i, 2 i + 1 of `acc`, units 2^(eu - FX_BIAS), their bits
// or-ed in ob) as a field: one exponent for the 24 reals of the pair of threads.
WD_DEV void store_field(const i64* acc, u64 ob, int eu, bool finite, bool live, int sp, int4* y, int L,
                        short* ye) {
  const int T = ob ? eu + bit_len(ob) : -FX_NONFINITE;
  const int top = max(T, __shfl_xor_sync(0xFFFFFFFFu, T, 1));
  const int n = min(max(top - FX_HI - eu, -FX_HI), FX_S + 60);
  if (!live) return;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const Lim a = lim_norm(acc[(2 * i) * TPB], n), c = lim_norm(acc[(2 * i + 1) * TPB], n);
    y[(size_t)i * L] = make_int4(a.h, a.l, c.h, c.l);
  }
  if (sp == 0) *ye = (short)(!finite ? FX_NONFINITE : top == -FX_NONFINITE ? FX_EMIN : eu + n);
}

// Row i of a packed Hermitian block times v in FP64 arithmetic: component j at v[j * step], its imaginary part `im`
// further on.
static __device__ __noinline__ double2 row_in_fp64(const double* b, const double* v, int step, int im, int i) {
  double2 q = make_double2(b[i] * v[i * step], b[i] * v[i * step + im]);
#pragma unroll 1
  for (int j = 0; j < 6; ++j) {
    if (j == i) continue;
    const int t = i > j ? tri_index(i, j) : tri_index(j, i);
    const double c = b[t], d = i > j ? b[t + 1] : -b[t + 1], x = v[j * step], y = v[j * step + im];
    q.x = fma(-d, y, fma(c, x, q.x));
    q.y = fma(d, x, fma(c, y, q.y));
  }
  return q;
}

// A product with A (APPLY: y = A x, RESID: y = u - A x) or a Jacobi sweep y = A_D^{-1}(u + kappa H x)
// of the field x (exponents xe); u FP64 (JACOBI: its exponents ue); y FP64, or a field (QOUT).  x64 (APPLY, RESID)
// is x itself, D64 the site blocks: where a site's own spinor is far above its neighbours', the common scale would
// lose its small components, and the site block is applied in FP64 arithmetic (not for a field, which has one scale).
// ST: the links and blocks of the CTA's sites are staged in shared memory.
template <int MODE, bool ST, bool QOUT>
__global__ void __launch_bounds__(TPB, 4)
fx_kernel(const int4* __restrict__ x, const short* __restrict__ xe, void* __restrict__ y,
          short* __restrict__ ye, const double2* __restrict__ u, const short* __restrict__ ue,
          const double* __restrict__ x64, const double* __restrict__ D64, const int4* __restrict__ W,
          const int4* __restrict__ D, const int4* __restrict__ nbt, int V, int L, int ek, int z0) {
  const unsigned npair = (unsigned)V * L;            // at most 2^30
  const unsigned p0 = blockIdx.x * (TPB / 2u), p1 = p0 + (threadIdx.x >> 1);
  const bool live = p1 < npair;
  const unsigned pair = live ? p1 : npair - 1;       // idle lanes follow the last pair
  const int sp = threadIdx.x & 1;
  const int s = (int)(pair / (unsigned)L);
  const int r = (int)(pair - (unsigned)s * L);
  extern __shared__ int4 stage[];
  int s0 = 0;
  const int4* sD = nullptr;
  if constexpr (ST) {       // the tables of this CTA's sites, contiguous in both
    s0 = (int)(p0 / (unsigned)L);
    const int ns = (int)(min(p0 + TPB / 2u - 1u, npair - 1u) / (unsigned)L) - s0 + 1;
    for (int i = threadIdx.x; i < ns * FX_WSTR; i += TPB) cp16(stage + i, W + (size_t)s0 * FX_WSTR + i);
    int4* const d = stage + ns * FX_WSTR;
    for (int i = threadIdx.x; i < ns * FX_DSTR; i += TPB) cp16(d + i, D + (size_t)s0 * FX_DSTR + i);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    sD = d;
  }
  // Per thread: neighbours with their shifts, and the lower spins' sums through mu 0, 1 and mu 2, 3
  // (later this chirality's sums, or results).
  __shared__ unsigned nbs[8][TPB];
  __shared__ i64 acc[2][6][TPB];
  const int t = threadIdx.x;
  const int eo = __ldg((MODE == MODE_JACOBI ? ue : xe) + (size_t)s * L + r);
  bool apart;
  const int E = neighbours_and_scale(nbt, xe + r, s, L, eo, &nbs[0][t], QOUT ? nullptr : &apart);
  const bool finite = E < FX_NONFINITE;
  const char* xo = reinterpret_cast<const char*>(x + (size_t)(3 * sp) * L + r);
  const unsigned stride = 192u * (unsigned)L;        // bytes per site
  const i64 cl = 16LL * L;
  const int4* U = ST ? stage + (s - s0) * FX_WSTR : W + (size_t)s * FX_WSTR;
  i64 au[6] = {0, 0, 0, 0, 0, 0};                    // the upper spin's sums
  Raw w;
  fetch(w, xo, nbs[0][t], stride, (9 - 6 * sp) * cl, cl);
  if constexpr (ST) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
  }
  // mu 0, 1 bring spin 3 - sp, mu 2, 3 spin 2 + sp to spin sp, with the signs of G_mu: mu 0 -i, -i;
  // mu 1 -1, +1; mu 2 -i, +i; mu 3 +1, +1 for sp = 0, 1.
#pragma unroll 1
  for (int hf = 0; hf < 2; ++hf) {
    const unsigned* nb = &nbs[4 * hf][t];
    const i64 od = (hf ? 6 : 9 - 6 * sp) * cl;
    i64* ad = &acc[hf][0][t];
    hop_pair<true, ST>(xo, nb, true, stride, -(hf & sp), od, cl, U, w, au, ad, z0);
    hop_pair<false, ST>(xo, nb + 2 * TPB, hf == 0, stride, hf ? -1 : -sp, od, cl, U + 18, w, au, ad, z0);
    U += 36;
    if (hf == 0) {
      // the last fetch took another partner spin: mu 2's
      const char* p = xo + (u64)(nb[4 * TPB] & NB_MASK) * stride + 6 * cl;
#pragma unroll
      for (int col = 0; col < 3; ++col) w.d[col] = __ldg(reinterpret_cast<const int4*>(p + col * cl));
    }
  }
  i64 hs[12];
  exchange(acc, au, sp, hs);
  const size_t base = (size_t)s * 12 * L + (size_t)(6 * sp) * L + r;
  const int4* Dc = ST ? sD + (s - s0) * FX_DSTR : D + (size_t)s * FX_DSTR;
  const int4 de = ldt<ST>(Dc + 72);
  const int eD = sp ? de.y : de.x;
  Dc += 36 * sp;
  const int eh = E + ek - FX_OP + FX_UP;       // the hopping sums' unit: 2^(eh - FX_BIAS)
  Fac v[6];
  if constexpr (MODE != MODE_JACOBI) {
    const int so = apart ? 0 : min(E - eo, 60);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const int4 a = __ldg(x + base + (size_t)i * L);
      v[i] = fac_of(lim_of(shl(a.x, FX_S) + a.y, FX_S + so), lim_of(shl(a.z, FX_S) + a.w, FX_S + so), z0);
    }
    // the site block's unit is 2^cs of the hopping sums'; with a large block these are shifted instead
    const int cs = eD - ek - FX_UP, cl_ = min(cs, FX_CS), cr = cs - cl_;
    const int e = eh + cr;
    i64* const slot = &acc[0][0][t];
#pragma unroll
    for (int q = 0; q < 12; ++q) slot[q * TPB] = hs[q];
#pragma unroll 1
    for (int i = 0; i < 6; ++i) {
      i64 re, im;
      block_row<ST>(Dc + 6 * i, v, re, im, z0);
      i64 hr = slot[(2 * i) * TPB], hi = slot[(2 * i + 1) * TPB];
      if (cr) {
        const int c = min(cr, 61);
        hr = shr_s(hr + (i64)((1ull << c) >> 1), c);
        hi = shr_s(hi + (i64)((1ull << c) >> 1), c);
      }
      if (!live) continue;
      double2 q;
      if (apart) {
        q = row_in_fp64(D64 + ((size_t)s * 2 + sp) * CLOV_REALS, x64 + 2 * base, 2 * L, 1, i);
        const double2 h = fx_out(slot[(2 * i) * TPB], slot[(2 * i + 1) * TPB], eh - FX_BIAS, eh, finite);
        q.x -= h.x;
        q.y -= h.y;
      } else {
        q = fx_out(shl(re, cl_) - hr, shl(im, cl_) - hi, e - FX_BIAS, e, finite);
      }
      if constexpr (MODE == MODE_RESID) {
        const double2 b = __ldg(u + base + (size_t)i * L);
        q.x = b.x - q.x;
        q.y = b.y - q.y;
      }
      reinterpret_cast<double2*>(y)[base + (size_t)i * L] = q;
    }
  } else {
    if constexpr (!QOUT) {
      if (apart) {
        double* const v64 = reinterpret_cast<double*>(&acc[0][0][t]);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const double2 a = __ldg(u + base + (size_t)i * L);
          const double2 h = fx_out(hs[2 * i], hs[2 * i + 1], eh - FX_BIAS, eh, finite);
          v64[(2 * i) * TPB] = a.x + h.x;
          v64[(2 * i + 1) * TPB] = a.y + h.y;
        }
      }
    }
    // v = u + kappa H x in the hopping sums' units: |u| = m 2^(ef - 1075), m shifted left by 10
    u64 bits = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const double2 a = __ldg(u + base + (size_t)i * L);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const double tv = q ? a.y : a.x;
        const int h = __double2hiint(tv);
        int ef;
        const u64 m = mantissa(h, (unsigned)__double2loint(tv), ef) << 10;
        const i64 uq = (i64)shr_u(m, eh - ef + (10 + 1075 - FX_BIAS));
        const i64 sg = (i64)(h >> 31);
        hs[2 * i + q] += (uq ^ sg) - sg;
        bits |= absbits(hs[2 * i + q]);
      }
    }
    bits |= (u64)__shfl_xor_sync(0xFFFFFFFFu, bits, 1);
    const int n1 = bit_len(bits) - FX_HI;
#pragma unroll
    for (int i = 0; i < 6; ++i) v[i] = fac_of(lim_norm(hs[2 * i], n1), lim_norm(hs[2 * i + 1], n1), z0);
    const int eu = eh + n1 + eD - FX_OP;       // the results' unit: 2^(eu - FX_BIAS)
    u64 ob = 0;
#pragma unroll 1
    for (int i = 0; i < 6; ++i) {
      i64 re, im;
      block_row<ST>(Dc + 6 * i, v, re, im, z0);
      if constexpr (QOUT) {
        ob |= absbits(re) | absbits(im);
        (&acc[0][0][t])[(2 * i) * TPB] = re;
        (&acc[0][0][t])[(2 * i + 1) * TPB] = im;
      } else if (live) {
        reinterpret_cast<double2*>(y)[base + (size_t)i * L] =
            apart ? row_in_fp64(D64 + ((size_t)s * 2 + sp) * CLOV_REALS, reinterpret_cast<double*>(&acc[0][0][t]),
                                2 * TPB, TPB, i)
                  : fx_out(re, im, eu - FX_BIAS, eu, finite);
      }
    }
    if constexpr (QOUT)
      store_field(&acc[0][0][t], ob, eu, finite, live, sp, reinterpret_cast<int4*>(y) + base, L,
                  ye + (size_t)s * L + r);
  }
}

// The first sweep from G = 0, y = A_D^{-1} u as a field, and u's exponents; two threads per (site, rhs).
__global__ void __launch_bounds__(TPB)
fx_first_kernel(const double2* __restrict__ u, short* __restrict__ ue, int4* __restrict__ y,
                short* __restrict__ ye, const int4* __restrict__ D, int V, int L, int z0) {
  const unsigned npair = (unsigned)V * L;
  const unsigned p1 = blockIdx.x * (TPB / 2u) + (threadIdx.x >> 1);
  const bool live = p1 < npair;
  const unsigned pair = live ? p1 : npair - 1;
  const int sp = threadIdx.x & 1;
  const int s = (int)(pair / (unsigned)L);
  const int r = (int)(pair - (unsigned)s * L);
  __shared__ i64 acc[12][TPB];
  const size_t base = (size_t)s * 12 * L + (size_t)(6 * sp) * L + r;
  double2 a[6];
  int e = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    a[i] = __ldg(u + base + (size_t)i * L);
    e = max(e, exponent_of(a[i]));
  }
  e = max(e, __shfl_xor_sync(0xFFFFFFFFu, e, 1));
  const short fe = field_exponent(e);
  const int E = fe;
  Fac v[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) v[i] = fac_of(fx_of(a[i].x, E), fx_of(a[i].y, E), z0);
  const int4* Dc = D + (size_t)s * FX_DSTR;
  const int4 de = __ldg(Dc + 72);
  const int eu = E + (sp ? de.y : de.x) - FX_OP;
  u64 ob = 0;
#pragma unroll 1
  for (int i = 0; i < 6; ++i) {
    i64 re, im;
    block_row<false>(Dc + 36 * sp + 6 * i, v, re, im, z0);
    ob |= absbits(re) | absbits(im);
    acc[2 * i][threadIdx.x] = re;
    acc[2 * i + 1][threadIdx.x] = im;
  }
  if (live && sp == 0) ue[(size_t)s * L + r] = fe;
  store_field(&acc[0][threadIdx.x], ob, eu, fe < FX_NONFINITE, live, sp, y + base, L, ye + (size_t)s * L + r);
}

// The field form of an FP64 block.
__global__ void __launch_bounds__(128)
fx_split_kernel(const double2* __restrict__ x, int4* __restrict__ q, short* __restrict__ xe, int V, int L) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= V * L) return;
  const int s = tid / L;
  const int r = tid - s * L;
  const size_t base = (size_t)s * 12 * L + r;
  double2 v[12];
  int e = 0;
#pragma unroll
  for (int i = 0; i < 12; ++i) {
    v[i] = __ldg(x + base + (size_t)i * L);
    e = max(e, exponent_of(v[i]));
  }
  const short fe = field_exponent(e);
  xe[tid] = fe;
#pragma unroll
  for (int i = 0; i < 12; ++i) {
    const Lim a = fx_of(v[i].x, fe), b = fx_of(v[i].y, fe);
    q[base + (size_t)i * L] = make_int4(a.h, a.l, b.h, b.l);
  }
}

// ------------------------------------------------------------------ tables (at creation)
__global__ void fx_neighbours_kernel(int* __restrict__ out, Geom g) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  int c[4];
  site_coords(g, s, c);
  for (int d = 0; d < 8; ++d) out[8 * (size_t)s + d] = neighbour(g, s, c, d >> 1, (d & 1) ? -1 : 1);
}

// m 2^-n rounded, with v's sign, as limbs.
WD_DEV Lim signed_limbs(u64 m, int n, double v) {
  u64 q;
  if (n > 0) q = (shr_u(m, n - 1) + 1) >> 1;
  else q = m << -n;
  return lim_of(__double2hiint(v) < 0 ? -(i64)q : (i64)q, FX_S);
}
// v 2^sc rounded (below 2^60), and kappa v 2^sc rounded, from integer products (no FP64 pipe).
WD_DEV Lim limbs(double v, int sc) {
  int ef;
  const u64 m = mantissa(__double2hiint(v), (unsigned)__double2loint(v), ef);
  return m ? signed_limbs(m, 1075 - ef - sc, v) : Lim{0, 0};
}
WD_DEV Lim limbs_kappa(double v, double kappa, int sc) {
  int ef, ek;
  const u64 m = mantissa(__double2hiint(v), (unsigned)__double2loint(v), ef);
  const u64 mk = mantissa(__double2hiint(kappa), (unsigned)__double2loint(kappa), ek);
  const u64 hi = __umul64hi(m << 11, mk << 11);          // |kappa v| = hi 2^(42 + ef + ek - 2150)
  const Lim a = hi ? signed_limbs(hi, 2150 - 42 - ef - ek - sc, v) : Lim{0, 0};
  return __double2hiint(kappa) < 0 ? lim_of(-(shl(a.h, FX_S) + a.l), FX_S) : a;
}

// kappa W for the eight directions of every site (W = U_mu(s) forward, U_mu(s - mu)^H backward), row by
// row, scaled by 2^(FX_OP - ek).
__global__ void fx_links_kernel(const double* __restrict__ links, int4* __restrict__ out,
                                const int* __restrict__ nbt, int V, double kappa, int ek) {
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= (long long)V * FX_WSTR) return;
  const int s = (int)(tid / FX_WSTR), rem = (int)(tid - (long long)s * FX_WSTR);
  const int d = rem / 9, e = rem - d * 9, mu = d >> 1;
  const bool fwd = (d & 1) == 0;
  const int sl = fwd ? s : __ldg(nbt + 8 * (size_t)s + d);
  const int ee = fwd ? e : (e % 3) * 3 + e / 3;
  const double2 p = __ldg(reinterpret_cast<const double2*>(links) + ((size_t)sl * 4 + mu) * 9 + ee);
  const int sc = FX_OP + FX_S - ek;
  const Lim a = limbs_kappa(p.x, kappa, sc), b = limbs_kappa(fwd ? p.y : -p.y, kappa, sc);
  out[tid] = make_int4(a.h, a.l, b.h, b.l);
}

// Site blocks: all six entries of every row, both chiralities, then the two exponents.  A block is
// scaled by 2^(FX_OP - e), e the exponent of its largest row sum and at least emin.  BK_SITES sites per CTA,
// one entry per thread at a time, so that the packed blocks are read and the tables written in order: 3.0 ms
// for both tables at 32^3x64 against 9.7 with a thread per block; wd_create 70.8 ms against 77.5 (16^3x32:
// 4.85 against 5.20).
constexpr int BK_SITES = 8, BK_TPB = 256;
__global__ void __launch_bounds__(BK_TPB)
fx_blocks_kernel(const double* __restrict__ cl, int4* __restrict__ out, int V, int emin) {
  __shared__ double b[2 * BK_SITES][CLOV_REALS], sums[2 * BK_SITES][6];
  __shared__ int ex[2 * BK_SITES];
  const int s0 = blockIdx.x * BK_SITES, ns = min(BK_SITES, V - s0), t = threadIdx.x;
  for (int e = t; e < 2 * ns * CLOV_REALS; e += BK_TPB) b[0][e] = cl[(size_t)s0 * 2 * CLOV_REALS + e];
  __syncthreads();
  if (t < 2 * ns * 6) {
    const int k = t / 6, i = t - 6 * k;
    double sum = fabs(b[k][i]);
    for (int j = 0; j < 6; ++j) {
      if (j == i) continue;
      const int q = i > j ? tri_index(i, j) : tri_index(j, i);
      sum += fabs(b[k][q]) + fabs(b[k][q + 1]);
    }
    sums[k][i] = sum;
  }
  __syncthreads();
  if (t < 2 * ns) {
    double worst = 0.0;
    for (int i = 0; i < 6; ++i) worst = fmax(worst, sums[t][i]);
    ex[t] = max(worst > 0.0 ? ilogb(worst) + 1 : emin, emin);
  }
  __syncthreads();
  for (int e = t; e < ns * FX_DSTR; e += BK_TPB) {
    const int s = e / FX_DSTR, q = e - s * FX_DSTR;
    int4 v = make_int4(ex[2 * s], ex[2 * s + 1], 0, 0);
    if (q < 72) {
      const int k = 2 * s + q / 36, i = q % 36 / 6, j = q % 6, sc = FX_OP + FX_S - ex[k];
      if (i == j) {
        const Lim p = limbs(b[k][i], sc);
        v = make_int4(p.h, p.l, 0, 0);
      } else {
        const int x = i > j ? tri_index(i, j) : tri_index(j, i);
        const Lim re = limbs(b[k][x], sc), im = limbs(i > j ? b[k][x + 1] : -b[k][x + 1], sc);
        v = make_int4(re.h, re.l, im.h, im.l);
      }
    }
    out[(size_t)s0 * FX_DSTR + e] = v;
  }
}

inline unsigned grid_of(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// Staging pays where a CTA's 64 pairs cover few sites (2.3 KB each, beside 23 KB of other shared
// memory): 8 CTA-sites or so leave four CTAs per SM, 23 (L = 3) two, 64 (L = 1) one.  Staged against read
// through L1, 8x16^3: L = 1 51 against 36 us, L = 2 65 / 56, L = 3 75 / 75, L = 4 82 / 90, L = 8 132 / 158,
// L = 16 250 / 293; 8^4: L = 3 20.7 / 22.0, L = 12 35.5 / 37.6.
constexpr int FX_STAGE_L = 3;

template <int MODE, bool QOUT>
cudaError_t launch_fx(const Op& op, const int4* x, const short* xe, void* y, short* ye, const double* u,
                      const short* ue, const double* x64, const int4* D, int L, cudaStream_t st) {
  const unsigned grid = grid_of(2LL * op.g.V * L, TPB);
  const double2* u2 = reinterpret_cast<const double2*>(u);
  const double* D64 = MODE == MODE_JACOBI ? op.clov_inv : op.clov;
  if (L >= FX_STAGE_L) {
    const int bytes = ((TPB / 2 - 1) / L + 2) * (FX_WSTR + FX_DSTR) * (int)sizeof(int4);
    cudaError_t e = cudaFuncSetAttribute(fx_kernel<MODE, true, QOUT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    fx_kernel<MODE, true, QOUT><<<grid, TPB, bytes, st>>>(x, xe, y, ye, u2, ue, x64, D64, op.fx_links, D,
                                                          op.fx_nb, op.g.V, L, op.fx_ek, 0);
  } else {
    fx_kernel<MODE, false, QOUT><<<grid, TPB, 0, st>>>(x, xe, y, ye, u2, ue, x64, D64, op.fx_links, D,
                                                       op.fx_nb, op.g.V, L, op.fx_ek, 0);
  }
  return cudaGetLastError();
}

cudaError_t split(const Op& op, const double* x, int4* q, short* e, int L, cudaStream_t st) {
  fx_split_kernel<<<grid_of((long long)op.g.V * L, 128), 128, 0, st>>>(reinterpret_cast<const double2*>(x), q,
                                                                      e, op.g.V, L);
  return cudaGetLastError();
}

}  // namespace

int fx_link_exponent(double kappa) {
  if (kappa == 0.0) return FX_EK;
  int e;
  std::frexp(std::fabs(kappa), &e);          // |kappa| < 2^e
  return e < FX_EK ? FX_EK : e;
}

cudaError_t launch_fx_tables(const Op& op, cudaStream_t st) {
  fx_neighbours_kernel<<<grid_of(op.g.V, 256), 256, 0, st>>>(reinterpret_cast<int*>(op.fx_nb), op.g);
  fx_links_kernel<<<grid_of((long long)op.g.V * FX_WSTR, 256), 256, 0, st>>>(
      op.links, op.fx_links, reinterpret_cast<const int*>(op.fx_nb), op.g.V, op.kappa, op.fx_ek);
  fx_blocks_kernel<<<grid_of(op.g.V, BK_SITES), BK_TPB, 0, st>>>(op.clov, op.fx_clov, op.g.V, op.fx_ek + FX_UP);
  fx_blocks_kernel<<<grid_of(op.g.V, BK_SITES), BK_TPB, 0, st>>>(op.clov_inv, op.fx_cinv, op.g.V, -1000);
  return cudaGetLastError();
}

cudaError_t launch_apply_fx(const Op& op, const double* x, double* y, void* q, int L, cudaStream_t st) {
  const cudaError_t e = split(op, x, static_cast<int4*>(q), op.fx_exp(0), L, st);
  if (e != cudaSuccess) return e;
  return launch_fx<MODE_APPLY, false>(op, static_cast<const int4*>(q), op.fx_exp(0), y, nullptr, nullptr,
                                      nullptr, x, op.fx_clov, L, st);
}

cudaError_t launch_resid_fx(const Op& op, const double* x, const double* b, double* y, void* q, int L,
                            cudaStream_t st) {
  const cudaError_t e = split(op, x, static_cast<int4*>(q), op.fx_exp(0), L, st);
  if (e != cudaSuccess) return e;
  return launch_fx<MODE_RESID, false>(op, static_cast<const int4*>(q), op.fx_exp(0), y, nullptr, b, nullptr, x,
                                      op.fx_clov, L, st);
}

cudaError_t launch_first_fx(const Op& op, const double* u, void* q_out, int slot, int L, cudaStream_t st) {
  fx_first_kernel<<<grid_of(2LL * op.g.V * L, TPB), TPB, 0, st>>>(
      reinterpret_cast<const double2*>(u), op.fx_exp(2), static_cast<int4*>(q_out), op.fx_exp(slot),
      op.fx_cinv, op.g.V, L, 0);
  return cudaGetLastError();
}

cudaError_t launch_sweep_fx(const Op& op, const void* q_in, int slot, const double* u, void* q_out,
                            double* g64, int L, cudaStream_t st) {
  const int4* x = static_cast<const int4*>(q_in);
  if (q_out)
    return launch_fx<MODE_JACOBI, true>(op, x, op.fx_exp(slot), q_out, op.fx_exp(1 - slot), u, op.fx_exp(2),
                                        nullptr, op.fx_cinv, L, st);
  return launch_fx<MODE_JACOBI, false>(op, x, op.fx_exp(slot), g64, nullptr, u, op.fx_exp(2), nullptr,
                                       op.fx_cinv, L, st);
}
