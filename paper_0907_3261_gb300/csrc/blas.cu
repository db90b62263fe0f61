// Tall-skinny block operations of preconditioned block BiCGGR (arXiv:0907.3261, Sec. 2, the
// algorithm box): the L x L Gram products R~_0^H V and R~_0^H R, the traces Tr[W^H R] and
// Tr[W^H W] that give zeta_k, the column norms of the stopping test, the L x L solves for alpha_k
// and gamma_k, and the block updates
//   U = (P - zeta V) alpha,  X += zeta F + G,  R -= zeta W + Y,  P = R + U gamma,  V = W + Y gamma.
//
// The updates and the Gram products are in blas_digits.cu; here are the traces, the norms, the L x L solves
// and the sums over blocks.
//
// A block is N rows of L complex numbers (row n at n*L).  Every kernel walks rows in chunks with a fixed
// chunk -> block assignment (block b takes chunks b, b + grid, ...) and accumulates its share of the
// reductions in a fixed order.  Each block writes its partial sums to a slot of `part`; a finalize kernel adds
// the slots in a fixed order.  Results are therefore bitwise reproducible from run to run (no float
// atomics).
#include "common.cuh"
#include "internal.h"

namespace {

constexpr int TS_THREADS = 256;
constexpr int CH = 32;                     // rows per chunk

WD_DEV Cx<double> ld2(const double* p, size_t e) {
  double2 v = *reinterpret_cast<const double2*>(p + 2 * e);
  return {v.x, v.y};
}
WD_DEV Cx<double> sm(const double2& v) { return {v.x, v.y}; }
WD_DEV double2 d2(Cx<double> a) { return make_double2(a.re, a.im); }

// Column norms ||A_col||^2 only.
__global__ void __launch_bounds__(TS_THREADS)
colnorm_kernel(const double* __restrict__ A, int L, long long rows, double2* __restrict__ part) {
  __shared__ double red[TS_THREADS];
  // thread t handles column t % L of rows strided by (TS_THREADS / L) within a chunk
  const int per = TS_THREADS / L;
  const int col = threadIdx.x % L, lane_row = threadIdx.x / L;
  double acc = 0.0;
  if (lane_row < per) {
    const long long nchunks = (rows + CH - 1) / CH;
    for (long long ck = blockIdx.x; ck < nchunks; ck += gridDim.x) {
      const long long r0 = ck * CH;
      const int nr = (int)min((long long)CH, rows - r0);
      for (int n = lane_row; n < nr; n += per) acc += cnorm2(ld2(A, (size_t)(r0 + n) * L + col));
    }
  }
  red[threadIdx.x] = (lane_row < per) ? acc : 0.0;
  __syncthreads();
  if (threadIdx.x < L) {
    double s = 0.0;
    for (int k = 0; k < per; ++k) s += red[k * L + threadIdx.x];
    part[(size_t)blockIdx.x * PART_STRIDE + WD_LMAX * WD_LMAX + threadIdx.x] = make_double2(s, 0.0);
  }
}

// Tr[W^H R] and Tr[W^H W] over all N*L entries.
__global__ void __launch_bounds__(TS_THREADS)
trace_kernel(const double* __restrict__ W, const double* __restrict__ R, long long count,
             double2* __restrict__ part) {
  __shared__ double red[3][TS_THREADS];
  Cx<double> wr = czero<double>();
  double ww = 0.0;
  const long long per_block = (long long)CH * WD_LMAX;
  const long long nchunks = (count + per_block - 1) / per_block;
  for (long long ck = blockIdx.x; ck < nchunks; ck += gridDim.x) {
    const long long e0 = ck * per_block;
    const long long e1 = min(count, e0 + per_block);
    for (long long e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
      const Cx<double> w = ld2(W, e), r = ld2(R, e);
      wr = cfmaj(w, r, wr);
      ww += cnorm2(w);
    }
  }
  red[0][threadIdx.x] = wr.re;
  red[1][threadIdx.x] = wr.im;
  red[2][threadIdx.x] = ww;
  __syncthreads();
  for (int off = TS_THREADS / 2; off > 0; off >>= 1) {
    if (threadIdx.x < off)
      for (int q = 0; q < 3; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    double2* p = part + (size_t)blockIdx.x * PART_STRIDE;
    p[0] = make_double2(red[0][0], red[1][0]);
    p[1] = make_double2(red[2][0], 0.0);
  }
}

// Sums the per-block partials: FIN_COLS of their numbers per block, FIN_ROWS threads on each, thread k on
// the slots k, k + FIN_ROWS, ...; the threads' sums are added in order.  which: GRAM_* target, -1 none;
// norms_out: where the column norms go (may be null); traces: Tr[W^H R], Tr[W^H W] instead.
// A chain of loads, so bound by latency: 608 slots, L = 12: 16 us, against about 110 us with one thread
// per number in one block.
constexpr int FIN_COLS = 16, FIN_ROWS = 16;

__global__ void __launch_bounds__(FIN_COLS* FIN_ROWS)
finalize_kernel(const double2* __restrict__ part, int nblocks, int L, SolverState* st, int which,
                double* norms_out, bool traces) {
  __shared__ double2 red[FIN_ROWS][FIN_COLS];
  const int col = threadIdx.x % FIN_COLS, k = threadIdx.x / FIN_COLS;
  const int n = traces ? 2 : which >= 0 ? L * L : 0;
  const int nb = (n + FIN_COLS - 1) / FIN_COLS;
  const bool norms = (int)blockIdx.x >= nb;
  const int t = norms ? col : blockIdx.x * FIN_COLS + col;
  const bool live = t < (norms ? L : n);
  double2 s = make_double2(0.0, 0.0);
  if (live) {
    const double2* p = part + (norms ? WD_LMAX * WD_LMAX : 0) + t;
#pragma unroll 8
    for (int b = k; b < nblocks; b += FIN_ROWS) {
      const double2 v = p[(size_t)b * PART_STRIDE];
      s.x += v.x;
      s.y += v.y;
    }
  }
  red[k][col] = s;
  __syncthreads();
  if (k || !live) return;
#pragma unroll
  for (int q = 1; q < FIN_ROWS; ++q) {
    s.x += red[q][col].x;
    s.y += red[q][col].y;
  }
  if (norms) norms_out[t] = s.x;
  else if (traces && t) st->trww = s.x;
  else (traces ? &st->trwr : which == GRAM_RTR ? st->rtr : which == GRAM_RTR_NEW ? st->rtr_new : st->rtv)[t] = s;
}

void finalize(const double2* part, int nblocks, int L, SolverState* st, int which, double* norms_out,
              bool traces, cudaStream_t s) {
  const int n = traces ? 2 : which >= 0 ? L * L : 0;
  const int grid = (n + FIN_COLS - 1) / FIN_COLS + (norms_out ? 1 : 0);
  finalize_kernel<<<grid, FIN_COLS * FIN_ROWS, 0, s>>>(part, nblocks, L, st, which, norms_out, traces);
}

// ---------------------------------------------------------------- L x L solves (one block)
// Solves C Z = Rhs by elimination with partial pivoting (largest modulus) and back substitution.  Thread
// e < 2 L^2 holds element (i, j) = (e % L, e / L) of [C | Rhs]; rows are not moved, a row's place in the pivots'
// order is kept instead.  A warp's FP64 instruction takes 64 cycles of its quarter of the SM whatever its
// lanes do, so the count per warp is what bounds the solve: elements are dense in the warps, moduli are
// compared as integers, and the column's owners alone form the pivot's reciprocal and the factors.  27 us at
// L = 12 and 8 at L = 4, against about 75 and 18 in one warp with a column per lane; an iteration of a 4^4,
// L = 12 solve 256 us against 353.
//
// The system is singular in the sense of the oracle when a pivot is not finite or its modulus is below
// 1e-13 times the largest pivot's.
constexpr double PIVOT_RTOL2 = 1e-26;      // squared moduli are compared

struct Lu {
  double2 u[WD_LMAX][2 * WD_LMAX];         // the pivot rows, in their order
  double2 c[WD_LMAX], f[WD_LMAX];          // a column, its factors
  double2 rp[WD_LMAX];                     // the pivots' reciprocals
  double2 x[WD_LMAX];                      // a row of the solution
  long long norm[WD_LMAX];                 // bits of the squared moduli, -1 for rows that have been pivots
  double pn[WD_LMAX];
  double2 extra;                           // a number that the block's last warp computes beside
};

// conj(c) / n for n = |c|^2.  Where 1 / n would leave the normal range (block norms around 1e-77) the parts are
// divided one by one; else one reciprocal serves both.
WD_DEV double2 reciprocal(double2 c, double n) {
  if (n > 0x1p-1000 && n < 0x1p1000) {
    const double r = 1.0 / n;
    return make_double2(c.x * r, -c.y * r);
  }
  return make_double2(c.x / n, -c.y / n);
}

inline int lu_threads(int L) { return (2 * L * L + 31) / 32 * 32 + 32; }

// m: this thread's element (i, j).  On return `order` is row i's place and, for j >= L, m the solution's element
// (order, j - L).  The same in every thread: true when the system is singular (`order` may then be L).
__device__ bool lu_solve(Lu& s, Cx<double>& m, int L, int i, int j, bool live, int& order) {
  order = L;                               // not yet a pivot
  for (int k = 0; k < L; ++k) {
    if (live && j == k) {
      s.c[i] = d2(m);
      s.norm[i] = order < L ? -1 : __double_as_longlong(cnorm2(m));
    }
    __syncthreads();
    int p = 0;
    long long best = -2;
    for (int q = 0; q < L; ++q) {
      const long long v = s.norm[q];
      if (v > best) {
        best = v;
        p = q;
      }
    }
    const bool mine = live && i == p;
    if (mine) {
      order = k;
      s.u[k][j] = d2(m);
    }
    if (live && j == k) {
      const double pn = __longlong_as_double(best);
      const double2 rp = reciprocal(s.c[p], pn);
      if (mine) {
        s.rp[k] = rp;
        s.pn[k] = pn;
      }
      s.f[i] = d2(cmul(m, sm(rp)));            // the factor of row i (of no use in the pivot's)
    }
    __syncthreads();
    if (live && order == L && j > k) {
      const double2 f = s.f[i], u = s.u[k][j];
      m.re = fma(f.y, u.y, fma(-f.x, u.x, m.re));
      m.im = fma(-f.y, u.x, fma(-f.x, u.y, m.im));
    }
  }
  long long lo = 0x7FFFFFFFFFFFFFFFll, hi = 0;
  for (int k = 0; k < L; ++k) {
    const long long v = __double_as_longlong(s.pn[k]);
    lo = min(lo, v);
    hi = max(hi, v);
  }
  const bool bad = hi >= 0x7FF0000000000000ll || lo <= 0 ||
                   !(__longlong_as_double(lo) >= PIVOT_RTOL2 * __longlong_as_double(hi));
  const bool rhs = live && j >= L;
  for (int k = L - 1; k >= 0; --k) {
    if (rhs && order == k) {
      m = cmul(m, sm(s.rp[k]));
      s.x[j - L] = d2(m);
    }
    __syncthreads();
    if (rhs && order < k) {
      const double2 u = s.u[order][k], x = s.x[j - L];
      m.re = fma(u.y, x.y, fma(-u.x, x.x, m.re));
      m.im = fma(-u.y, x.x, fma(-u.x, x.y, m.im));
    }
    __syncthreads();
  }
  return bad;
}

// alpha_k from (R~_0^H V_k) alpha_k = R~_0^H R_k, and zeta_k = Tr[W^H R] / Tr[W^H W].
__global__ void solve_alpha_kernel(SolverState* st, int L) {
  __shared__ Lu s;
  if (st->status != ST_OK) return;
  const int e = threadIdx.x, j = e / L, i = e - j * L;
  const bool live = j < 2 * L;
  if (e == blockDim.x - 32) {
    const double ww = st->trww;
    const double2 wr = st->trwr;
    const double2 z = make_double2(wr.x / ww, wr.y / ww);
    // an imaginary part of NaN marks a zeta that cannot be used
    const bool bad = !(ww > 0.0) || !isfinite(z.x) || !isfinite(z.y);
    s.extra = bad ? make_double2(0.0, __longlong_as_double(0x7FF8000000000000ll)) : z;
  }
  Cx<double> m = czero<double>();
  if (live) m = j < L ? sm(st->rtv[i * L + j]) : sm(st->rtr[i * L + j - L]);
  int row;
  const bool bad = lu_solve(s, m, L, i, j, live, row);
  if (live && j >= L) st->alpha[(bad ? i : row) * L + j - L] = bad ? make_double2(0, 0) : d2(m);
  if (e == 0) {
    const bool zbad = isnan(s.extra.y);
    st->zeta = zbad ? make_double2(0, 0) : s.extra;
    if (bad) st->status = ST_ALPHA_SINGULAR;
    else if (zbad) st->status = ST_ZETA_BAD;
  }
}

// gamma_k from (R~_0^H R_k) gamma_k = R~_0^H R_{k+1} / zeta_k; then R~_0^H R_k <- R~_0^H R_{k+1}.
__global__ void solve_gamma_kernel(SolverState* st, int L) {
  __shared__ Lu s;
  if (st->status != ST_OK) return;
  const int e = threadIdx.x, j = e / L, i = e - j * L;
  const bool live = j < 2 * L;
  if (e == blockDim.x - 32) {
    const double2 z = st->zeta;
    s.extra = reciprocal(z, z.x * z.x + z.y * z.y);
  }
  Cx<double> m = czero<double>();
  if (live) m = j < L ? sm(st->rtr[i * L + j]) : sm(st->rtr_new[i * L + j - L]);
  const Cx<double> next = m;
  __syncthreads();
  if (live && j >= L) m = cmul(m, sm(s.extra));
  int row;
  const bool bad = lu_solve(s, m, L, i, j, live, row);
  if (live && j >= L) {
    st->gamma[(bad ? i : row) * L + j - L] = bad ? make_double2(0, 0) : d2(m);
    st->rtr[i * L + j - L] = d2(next);
  }
  if (e == 0 && bad) st->status = ST_GAMMA_SINGULAR;
}

// Four blocks of TS_THREADS per SM, for the current device (its SM count is read once per device).
constexpr int MAX_DEVICES = 64;
int g_sm_count[MAX_DEVICES] = {};

int max_blocks() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) {
    cudaGetLastError();
    return 4 * 152;
  }
  if (!g_sm_count[dev]) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      n = 152;
    }
    g_sm_count[dev] = n;
  }
  return 4 * g_sm_count[dev];
}

inline int blocks_for(long long rows) {
  const long long nchunks = (rows + CH - 1) / CH;
  const long long cap = max_blocks();
  return (int)(nchunks < cap ? (nchunks > 0 ? nchunks : 1) : cap);
}

// Grid of the digit kernels: a block takes 64 rows at a time, `per_sm` (at most 4) are resident on an SM.
inline int digit_blocks(long long rows, int per_sm) {
  const long long n = (rows + 63) / 64, cap = max_blocks() / 4 * per_sm;
  return (int)(n < cap ? (n > 0 ? n : 1) : cap);
}

}  // namespace

int ts_blocks(long long rows) { return blocks_for(rows); }
int ts_max_blocks() { return max_blocks(); }

cudaError_t launch_gram(const double* A, const double* B, int L, long long rows, double2* part,
                        SolverState* st, int which, bool norms_of_b, cudaStream_t s) {
  const int nb = digit_blocks(rows, gram_blocks(L, false));
  const cudaError_t e = launch_gram_dg(A, B, L, rows, nb, part, norms_of_b, s);
  if (e != cudaSuccess) return e;
  finalize(part, nb, L, st, which, norms_of_b ? st->rnorm2 : nullptr, false, s);
  return cudaGetLastError();
}

cudaError_t launch_colnorms(const double* A, int L, long long rows, double2* part,
                            double* out_norm2, cudaStream_t s) {
  const int nb = blocks_for(rows);
  colnorm_kernel<<<nb, TS_THREADS, 0, s>>>(A, L, rows, part);
  finalize(part, nb, L, nullptr, -1, out_norm2, false, s);
  return cudaGetLastError();
}

cudaError_t launch_traces(const double* W, const double* R, int L, long long rows,
                          double2* part, SolverState* st, cudaStream_t s) {
  const int nb = blocks_for(rows);
  trace_kernel<<<nb, TS_THREADS, 0, s>>>(W, R, rows * L, part);
  finalize(part, nb, L, st, -1, nullptr, true, s);
  return cudaGetLastError();
}

cudaError_t launch_solve_alpha(SolverState* st, int L, cudaStream_t s) {
  solve_alpha_kernel<<<1, lu_threads(L), 0, s>>>(st, L);
  return cudaGetLastError();
}

cudaError_t launch_solve_gamma(SolverState* st, int L, cudaStream_t s) {
  solve_gamma_kernel<<<1, lu_threads(L), 0, s>>>(st, L);
  return cudaGetLastError();
}

cudaError_t launch_update_u(const double* P, const double* V, double* U, int L, long long rows,
                            const SolverState* st, cudaStream_t s, bool df) {
  return launch_update_u_dg(P, V, U, L, rows, digit_blocks(rows, update_u_blocks(L, df)), st, s, df);
}

cudaError_t launch_update_xr(double* X, const double* F, const double* G, double* R,
                             const double* W, const double* Y, const double* Rt, int L,
                             long long rows, double2* part, SolverState* st, cudaStream_t s,
                             bool df) {
  const int nb = digit_blocks(rows, gram_blocks(L, df));
  const cudaError_t e = launch_update_xr_dg(X, F, G, R, W, Y, Rt, L, rows, nb, part, st, s, df);
  if (e != cudaSuccess) return e;
  finalize(part, nb, L, st, GRAM_RTR_NEW, st->rnorm2, false, s);
  return cudaGetLastError();
}

cudaError_t launch_update_pv(double* P, double* V, const double* R, const double* W,
                             const double* U, const double* Y, const double* Rt, int L,
                             long long rows, double2* part, SolverState* st, cudaStream_t s,
                             bool df) {
  const int nb = digit_blocks(rows, update_pv_blocks(L, df));
  const cudaError_t e = launch_update_pv_dg(P, V, R, W, U, Y, Rt, L, rows, nb, part, st, s, df);
  if (e != cudaSuccess) return e;
  finalize(part, nb, L, st, GRAM_RTV, nullptr, false, s);
  return cudaGetLastError();
}
