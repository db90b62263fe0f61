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

// ---------------------------------------------------------------- L x L solves (one warp)
// Solves C Z = Rhs in place: M is the augmented L x 2L matrix [C | Rhs] in shared memory,
// row-major with leading dimension 2*WD_LMAX.  Partial pivoting by the largest modulus.  Returns
// true when the system is singular in the sense of the oracle: a pivot that is not finite or whose
// modulus is below 1e-13 times the largest pivot modulus.
constexpr double PIVOT_RTOL = 1e-13;
constexpr int LD = 2 * WD_LMAX;

__device__ bool lu_solve_warp(Cx<double>* M, int L) {
  const int lane = threadIdx.x;
  double pmax = 0.0, pmin = 1e308;
  bool bad = false;
  for (int k = 0; k < L; ++k) {
    int p = k;
    double best = cnorm2(M[k * LD + k]);
    for (int i = k + 1; i < L; ++i) {
      const double v = cnorm2(M[i * LD + k]);
      if (v > best) { best = v; p = i; }
    }
    __syncwarp();
    if (p != k && lane < 2 * L) {
      const Cx<double> tmp = M[k * LD + lane];
      M[k * LD + lane] = M[p * LD + lane];
      M[p * LD + lane] = tmp;
    }
    __syncwarp();
    const Cx<double> piv = M[k * LD + k];
    const double pa = sqrt(cnorm2(piv));
    if (!isfinite(pa) || pa == 0.0) bad = true;
    pmax = fmax(pmax, pa);
    pmin = fmin(pmin, pa);
    const double pn = cnorm2(piv);
    const Cx<double> rp = cmake(piv.re / pn, -piv.im / pn);
    for (int i = k + 1; i < L; ++i) {
      const Cx<double> f = cmul(M[i * LD + k], rp);
      __syncwarp();
      if (lane > k && lane < 2 * L) M[i * LD + lane] = M[i * LD + lane] - cmul(f, M[k * LD + lane]);
      if (lane == k) M[i * LD + k] = f;
      __syncwarp();
    }
  }
  if (!(pmin >= PIVOT_RTOL * pmax)) bad = true;
  // back substitution, one right-hand-side column per lane
  if (lane >= L && lane < 2 * L) {
    for (int i = L - 1; i >= 0; --i) {
      Cx<double> v = M[i * LD + lane];
      for (int jj = i + 1; jj < L; ++jj) v = v - cmul(M[i * LD + jj], M[jj * LD + lane]);
      const Cx<double> d = M[i * LD + i];
      const double dn = cnorm2(d);
      M[i * LD + lane] = cmul(v, cmake(d.re / dn, -d.im / dn));
    }
  }
  __syncwarp();
  return bad;
}

// alpha_k from (R~_0^H V_k) alpha_k = R~_0^H R_k, and zeta_k = Tr[W^H R] / Tr[W^H W].
__global__ void solve_alpha_kernel(SolverState* st, int L) {
  __shared__ Cx<double> M[WD_LMAX * LD];
  if (st->status != ST_OK) return;
  const int lane = threadIdx.x;
  for (int i = 0; i < L; ++i)
    if (lane < L) {
      M[i * LD + lane] = sm(st->rtv[i * L + lane]);
      M[i * LD + L + lane] = sm(st->rtr[i * L + lane]);
    }
  __syncwarp();
  const bool bad = lu_solve_warp(M, L);
  if (lane < L)
    for (int i = 0; i < L; ++i) st->alpha[i * L + lane] = bad ? make_double2(0, 0) : d2(M[i * LD + L + lane]);
  if (lane == 0) {
    const double ww = st->trww;
    const Cx<double> wr = sm(st->trwr);
    Cx<double> z = cmake(wr.re / ww, wr.im / ww);
    bool zbad = !(ww > 0.0) || !isfinite(z.re) || !isfinite(z.im);
    st->zeta = zbad ? make_double2(0, 0) : d2(z);
    if (bad) st->status = ST_ALPHA_SINGULAR;
    else if (zbad) st->status = ST_ZETA_BAD;
  }
}

// gamma_k from (R~_0^H R_k) gamma_k = R~_0^H R_{k+1} / zeta_k; then R~_0^H R_k <- R~_0^H R_{k+1}.
__global__ void solve_gamma_kernel(SolverState* st, int L) {
  __shared__ Cx<double> M[WD_LMAX * LD];
  if (st->status != ST_OK) return;
  const int lane = threadIdx.x;
  const Cx<double> z = sm(st->zeta);
  const double zn = cnorm2(z);
  const Cx<double> rz = cmake(z.re / zn, -z.im / zn);
  for (int i = 0; i < L; ++i)
    if (lane < L) {
      M[i * LD + lane] = sm(st->rtr[i * L + lane]);
      M[i * LD + L + lane] = cmul(sm(st->rtr_new[i * L + lane]), rz);
    }
  __syncwarp();
  const bool bad = lu_solve_warp(M, L);
  if (lane < L)
    for (int i = 0; i < L; ++i) {
      st->gamma[i * L + lane] = bad ? make_double2(0, 0) : d2(M[i * LD + L + lane]);
      st->rtr[i * L + lane] = st->rtr_new[i * L + lane];
    }
  if (lane == 0 && bad) st->status = ST_GAMMA_SINGULAR;
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
  const int nb = digit_blocks(rows, L > 12 ? 3 : 4);
  launch_gram_dg(A, B, L, rows, nb, part, norms_of_b, s);
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
  solve_alpha_kernel<<<1, 32, 0, s>>>(st, L);
  return cudaGetLastError();
}

cudaError_t launch_solve_gamma(SolverState* st, int L, cudaStream_t s) {
  solve_gamma_kernel<<<1, 32, 0, s>>>(st, L);
  return cudaGetLastError();
}

cudaError_t launch_update_u(const double* P, const double* V, double* U, int L, long long rows,
                            const SolverState* st, cudaStream_t s, bool df) {
  return launch_update_u_dg(P, V, U, L, rows, digit_blocks(rows, 4), st, s, df);
}

cudaError_t launch_update_xr(double* X, const double* F, const double* G, double* R,
                             const double* W, const double* Y, const double* Rt, int L,
                             long long rows, double2* part, SolverState* st, cudaStream_t s,
                             bool df) {
  const int nb = digit_blocks(rows, L > 12 ? 3 : 4);
  launch_update_xr_dg(X, F, G, R, W, Y, Rt, L, rows, nb, part, st, s, df);
  finalize(part, nb, L, st, GRAM_RTR_NEW, st->rnorm2, false, s);
  return cudaGetLastError();
}

cudaError_t launch_update_pv(double* P, double* V, const double* R, const double* W,
                             const double* U, const double* Y, const double* Rt, int L,
                             long long rows, double2* part, SolverState* st, cudaStream_t s,
                             bool df) {
  const int nb = digit_blocks(rows, L > 8 ? 3 : 4);
  launch_update_pv_dg(P, V, R, W, U, Y, Rt, L, rows, nb, part, st, s, df);
  finalize(part, nb, L, st, GRAM_RTV, nullptr, false, s);
  return cudaGetLastError();
}
