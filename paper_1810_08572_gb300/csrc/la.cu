// Sparse linear algebra kernels and Krylov drivers (Section 2.5: the paper
// uses AMG-preconditioned Krylov solvers; these are the GPU-native ones).
#include <cstdlib>

#include "la.cuh"
#include "reduce.cuh"

namespace fvs {

// ---------------------------------------------------------------------------
// SpMV and residual (ELL, one thread per row, slot-major coalesced loads)
// ---------------------------------------------------------------------------
// the row kernels by width (7: face-only rows) and by whether the matrix streams
#define FVS_BY_ROW(A_, CALL)                                                     \
  do {                                                                           \
    const bool big_ = (A_).n * (int64_t)(A_).w * 12 > L2_KEEP_BYTES;             \
    if ((A_).w == 7 && big_) { constexpr int W = 7; constexpr bool CS = true; CALL; }        \
    else if ((A_).w == 7) { constexpr int W = 7; constexpr bool CS = false; CALL; }          \
    else if (big_) { constexpr int W = 0; constexpr bool CS = true; CALL; }      \
    else { constexpr int W = 0; constexpr bool CS = false; CALL; }               \
    FVS_COUNT_LAUNCH();                                                          \
  } while (0)

template <int W, bool CS>
__global__ void k_residual(int64_t n, int w, const int32_t* __restrict__ col, const double* __restrict__ val,
                           const double* __restrict__ x, const double* __restrict__ b, double* __restrict__ r,
                           const double* __restrict__ dextra) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double acc = ell_row<W, CS>(n, w, col, val, x, i, dextra ? dextra[i] * x[i] : 0.0);
    r[i] = b[i] - acc;
  }
}

fvs_status residual(cudaStream_t s, const Ell& A, const double* x, const double* b, double* r,
                    const double* dextra) {
  if (A.n == 0) return FVS_OK;
  ProfScope ps(&A, "residual", (double)A.n * (12.0 * A.w + 24.0 + (dextra ? 8.0 : 0.0)), s);
  FVS_BY_ROW(A, (k_residual<W, CS><<<stride_grid(A.n, 256), 256, 0, s>>>(A.n, A.w, A.col, A.val, x, b, r, dextra)));
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

// sc[s0] = a . b (and sc[s1] = c . d with c given)
template <bool TWO>
__global__ void __launch_bounds__(RB) k_dot2(int64_t n, const double* __restrict__ a, const double* __restrict__ b,
                                             const double* __restrict__ c, const double* __restrict__ d,
                                             double* part, unsigned int* ticket, double* sc, int s0, int s1) {
  double x = 0.0, y = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    x = fma(a[i], b[i], x);
    if (TWO) y = fma(c[i], d[i], y);
  }
  if (grid_fold<OpSum, TWO ? 2 : 1>(x, y, part, ticket)) {
    sc[s0] = x;
    if (TWO) sc[s1] = y;
  }
}

// sc[s0] = max |a - b|, sc[s1] = max |c - d|
__global__ void __launch_bounds__(RB) k_maxdiff2(int64_t n, const double* __restrict__ a,
                                                 const double* __restrict__ b, const double* __restrict__ c,
                                                 const double* __restrict__ d, double* part, unsigned int* ticket,
                                                 double* sc, int s0, int s1) {
  double x = 0.0, y = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    x = fmax(x, fabs(a[i] - b[i]));
    if (c) y = fmax(y, fabs(c[i] - d[i]));
  }
  if (grid_fold<OpMax, 2>(x, y, part, ticket)) {
    sc[s0] = x;
    if (s1 >= 0) sc[s1] = y;
  }
}

fvs_status Reducer::init() {
  cudaStream_t st = g_alloc_stream;
  blocks = 8 * sm_count();   // full occupancy for the fused SpMV + reduction kernels
  FVS_TRY(part.alloc(3 * (size_t)blocks));
  FVS_TRY(sc.alloc(S_NSLOT));
  FVS_TRY(sc.zero(st));
  FVS_TRY(ticket.alloc(1));
  FVS_TRY(ticket.zero(st));
  FVS_TRY(iter.alloc(3));
  FVS_TRY(iter.zero(st));
  if (!host) FVS_CUDA(cudaMallocHost(&host, S_NSLOT * sizeof(double)));
  return FVS_OK;
}

fvs_status Reducer::dot(cudaStream_t s, int64_t n, const double* x, const double* y, int slot) {
  k_dot2<false><<<vgrid(n), RB, 0, s>>>(n, x, y, nullptr, nullptr, part, ticket, sc, slot, -1); FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

fvs_status Reducer::dot2(cudaStream_t s, int64_t n, const double* a, const double* b, const double* c,
                         const double* d, int s0, int s1) {
  k_dot2<true><<<vgrid(n), RB, 0, s>>>(n, a, b, c, d, part, ticket, sc, s0, s1); FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

fvs_status Reducer::max_abs_diff2(cudaStream_t s, int64_t n, const double* a, const double* b,
                                  const double* c, const double* d, int s0, int s1) {
  k_maxdiff2<<<vgrid(n), RB, 0, s>>>(n, a, b, c, d, part, ticket, sc, s0, s1); FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

fvs_status Reducer::fetch(cudaStream_t s) {
  FVS_CUDA(cudaMemcpyAsync(host, sc.p, S_NSLOT * sizeof(double), cudaMemcpyDeviceToHost, s));
  FVS_CUDA(cudaStreamSynchronize(s));
  return FVS_OK;
}

// ---------------------------------------------------------------------------
// vector kernels
// ---------------------------------------------------------------------------
#define GRID_STRIDE(i, n) \
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

__global__ void k_copy(int64_t n, const double* __restrict__ a, double* __restrict__ b) {
  GRID_STRIDE(i, n) b[i] = a[i];
}
__global__ void k_fill(int64_t n, double v, double* __restrict__ a) {
  GRID_STRIDE(i, n) a[i] = v;
}
fvs_status vcopy(cudaStream_t s, int64_t n, const double* a, double* b) {
  if (n <= 0) return FVS_OK;
  k_copy<<<stride_grid(n, 256), 256, 0, s>>>(n, a, b); FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}
fvs_status vfill(cudaStream_t s, int64_t n, double v, double* a) {
  if (n <= 0) return FVS_OK;
  k_fill<<<stride_grid(n, 256), 256, 0, s>>>(n, v, a); FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

__global__ void k_jacobi_apply(int64_t n, const double* __restrict__ diag, const double* __restrict__ dextra,
                               const double* __restrict__ r, double* __restrict__ z) {
  GRID_STRIDE(i, n) {
    const double d = diag[i] + (dextra ? dextra[i] : 0.0);
    z[i] = r[i] / d;
  }
}

// z = dinv r: the inverse diagonal is formed once per linear system by its
// owner (an FP64 division per row per application costs more than the
// memory traffic of this kernel on this part)
__global__ void k_jacobi_mul(int64_t n, const double* __restrict__ dinv, const double* __restrict__ r,
                             double* __restrict__ z) {
  GRID_STRIDE(i, n) z[i] = dinv[i] * r[i];
}

fvs_status JacobiPrecond::apply(cudaStream_t s, const double* r, double* z) {
  if (A->n == 0) return FVS_OK;
  if (dinv) k_jacobi_mul<<<stride_grid(A->n, 256), 256, 0, s>>>(A->n, dinv, r, z);
  else k_jacobi_apply<<<stride_grid(A->n, 256), 256, 0, s>>>(A->n, A->diag, dextra, r, z);
  FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

fvs_status KrylovWork::ensure(int64_t n) {
  const size_t m = (size_t)n + 1;
  FVS_TRY(r.alloc(m)); FVS_TRY(rh.alloc(m)); FVS_TRY(p.alloc(m)); FVS_TRY(ph.alloc(m));
  FVS_TRY(v.alloc(m)); FVS_TRY(sv.alloc(m)); FVS_TRY(sh.alloc(m)); FVS_TRY(t.alloc(m));
  FVS_TRY(z.alloc(m)); FVS_TRY(q.alloc(m));
  return FVS_OK;
}

// safe quotient for Krylov scalars (a breakdown shows up as a stalled residual)
__device__ __forceinline__ double sdiv(double a, double b) { return b != 0.0 ? a / b : 0.0; }

// ---------------------------------------------------------------------------
// Reductions fused into the Krylov kernels, and the scalars they finish
// ---------------------------------------------------------------------------
enum { FIN_RV = 0, FIN_TSTT = 1, FIN_RR_RHO = 2, FIN_PQ = 3, FIN_RR = 4, FIN_START = 5, FIN_TRUE = 6 };

template <int MODE>
__device__ __forceinline__ bool finish2(double x, double y, double* part, unsigned int* ticket, double* sc) {
  constexpr int NS = MODE == FIN_TSTT || MODE == FIN_RR_RHO || MODE == FIN_START ? 2 : 1;
  if (!grid_fold<OpSum, NS>(x, y, part, ticket)) return false;
  if (MODE == FIN_RV) {
    sc[S_RV] = x;
    sc[S_ALPHA] = sdiv(sc[S_RHO], x);
  } else if (MODE == FIN_TSTT) {
    sc[S_TS] = x;
    sc[S_TT] = y;
    sc[S_OMEGA] = sdiv(x, y);
  } else if (MODE == FIN_RR_RHO) {
    const double rho = sc[S_RHO];
    sc[S_RR] = x;
    sc[S_RHO] = y;
    sc[S_BETA] = sdiv(y, rho) * sdiv(sc[S_ALPHA], sc[S_OMEGA]);
    sc[S_FIRST] = 0.0;
  } else if (MODE == FIN_PQ) {
    sc[S_PQ] = x;
    sc[S_ALPHA] = sdiv(sc[S_RZ], x);
  } else if (MODE == FIN_RR) {
    sc[S_RR] = x;
    sc[S_FIRST] = 0.0;
  } else if (MODE == FIN_START) {
    sc[S_RR] = sc[S_RHO] = x;
    sc[S_BB] = y;
  } else if (MODE == FIN_TRUE) {
    sc[S_TRUE] = x;
  }
  return true;
}

// y = A x (+ dextra x); sums d.y (and y.y in FIN_TSTT)
template <int MODE, bool DX, int W, bool CS>
__global__ void __launch_bounds__(RB, W > 0 ? 6 : 8) k_spmv_dot(int64_t n, int w, const int32_t* __restrict__ col,
                                                    const double* __restrict__ val, const double* __restrict__ x,
                                                    double* __restrict__ y, const double* __restrict__ dextra,
                                                    const double* __restrict__ d, double* part,
                                                    unsigned int* ticket, double* sc) {
  double a = 0.0, b = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    const double acc = ell_row<W, CS>(n, w, col, val, x, i, DX ? dextra[i] * x[i] : 0.0);
    y[i] = acc;
    a = fma(d[i], acc, a);
    if (MODE == FIN_TSTT) b = fma(acc, acc, b);
  }
  finish2<MODE>(a, b, part, ticket, sc);
}

template <int PM>
__device__ __forceinline__ double first_weight(const FirstSweep& f) {
  return PM != 0 && f.w ? f.w[0] : 1.0;
}
template <int PM>
__device__ __forceinline__ void first_sweep(const FirstSweep& f, double w, int64_t i, double v) {
  if (PM == 1) f.x[i] = w * f.dinv[i] * v;
  if (PM == 2) {
    const float b = (float)v;
    f.bf[i] = b;
    f.xf[i] = (float)w * f.dinvf[i] * b;
  }
}
// the first sweep alone (before the first iteration of a CG recurrence)
template <int PM>
__global__ void k_first_sweep(int64_t n, FirstSweep f, const double* __restrict__ v) {
  const double w = first_weight<PM>(f);
  GRID_STRIDE(i, n) first_sweep<PM>(f, w, i, v[i]);
}

// Device-driven solve loop: the thread that finishes the last reduction of an
// iteration decides whether the conditional while-node runs the body again
// (no host round trip, no launch of its own).  Bounded by it[1]; a NaN
// residual or a breakdown of the BiCGStab recurrence also stops the loop (the
// host then restarts or reports).
struct LoopCtl {
  cudaGraphConditionalHandle h;
  int* it = nullptr;    // counter and bound; null: no loop
};
__device__ __forceinline__ void loop_next(const LoopCtl& c, double* sc, bool alive) {
  if (!c.it) return;
  const int n = ++c.it[0];
  sc[S_ITER] = (double)n;
  const double rr = sc[S_RR];
  cudaGraphSetConditional(c.h, n < c.it[1] && rr > sc[S_TOL2] && rr == rr && rr < 1e300 && alive ? 1u : 0u);
}

// BiCGStab without a projection: start (r = rh = b - A x, sums r.r = rh.r and
// b.b) and end (r.r of the true residual, r itself not stored) in one launch
// each instead of a residual, a copy and two dot products (2,097,152 rows of
// 27 entries: 128 and 124 us, the residual alone 126 us; at 184,320 rows 19
// and 17 us, where the separate launches took 45 and 31)
template <int MODE, bool DX, int W, bool CS>
__global__ void __launch_bounds__(RB, W > 0 ? 6 : 8) k_residual_dot(int64_t n, int w, const int32_t* __restrict__ col,
                                                        const double* __restrict__ val, const double* __restrict__ x,
                                                        const double* __restrict__ dextra,
                                                        const double* __restrict__ b, double* __restrict__ r,
                                                        double* __restrict__ rh, double* part,
                                                        unsigned int* ticket, double* sc, const int* go) {
  if (MODE == FIN_TRUE && go && !*go) return;   // no loop was entered: the start's residual stands
  double rr = 0.0, bb = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    const double acc = ell_row<W, CS>(n, w, col, val, x, i, DX ? dextra[i] * x[i] : 0.0);
    const double bi = b[i], ri = bi - acc;
    if (MODE == FIN_START) {
      r[i] = ri;
      rh[i] = ri;
      bb = fma(bi, bi, bb);
    }
    rr = fma(ri, ri, rr);
  }
  finish2<MODE>(rr, bb, part, ticket, sc);
}

// BiCGStab: x += alpha ph + omega sh ; r = s - omega t ; sums r.r and rh.r
__global__ void __launch_bounds__(RB) k_bicg_xr_dot(int64_t n, double* __restrict__ sc,
                                                    const double* __restrict__ ph, const double* __restrict__ sh,
                                                    const double* __restrict__ sv, const double* __restrict__ t,
                                                    const double* __restrict__ rh, double* __restrict__ x,
                                                    double* __restrict__ r, double* part, unsigned int* ticket,
                                                    LoopCtl ctl) {
  const double alpha = sc[S_ALPHA], omega = sc[S_OMEGA];
  double a = 0.0, b = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    x[i] = fma(alpha, ph[i], fma(omega, sh[i], x[i]));
    const double ri = fma(-omega, t[i], sv[i]);
    r[i] = ri;
    a = fma(ri, ri, a);
    b = fma(rh[i], ri, b);
  }
  if (finish2<FIN_RR_RHO>(a, b, part, ticket, sc))
    loop_next(ctl, sc, sc[S_TT] != 0.0 && sc[S_RV] != 0.0 && sc[S_RHO] != 0.0);
}

// CG: x += alpha p ; r -= alpha q ; sums r.r, and the preconditioner's first
// sweep on the new r
template <int PM>
__global__ void __launch_bounds__(RB) k_cg_xr_dot(int64_t n, double* __restrict__ sc, const double* __restrict__ p,
                                                  const double* __restrict__ q, double* __restrict__ x,
                                                  double* __restrict__ r, FirstSweep f, double* part,
                                                  unsigned int* ticket, LoopCtl ctl) {
  const double alpha = sc[S_ALPHA], w = first_weight<PM>(f);
  double a = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    x[i] += alpha * p[i];
    const double ri = r[i] - alpha * q[i];
    r[i] = ri;
    first_sweep<PM>(f, w, i, ri);
    a = fma(ri, ri, a);
  }
  if (finish2<FIN_RR>(a, 0.0, part, ticket, sc)) loop_next(ctl, sc, true);
}
// CG: sums r.z and forms beta with the one before; with a mean to project out of z also the
// mean of z over its rows, which k_cg_p subtracts as it reads z, and the sum
// of r over them (zero but for rounding, which counts near the attainable
// residual): r.z of the projected z is r.z - mean sum(r)
__device__ __forceinline__ bool in_mean(const MeanPart& m, int64_t i) {
  return !m.lab || (m.want < 0 ? m.lab[i] >= 0 : m.lab[i] == m.want);
}
template <bool MEAN>
__global__ void __launch_bounds__(RB) k_dot_rz(int64_t n, const double* __restrict__ r, const double* __restrict__ z,
                                               MeanPart m, double* part, unsigned int* ticket, double* sc) {
  double v[MEAN ? 3 : 1] = {};
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    const double zi = z[i], ri = r[i];
    v[0] = fma(ri, zi, v[0]);
    if (MEAN && in_mean(m, i)) {
      v[MEAN ? 1 : 0] += zi;
      v[MEAN ? 2 : 0] += ri;
    }
  }
  if (!grid_fold<OpSum, MEAN ? 3 : 1>(v, part, ticket)) return;
  double rz = v[0];
  if (MEAN) {
    const double c = m.cnt ? *m.cnt : (double)n, mean = c > 0.0 ? v[MEAN ? 1 : 0] / c : 0.0;
    sc[S_MEAN] = mean;
    rz -= mean * v[MEAN ? 2 : 0];
  }
  const double old = sc[S_RZ];
  sc[S_RZ] = rz;
  sc[S_BETA] = sdiv(rz, old);
}

// BiCGStab: p = r + beta (p - omega v), beta = (rho/rho_old)(alpha/omega),
// and the preconditioner's first sweep on p
template <int PM>
__global__ void k_bicg_p(int64_t n, const double* __restrict__ sc, const double* __restrict__ r,
                         const double* __restrict__ v, double* __restrict__ p, int first, FirstSweep f) {
  first = first || sc[S_FIRST] != 0.0;
  const double beta = sc[S_BETA], om = sc[S_OMEGA], w = first_weight<PM>(f);
  GRID_STRIDE(i, n) {
    const double pi = first ? r[i] : r[i] + beta * (p[i] - om * v[i]);
    p[i] = pi;
    first_sweep<PM>(f, w, i, pi);
  }
}
// s = r - alpha v, alpha = rho / (rh . v), and the first sweep on s
template <int PM>
__global__ void k_bicg_s(int64_t n, const double* __restrict__ sc, const double* __restrict__ r,
                         const double* __restrict__ v, double* __restrict__ sv, FirstSweep f) {
  const double alpha = sc[S_ALPHA], w = first_weight<PM>(f);
  GRID_STRIDE(i, n) {
    const double si = r[i] - alpha * v[i];
    sv[i] = si;
    first_sweep<PM>(f, w, i, si);
  }
}
template <bool MEAN>
__global__ void k_cg_p(int64_t n, const double* __restrict__ sc, const double* __restrict__ z,
                       double* __restrict__ p, int first, MeanPart m) {
  first = first || sc[S_FIRST] != 0.0;
  const double beta = sc[S_BETA], mean = MEAN ? sc[S_MEAN] : 0.0;
  GRID_STRIDE(i, n) {
    double zi = z[i];
    if (MEAN && in_mean(m, i)) zi -= mean;
    p[i] = first ? zi : zi + beta * p[i];
  }
}
#define FVS_BY_MODE(mode_, CALL)   \
  do {                             \
    if ((mode_) == 2) { constexpr int PM = 2; CALL; } \
    else if ((mode_) == 1) { constexpr int PM = 1; CALL; } \
    else { constexpr int PM = 0; CALL; } \
    FVS_COUNT_LAUNCH();            \
    FVS_LAUNCH_CHECK();            \
  } while (0)

constexpr int MAX_RESTARTS = 3;   // from the true residual, once the recursive one has met the tolerance

template <int MODE, bool DX>
static void launch_spmv_dot(cudaStream_t s, Reducer& red, const Ell& A, const double* x, double* y,
                            const double* dextra, const double* d) {
  FVS_BY_ROW(A, (k_spmv_dot<MODE, DX, W, CS><<<red.rgrid(red.grid(A.n), W > 0 ? 6 : 8), RB, 0, s>>>(
      A.n, A.w, A.col, A.val, x, y, dextra, d, red.part, red.ticket, red.sc)));
}
template <int MODE>
static fvs_status spmv_dot(cudaStream_t s, Reducer& red, const Ell& A, const double* x, double* y,
                           const double* dextra, const double* d) {
  ProfScope ps(&A, "spmv", (double)A.n * (12.0 * A.w + 24.0 + (dextra ? 8.0 : 0.0)), s);
  if (dextra) launch_spmv_dot<MODE, true>(s, red, A, x, y, dextra, d);
  else launch_spmv_dot<MODE, false>(s, red, A, x, y, dextra, d);
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

template <int MODE, bool DX>
static void launch_residual_dot(cudaStream_t s, Reducer& red, const Ell& A, const double* x, const double* dextra,
                                const double* b, double* r, double* rh, const int* go) {
  FVS_BY_ROW(A, (k_residual_dot<MODE, DX, W, CS><<<red.rgrid(red.grid(A.n), W > 0 ? 6 : 8), RB, 0, s>>>(
      A.n, A.w, A.col, A.val, x, dextra, b, r, rh, red.part, red.ticket, red.sc, go)));
}
template <int MODE>
static fvs_status residual_dot(cudaStream_t s, Reducer& red, const Ell& A, const double* x, const double* dextra,
                               const double* b, double* r, double* rh, const int* go = nullptr) {
  ProfScope ps(&A, "residual", (double)A.n * (12.0 * A.w + (MODE == FIN_START ? 32.0 : 16.0) + (dextra ? 8.0 : 0.0)), s);
  if (dextra) launch_residual_dot<MODE, true>(s, red, A, x, dextra, b, r, rh, go);
  else launch_residual_dot<MODE, false>(s, red, A, x, dextra, b, r, rh, go);
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

// ---------------------------------------------------------------------------
// CUDA-graph replay of one Krylov iteration (launch overhead dominates the
// small levels of the V-cycle and small meshes).  The first iteration runs
// eagerly; the next ones replay a captured graph while its key (operator,
// vectors, preconditioner state) is unchanged.  Disabled while kernels are
// being timed and by FVS_NO_GRAPHS.
// ---------------------------------------------------------------------------
bool graphs_enabled() {
  static int cached = -1;
  if (cached < 0) cached = getenv("FVS_NO_GRAPHS") ? 0 : 1;
  return cached == 1 && !(g_prof && g_prof->on);
}

static uint64_t mixk(uint64_t h, uint64_t v) {
  h ^= v + 0x9e3779b97f4a7c15ULL + (h << 6) + (h >> 2);
  return h;
}

static uint64_t graph_key(const Ell& A, const double* dextra, const Precond& M, const double* b, const double* x,
                          const KrylovWork& w, const Reducer& red) {
  uint64_t h = 1469598103934665603ULL;
  h = mixk(h, (uint64_t)(uintptr_t)A.val.p);
  h = mixk(h, (uint64_t)(uintptr_t)A.col.p);
  h = mixk(h, (uint64_t)A.n * 131 + (uint64_t)A.w);
  h = mixk(h, (uint64_t)(uintptr_t)dextra);
  h = mixk(h, M.signature());
  h = mixk(h, (uint64_t)(uintptr_t)b);
  h = mixk(h, (uint64_t)(uintptr_t)x);
  h = mixk(h, (uint64_t)(uintptr_t)w.r.p);
  h = mixk(h, (uint64_t)(uintptr_t)w.p.p);
  h = mixk(h, (uint64_t)(uintptr_t)red.sc.p);
  h = mixk(h, (uint64_t)(uintptr_t)red.part.p);
  return h ? h : 1;
}

template <typename F>
static fvs_status run_body(cudaStream_t s, IterGraph* g, uint64_t key, bool first, F& body) {
  if (first || !g || g->disabled || !graphs_enabled() || s == nullptr) return body(first, LoopCtl());
  if (!g->exec || g->key != key) {
    g->reset();
    cudaGraph_t graph = nullptr;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      g->disabled = true;
      return body(first, LoopCtl());
    }
    const unsigned long long before = __atomic_load_n(&g_launches, __ATOMIC_RELAXED);
    fvs_status r = body(false, LoopCtl());
    g->kernels = __atomic_load_n(&g_launches, __ATOMIC_RELAXED) - before;
    __atomic_sub_fetch(&g_launches, g->kernels, __ATOMIC_RELAXED);   // counted when replayed
    cudaError_t e = cudaStreamEndCapture(s, &graph);
    if (r != FVS_OK || e != cudaSuccess || !graph) {
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      g->disabled = true;
      return body(first, LoopCtl());
    }
    e = cudaGraphInstantiate(&g->exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
      cudaGetLastError();
      g->exec = nullptr;
      g->disabled = true;
      return body(first, LoopCtl());
    }
    g->key = key;
  }
  FVS_CUDA(cudaGraphLaunch(g->exec, s));
  __atomic_add_fetch(&g_launches, g->kernels, __ATOMIC_RELAXED);
  return FVS_OK;
}

__host__ __device__ __forceinline__ bool bad(double v) { return !(v == v) || v > 1e300 || v < -1e300; }

// what a residual is measured against
__host__ __device__ __forceinline__ double residual_scale(double bb, double floor) {
  const double b = fmax(sqrt(bb), floor);
  return b == 0.0 ? 1.0 : b;
}

// The loop's bound and tolerance lie in memory, so that a loop captured once
// serves every solve.  At the start of a solve the loop is entered only if
// the residual just formed is finite and above the tolerance.
__global__ void k_loop_init(double* sc, int* it, int maxit, double rtol, double floor, int fresh, int start) {
  const double bn = residual_scale(sc[S_BB], floor);
  sc[S_FIRST] = fresh ? 1.0 : 0.0;
  it[0] = 0;
  it[1] = maxit;
  sc[S_ITER] = 0.0;
  sc[S_TOL2] = (rtol * bn) * (rtol * bn);
  int go = 1;
  if (start) {
    const double rn = sqrt(sc[S_RR]);
    sc[S_START] = sc[S_RR];
    go = !(bad(rn) || bad(bn) || rn / bn <= rtol);
  }
  it[2] = go;
}
__global__ void k_loop_gate(cudaGraphConditionalHandle h, const int* it) { cudaGraphSetConditional(h, it[2] ? 1u : 0u); }

// Runs up to maxit iterations of body() as one graph launch with a
// conditional while-node; returns false (nothing launched) when the loop
// graph cannot be used, so the caller iterates from the host instead.
template <typename F>
static bool run_loop(cudaStream_t s, IterGraph* g, uint64_t key, Reducer& red, double rtol, double floor, int maxit,
                     bool fresh, bool start, F& body, fvs_status& st) {
  st = FVS_OK;
  if (!g || g->loop_disabled || !graphs_enabled() || s == nullptr || maxit <= 0) return false;
  if (!g->loop || g->loop_key != key) {
    if (g->loop) cudaGraphExecDestroy(g->loop);
    g->loop = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphConditionalHandle h;
    bool ok = cudaGraphCreate(&graph, 0) == cudaSuccess;
    ok = ok && cudaGraphConditionalHandleCreate(&h, graph, 1, cudaGraphCondAssignDefault) == cudaSuccess;
    cudaGraphNodeParams p = {};
    cudaGraphNode_t node, gate;
    if (ok) {
      const int* itp = red.iter.p;
      void* args[] = {&h, &itp};
      cudaKernelNodeParams kp = {};
      kp.func = (void*)k_loop_gate;
      kp.gridDim = dim3(1);
      kp.blockDim = dim3(1);
      kp.kernelParams = args;
      ok = cudaGraphAddKernelNode(&gate, graph, nullptr, 0, &kp) == cudaSuccess;
    }
    if (ok) {
      p.type = cudaGraphNodeTypeConditional;
      p.conditional.handle = h;
      p.conditional.type = cudaGraphCondTypeWhile;
      p.conditional.size = 1;
      ok = cudaGraphAddNode(&node, graph, &gate, nullptr, 1, &p) == cudaSuccess;
    }
    if (ok) {
      cudaGraph_t bodyg = p.conditional.phGraph_out[0];
      ok = cudaStreamBeginCaptureToGraph(s, bodyg, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) ==
           cudaSuccess;
      if (ok) {
        const unsigned long long before = __atomic_load_n(&g_launches, __ATOMIC_RELAXED);
        LoopCtl ctl;
        ctl.h = h;
        ctl.it = red.iter.p;
        fvs_status r = body(false, ctl);
        g->loop_kernels = __atomic_load_n(&g_launches, __ATOMIC_RELAXED) - before;
        __atomic_sub_fetch(&g_launches, g->loop_kernels, __ATOMIC_RELAXED);
        cudaGraph_t out = nullptr;
        const cudaError_t e = cudaStreamEndCapture(s, &out);
        ok = r == FVS_OK && e == cudaSuccess;
      }
    }
    if (ok) ok = cudaGraphInstantiate(&g->loop, graph, 0) == cudaSuccess;
    if (graph) cudaGraphDestroy(graph);
    if (!ok) {
      cudaGetLastError();
      if (g->loop) cudaGraphExecDestroy(g->loop);
      g->loop = nullptr;
      g->loop_disabled = true;
      return false;
    }
    g->loop_key = key;
  }
  k_loop_init<<<1, 1, 0, s>>>(red.sc.p, red.iter.p, maxit, rtol, floor, fresh ? 1 : 0, start ? 1 : 0);
  FVS_COUNT_LAUNCH();
  FVS_COUNT_LAUNCH();   // the gate
  const cudaError_t e = cudaGraphLaunch(g->loop, s);
  if (e != cudaSuccess) {
    set_error("cudaGraphLaunch: %s", cudaGetErrorString(e));
    st = FVS_ERR_CUDA;
  }
  return true;
}

fvs_status bicgstab(cudaStream_t s, Reducer& red, KrylovWork& w, const Ell& A, const double* dextra,
                    Precond& M, const double* b, double* x, double rtol, int maxit, Projector* proj,
                    SolveResult& res, double bnorm_floor, IterGraph* graph,
                    const std::function<fvs_status()>* tail, double asked) {
  const int64_t n = A.n;
  res = SolveResult();
  if (n == 0) {
    res.converged = true;
    return FVS_OK;
  }
  FVS_TRY(w.ensure(n));
  const int grid = stride_grid(n, 256);
  // r = rh = b - A x; ||b|| of the (projected) right side; rho_0 = rh . r
  if (!proj) {
    FVS_TRY(residual_dot<FIN_START>(s, red, A, x, dextra, b, w.r, w.rh));
  } else {
    FVS_TRY(residual(s, A, x, b, w.r, dextra));
    FVS_TRY(proj->apply(s, w.r));
    FVS_TRY(vcopy(s, n, w.r, w.rh));
    FVS_TRY(vcopy(s, n, b, w.q));
    FVS_TRY(proj->apply(s, w.q));
    FVS_TRY(red.dot2(s, n, w.q, w.q, w.r, w.r, S_BB, S_RR));
    FVS_TRY(red.dot(s, n, w.rh, w.r, S_RHO));
  }
  // K x has zero sum on every singular part (zero column sums), so the
  // Krylov vectors stay in the range once r is projected
  const FirstSweep fp = M.first(w.ph), fs = M.first(w.sh);
  auto body = [&](bool first, const LoopCtl& ctl) -> fvs_status {
    FVS_BY_MODE(fp.mode, (k_bicg_p<PM><<<grid, 256, 0, s>>>(n, red.sc, w.r, w.v, w.p, first ? 1 : 0, fp)));
    FVS_TRY(M.rest(s, w.p, w.ph));
    FVS_TRY(spmv_dot<FIN_RV>(s, red, A, w.ph, w.v, dextra, w.rh));
    FVS_BY_MODE(fs.mode, (k_bicg_s<PM><<<grid, 256, 0, s>>>(n, red.sc, w.r, w.v, w.sv, fs)));
    FVS_TRY(M.rest(s, w.sv, w.sh));
    FVS_TRY(spmv_dot<FIN_TSTT>(s, red, A, w.sh, w.t, dextra, w.sv));
    k_bicg_xr_dot<<<red.rgrid(red.vgrid(n), 5), RB, 0, s>>>(n, red.sc, w.ph, w.sh, w.sv, w.t, w.rh, x, w.r, red.part,
                                              red.ticket, ctl); FVS_COUNT_LAUNCH();
    FVS_LAUNCH_CHECK();
    return FVS_OK;
  };
  const uint64_t key = graph_key(A, dextra, M, b, x, w, red) ^ 0x6b696367ULL;
  // r.r of the true residual (projected: formed in q, so that r stays)
  auto true_residual = [&](const int* go) -> fvs_status {
    if (!proj) return residual_dot<FIN_TRUE>(s, red, A, x, dextra, b, nullptr, nullptr, go);
    FVS_TRY(residual(s, A, x, b, w.q, dextra));
    FVS_TRY(proj->apply(s, w.q));
    return red.dot(s, n, w.q, w.q, S_TRUE);
  };
  // what follows the loop on the device; true: its scalars are of this x
  auto queue_loop = [&](int left, bool fresh, bool start, bool& looped) -> fvs_status {
    fvs_status st = FVS_OK;
    looped = run_loop(s, graph, key, red, rtol, bnorm_floor, left, fresh, start, body, st);
    FVS_TRY(st);
    if (!looped) return FVS_OK;
    FVS_TRY(true_residual(red.iter.p + 2));
    if (tail) FVS_TRY((*tail)());
    return FVS_OK;
  };
  // the iterations run as one device-driven loop, or the first of a
  // recurrence from the host and one graph replay each after that
  bool looped = false;
  FVS_TRY(queue_loop(maxit, true, true, looped));
  FVS_TRY(red.fetch(s));
  const double bnorm = residual_scale(red.host[S_BB], bnorm_floor);
  double rn = sqrt(red.host[looped ? S_START : S_RR]);
  res.relres = rn / bnorm;
  res.tail_done = looped && tail;
  if (bad(rn) || bad(bnorm)) return FVS_OK;   // non-finite data: not converged, no iterations
  if (res.relres <= rtol) {
    res.converged = true;
    return FVS_OK;
  }
  const double tol2 = (rtol * bnorm) * (rtol * bnorm);
  const double accept = 10.0 * (asked > rtol ? asked : rtol);
  bool queued = looped, fresh = true;
  int it = 0;
  double best = 0.0;   // true residual before a restart (its iterate in w.z)
  for (int again = 0;; ++again) {
    while (it < maxit) {
      if (!queued) {
        FVS_TRY(queue_loop(maxit - it, fresh, false, looped));
        if (!looped) FVS_TRY(run_body(s, graph, key, fresh, body));
        FVS_TRY(red.fetch(s));
      }
      queued = fresh = false;
      res.tail_done = looped && tail;
      const int done = looped ? (int)red.host[S_ITER] : 1;
      if (looped) __atomic_add_fetch(&g_launches, graph->loop_kernels * (unsigned long long)done, __ATOMIC_RELAXED);
      it += done;
      rn = sqrt(red.host[S_RR]);
      res.iters = it;
      res.relres = rn / bnorm;
      if (bad(rn)) {
        if (again > 0) {
          FVS_TRY(vcopy(s, n, w.z, x));
          res.relres = best;
          res.tail_done = false;
        }
        return FVS_OK;
      }
      if (res.relres <= rtol || red.host[S_RR] <= tol2) {
        res.converged = true;
        break;
      }
      // restart on breakdown of the shadow residual
      if (red.host[S_TT] == 0.0 || red.host[S_RV] == 0.0 || red.host[S_RHO] == 0.0) {
        FVS_TRY(residual(s, A, x, b, w.r, dextra));
        if (proj) FVS_TRY(proj->apply(s, w.r));
        FVS_TRY(vcopy(s, n, w.r, w.rh));
        FVS_TRY(red.dot(s, n, w.rh, w.r, S_RHO));
        fresh = true;
      }
    }
    // the true residual (the recursive one drifts)
    if (!looped) {
      FVS_TRY(true_residual(nullptr));
      FVS_TRY(red.fetch(s));
    }
    res.relres = sqrt(red.host[S_TRUE]) / bnorm;
    const bool met = res.converged;   // the recursive residual reached rtol
    res.converged = res.relres <= accept && !bad(res.relres);
    // the recursive residual drifted too far from the true one (tight
    // tolerances on large systems): start again from the true residual
    // rather than give the solve up; an attempt that ends further off than it
    // began is undone
    if (again > 0 && !(res.relres <= best)) {
      FVS_TRY(vcopy(s, n, w.z, x));
      res.relres = best;
      res.converged = false;
      res.tail_done = false;
      break;
    }
    if (res.converged || !met || bad(res.relres) || again == MAX_RESTARTS || it >= maxit) break;
    best = res.relres;
    FVS_TRY(vcopy(s, n, x, w.z));
    if (!proj) {
      FVS_TRY(residual_dot<FIN_START>(s, red, A, x, dextra, b, w.r, w.rh));
    } else {
      // the null vectors' share of x, which a long recurrence can let grow until
      // its rounding in A x is the residual, is taken out first
      FVS_TRY(proj->apply(s, x));
      FVS_TRY(residual(s, A, x, b, w.r, dextra));
      FVS_TRY(proj->apply(s, w.r));
      FVS_TRY(vcopy(s, n, w.r, w.rh));
      FVS_TRY(red.dot(s, n, w.rh, w.r, S_RHO));
    }
    fresh = true;
  }
  return FVS_OK;
}

// ---------------------------------------------------------------------------
// preconditioned CG (symmetric systems)
// ---------------------------------------------------------------------------
fvs_status pcg(cudaStream_t s, Reducer& red, KrylovWork& w, const Ell& A, Precond& M, const double* b,
               double* x, double rtol, int maxit, Projector* proj, SolveResult& res, IterGraph* graph) {
  const int64_t n = A.n;
  res = SolveResult();
  if (n == 0) {
    res.converged = true;
    return FVS_OK;
  }
  FVS_TRY(w.ensure(n));
  const int grid = stride_grid(n, 256);
  FVS_TRY(residual(s, A, x, b, w.r, nullptr));
  if (proj) FVS_TRY(proj->apply(s, w.r));
  const double* bb = b;
  if (proj) {
    FVS_TRY(vcopy(s, n, b, w.q));
    FVS_TRY(proj->apply(s, w.q));
    bb = w.q;
  }
  FVS_TRY(red.dot2(s, n, bb, bb, w.r, w.r, S_BB, S_RR));
  const FirstSweep f = M.first(w.z);
  MeanPart mp;
  const int how = proj ? proj->single(mp) : 0;
  auto body = [&](bool first, const LoopCtl& ctl) -> fvs_status {
    // (the first sweep on r is done already)
    FVS_TRY(M.rest(s, w.r, w.z));
    if (how == 2) FVS_TRY(proj->apply(s, w.z));
    if (how == 1) {
      k_dot_rz<true><<<red.vgrid(n), RB, 0, s>>>(n, w.r, w.z, mp, red.part, red.ticket, red.sc); FVS_COUNT_LAUNCH();
      k_cg_p<true><<<grid, 256, 0, s>>>(n, red.sc, w.z, w.p, first ? 1 : 0, mp); FVS_COUNT_LAUNCH();
    } else {
      k_dot_rz<false><<<red.vgrid(n), RB, 0, s>>>(n, w.r, w.z, mp, red.part, red.ticket, red.sc); FVS_COUNT_LAUNCH();
      k_cg_p<false><<<grid, 256, 0, s>>>(n, red.sc, w.z, w.p, first ? 1 : 0, mp); FVS_COUNT_LAUNCH();
    }
    FVS_LAUNCH_CHECK();
    FVS_TRY(spmv_dot<FIN_PQ>(s, red, A, w.p, w.q, nullptr, w.p));
    FVS_BY_MODE(f.mode, (k_cg_xr_dot<PM><<<red.vgrid(n), RB, 0, s>>>(n, red.sc, w.p, w.q, x, w.r, f, red.part,
                                                                    red.ticket, ctl)));
    return FVS_OK;
  };
  auto prepare = [&]() -> fvs_status {
    if (f.mode == 1) { k_first_sweep<1><<<grid, 256, 0, s>>>(n, f, w.r); FVS_COUNT_LAUNCH(); }
    if (f.mode == 2) { k_first_sweep<2><<<grid, 256, 0, s>>>(n, f, w.r); FVS_COUNT_LAUNCH(); }
    FVS_LAUNCH_CHECK();
    return FVS_OK;
  };
  FVS_TRY(prepare());
  const uint64_t key = graph_key(A, nullptr, M, b, x, w, red) ^ (0x70636770ULL + (uint64_t)how);
  // r.r of the true residual (formed in q, so that r stays)
  auto true_residual = [&]() -> fvs_status {
    FVS_TRY(residual(s, A, x, b, w.q, nullptr));
    if (proj) FVS_TRY(proj->apply(s, w.q));
    return red.dot(s, n, w.q, w.q, S_TRUE);
  };
  auto queue_loop = [&](int left, bool fresh, bool start, bool& looped) -> fvs_status {
    fvs_status st = FVS_OK;
    looped = run_loop(s, graph, key, red, rtol, 0.0, left, fresh, start, body, st);
    FVS_TRY(st);
    return looped ? true_residual() : FVS_OK;
  };
  // as in bicgstab
  bool looped = false;
  FVS_TRY(queue_loop(maxit, true, true, looped));
  FVS_TRY(red.fetch(s));
  const double bnorm = residual_scale(red.host[S_BB], 0.0);
  res.relres = sqrt(red.host[looped ? S_START : S_RR]) / bnorm;
  if (bad(res.relres) || bad(bnorm)) return FVS_OK;   // non-finite data: not converged
  if (res.relres <= rtol) {
    res.converged = true;
    return FVS_OK;
  }
  const double tol2 = (rtol * bnorm) * (rtol * bnorm);
  bool queued = looped, fresh = true;
  int it = 0;
  double best = 0.0;   // true residual before a restart (its iterate in w.v)
  for (int again = 0;; ++again) {
    while (it < maxit) {
      if (!queued) {
        FVS_TRY(queue_loop(maxit - it, fresh, false, looped));
        if (!looped) FVS_TRY(run_body(s, graph, key, fresh, body));
        FVS_TRY(red.fetch(s));
      }
      queued = fresh = false;
      const int done = looped ? (int)red.host[S_ITER] : 1;
      if (looped) __atomic_add_fetch(&g_launches, graph->loop_kernels * (unsigned long long)done, __ATOMIC_RELAXED);
      it += done;
      const double rn = sqrt(red.host[S_RR]);
      res.iters = it;
      res.relres = rn / bnorm;
      if (bad(rn)) {
        if (again > 0) {
          FVS_TRY(vcopy(s, n, w.v, x));
          res.relres = best;
        }
        return FVS_OK;
      }
      if (res.relres <= rtol || red.host[S_RR] <= tol2) {
        res.converged = true;
        break;
      }
    }
    if (!looped) {
      FVS_TRY(true_residual());
      FVS_TRY(red.fetch(s));
    }
    res.relres = sqrt(red.host[S_TRUE]) / bnorm;
    const bool met = res.converged;
    res.converged = res.relres <= rtol * 10.0 && !bad(res.relres);
    if (again > 0 && !(res.relres <= best)) {
      FVS_TRY(vcopy(s, n, w.v, x));
      res.relres = best;
      res.converged = false;
      break;
    }
    if (res.converged || !met || bad(res.relres) || again == MAX_RESTARTS || it >= maxit) break;
    best = res.relres;
    FVS_TRY(vcopy(s, n, x, w.v));
    fresh = true;    // from the true residual, as in bicgstab
    if (proj) {
      FVS_TRY(proj->apply(s, x));
      FVS_TRY(residual(s, A, x, b, w.q, nullptr));
      FVS_TRY(proj->apply(s, w.q));
    }
    FVS_TRY(vcopy(s, n, w.q, w.r));
    FVS_TRY(prepare());
  }
  return FVS_OK;
}

}  // namespace fvs
