// Sparse linear algebra of the solver: ELL matrices, SpMV, deterministic
// reductions, Jacobi, and the Krylov drivers (BiCGStab, CG).
#pragma once

#include <functional>

#include "common.cuh"

namespace fvs {

// ELL matrix stored slot-major: entry k of row i at [k*n + i], so that one
// thread per row reads consecutive addresses across a warp.  Unused slots
// hold col = i and val = 0.
struct Ell {
  int64_t n = 0;
  int w = 0;
  DBuf<int32_t> col;
  DBuf<double> val;
  DBuf<double> diag;   // diagonal (Jacobi)
  DBuf<float> valf;    // FP32 copies for the mixed-precision V-cycle
  DBuf<float> diagf;
  fvs_status alloc(int64_t rows, int width) {
    n = rows;
    w = width;
    FVS_TRY(col.alloc((size_t)rows * width + 1));
    FVS_TRY(val.alloc((size_t)rows * width + 1));
    FVS_TRY(diag.alloc((size_t)rows + 1));
    return FVS_OK;
  }
};

// Scalar slots of the Krylov drivers (device memory).
enum Slot {
  S_RHO = 0, S_ALPHA, S_OMEGA, S_RV, S_TS, S_TT, S_RR, S_BB, S_RZ, S_PQ,
  S_TMP0, S_TMP1, S_TOL2, S_ITER, S_FIRST, S_BETA, S_MEAN, S_START, S_TRUE, S_NSLOT
};

// Reduction scratch owned by a solver: block partials + scalar slots +
// pinned host mirror.
struct Reducer {
  int blocks = 0;
  DBuf<double> part;   // [2*blocks]
  DBuf<double> sc;     // [S_NSLOT]
  DBuf<unsigned int> ticket;   // last-block counter of the fused reductions
  DBuf<int> iter;              // device-driven solve loops: iteration counter and its bound
  double* host = nullptr;  // pinned [S_NSLOT]
  fvs_status init();
  // blocks of 256 threads of a reduction over n rows: a row a thread up to
  // one full wave, then grid-stride
  int grid(int64_t n) const {
    const int64_t g = (n + 255) / 256;
    return (int)(g < 1 ? 1 : (g < blocks ? g : blocks));
  }
  // at most per blocks an SM, what the kernel's registers let reside, so that
  // the stride loop ends in one wave (the seven-slot SpMV at 40 registers six,
  // k_bicg_xr_dot at 48 five: a casting of 422,000 cells 37.0 -> 36.3 ms,
  // 128^3, three steps 154.0 -> 153.3)
  int rgrid(int g, int per) const { return g < blocks / 8 * per ? g : blocks / 8 * per; }
  // the same for kernels that only pass over vectors: half a wave where a
  // full one would leave a thread fewer than two rows.  The partials that the
  // last block folds halve, and the loads in flight still cover the L2 cache:
  // AMG-CG on 442,368 rows 6.77 -> 6.61 ms, a casting of 422,000 cells
  // 37.4 -> 36.5 ms
  int vgrid(int64_t n) const {
    const int64_t g = (n + 255) / 256, top = n < 512 * (int64_t)blocks ? blocks / 2 : blocks;
    return (int)(g < 1 ? 1 : (g < top ? g : top));
  }
  ~Reducer() { if (host) cudaFreeHost(host); }
  // out[slot] = x . y  (deterministic: fixed blocks, fixed order)
  fvs_status dot(cudaStream_t s, int64_t n, const double* x, const double* y, int slot);
  // two dots in one pass: sc[s0] = a.b, sc[s1] = c.d
  fvs_status dot2(cudaStream_t s, int64_t n, const double* a, const double* b,
                  const double* c, const double* d, int s0, int s1);
  fvs_status max_abs_diff2(cudaStream_t s, int64_t n, const double* a, const double* b,
                           const double* c, const double* d, int s0, int s1);
  fvs_status fetch(cudaStream_t s);   // copies sc -> host and waits
};

// r = b - A x (- dextra .* x)
fvs_status residual(cudaStream_t s, const Ell& A, const double* x, const double* b, double* r,
                    const double* dextra = nullptr);

// What a preconditioner does first with its right side v, row by row: the
// Krylov kernel that forms v does it in the same pass (one launch and one
// read of v less; with the mean projected as CG forms p and the loop's end
// decided by the last reduction, a CG iteration on a two-level hierarchy of
// 4,096 rows went from 19 launches to 13, an FP32 cycle loses three passes).
//   mode 1: x = w dinv v (w null: 1)
//   mode 2: bf = (float) v, xf = w dinvf bf
struct FirstSweep {
  int mode = 0;
  const double* w = nullptr;
  const double* dinv = nullptr;
  double* x = nullptr;
  const float* dinvf = nullptr;
  float *bf = nullptr, *xf = nullptr;
};

// Preconditioner interface: z = M^-1 r.
struct Precond {
  virtual ~Precond() {}
  virtual fvs_status apply(cudaStream_t s, const double* r, double* z) = 0;
  // apply() in two parts: first(z) names the row-wise start (mode 0: none),
  // rest() does what remains once the caller has done it
  virtual FirstSweep first(double* z) { (void)z; return FirstSweep(); }
  virtual fvs_status rest(cudaStream_t s, const double* r, double* z) { return apply(s, r, z); }
  // identifies the state the launches depend on (a captured iteration is
  // replayed only while it is unchanged)
  virtual uint64_t signature() const = 0;
};

// One Krylov iteration captured as a CUDA graph and replayed while the
// operator, vectors and preconditioner stay the same.
struct IterGraph {
  cudaGraphExec_t exec = nullptr;
  uint64_t key = 0;
  unsigned long long kernels = 0;   // launches per replay (for the launch counter)
  bool disabled = false;
  // whole-solve loop: a conditional while-node whose body is one iteration
  cudaGraphExec_t loop = nullptr;
  uint64_t loop_key = 0;
  unsigned long long loop_kernels = 0;
  bool loop_disabled = false;
  ~IterGraph() { reset(); }
  void reset() {
    if (exec) cudaGraphExecDestroy(exec);
    exec = nullptr;
    key = 0;
    if (loop) cudaGraphExecDestroy(loop);
    loop = nullptr;
    loop_key = 0;
  }
};
bool graphs_enabled();

// Jacobi: z = r / (diag + dextra)
struct JacobiPrecond : Precond {
  const Ell* A = nullptr;
  const double* dextra = nullptr;
  const double* dinv = nullptr;   // optional 1 / (diag + dextra), kept by the caller: z = dinv r
  fvs_status apply(cudaStream_t s, const double* r, double* z) override;
  FirstSweep first(double* z) override {
    FirstSweep f;
    if (dinv && A->n > 0) {
      f.mode = 1;
      f.dinv = dinv;
      f.x = z;
    }
    return f;
  }
  fvs_status rest(cudaStream_t s, const double* r, double* z) override { return dinv ? FVS_OK : apply(s, r, z); }
  uint64_t signature() const override {
    return (uint64_t)(uintptr_t)A->diag.p * 31u + (uint64_t)(uintptr_t)dextra * 17u +
           (uint64_t)(uintptr_t)dinv * 13u + (uint64_t)A->n;
  }
};

// Line preconditioner: z = P^-1 r with P the diagonal (plus dextra) and the
// couplings along chains of cells, each cell joined to the neighbours it is
// most strongly coupled to where that choice is mutual (a row's two largest
// off-diagonal magnitudes).  Strongly anisotropic cells (thin in one
// direction) make those chains lines across the thin direction, where
// Jacobi converges slowly.  P restricted to one chain is tridiagonal and is
// solved exactly; cells on no chain take the Jacobi step.  The chains are
// found once from the operator (build) and stored 32 lines to a group,
// position-major within the group, so a warp's loads at one position are
// contiguous; factor() recomputes the tridiagonal factors from the current
// values, apply() does one forward and one backward substitution per line.
struct LinePrecond : Precond {
  const Ell* A = nullptr;
  const double* dextra = nullptr;   // extra diagonal at factor() time (or null)
  int64_t n = 0;
  int w = 0;
  const int32_t* built_from = nullptr;   // column array the chains were found in
  int64_t nlines = 0, ngroups = 0, padded = 0;
  int max_len = 0;
  DBuf<int64_t> goff;      // [ngroups] first entry of each group
  DBuf<int32_t> llen;      // [ngroups * 32] length of each line (0: no line)
  DBuf<int32_t> cell;      // [padded] cell at (group, position, lane)
  DBuf<int8_t> sprev, snext;   // slot of the previous / next cell of the line in the cell's row (-1: none)
  DBuf<double> lo, inv, cp;    // sub-diagonal, 1 / pivot, super-diagonal / pivot
  DBuf<double> yl;             // forward substitution, in line order
  bool ready = false;
  // per row of the operator: sum of its off-diagonal magnitudes, and of those
  // that the lines leave out
  DBuf<double> off, rest;
  bool weighed = false;
  // Whether the lines pay at the given inverse diagonal, which holds the state
  // (latent heat makes the rows of mushy cells several times as dominant): asked
  // in every step, so that a step depends on its state and not on the ones
  // before it (35 us), unless no state could take them at that step size: may()
  // asks for the largest gain, without latent heat, from scale times an operator
  // that does not depend on the state, and is asked once per operator and step
  // size.  With a and b the mean shares of a row's diagonal
  // that Jacobi and the lines leave out, the iterations go down by about
  // sqrt((1 + a)(1 - b) / ((1 - a)(1 + b))), and an iteration costs about 1.4
  // (27-point rows) or twice (face-only rows) as much.  All melt on 128^3
  // thin cells (gain 5): 142 -> 25 inner iterations, 193 -> 158 ms for three
  // steps.  Half frozen on 96^3 (gain 2.5): 107 -> 97 ms, but near the solidus
  // the two solutions, each within the tolerance, differed by up to 2e-8 of u
  // in single cells, so the line is drawn above it.  Below MIN_ROWS a
  // substitution's serial walk costs more than the iterations it saves.
  static constexpr int64_t MIN_ROWS = 65536;
  static constexpr double GAIN_WIDE = 3.0, GAIN_FACE = 4.0;
  static fvs_status may(cudaStream_t s, Reducer& red, const Ell& A, double scale, const double* rcp, const double* V,
                        double idt, bool& use);
  fvs_status worth(cudaStream_t s, Reducer& red, const Ell& A, const double* dinv, bool& use);
  fvs_status build(cudaStream_t s, const Ell& A);
  void drop();     // gives all its memory back
  fvs_status factor(cudaStream_t s);
  fvs_status apply(cudaStream_t s, const double* r, double* z) override;
  uint64_t signature() const override {
    uint64_t h = (uint64_t)n * 131u + (uint64_t)ngroups;
    for (const void* q : {(const void*)goff.p, (const void*)llen.p, (const void*)cell.p, (const void*)lo.p,
                          (const void*)inv.p, (const void*)cp.p, (const void*)yl.p})
      h = h * 1099511628211ULL ^ (uint64_t)(uintptr_t)q;
    return h;
  }
};

struct KrylovWork {
  DBuf<double> r, rh, p, ph, v, sv, sh, t, z, q;
  fvs_status ensure(int64_t n);
};

struct SolveResult {
  int iters = 0;
  double relres = 0.0;
  bool converged = false;
  bool tail_done = false;   // the caller's tail ran on the returned x and its scalars are in Reducer::host
};

// Right-preconditioned BiCGStab on A x = b (x holds the initial guess).
// proj: optional projection applied to the right side and residual updates
// (null-space handling of the pressure system).
// The projection as the mean over one set of rows, where it is that.
struct MeanPart {
  const int32_t* lab = nullptr;    // null: every row
  int want = -1;                   // rows with lab == want (< 0: lab >= 0)
  const double* cnt = nullptr;     // row count on the device (null: n)
};
struct Projector {
  virtual ~Projector() {}
  virtual fvs_status apply(cudaStream_t s, double* v) = 0;
  // 0: nothing to project, 1: the mean over m's rows, 2: neither (use apply)
  virtual int single(MeanPart& m) { (void)m; return 2; }
};

// The residual is measured against max(||b||, bnorm_floor).
//
// A solve whose loop runs on the device waits for the host once: the start's
// scalars, the loop and the true residual are queued together and fetched in
// one copy, the loop being entered only where the start says so.  tail, if
// given, queues what the caller does next with x ahead of that copy (it must
// bear being queued again on a later x; res.tail_done says whether its last
// run holds).  Before, a solve waited three times and the energy pass a
// fourth: a step on 4,096 cells 1.77 -> 1.67 ms, on 184,320 conducting cells
// 2.50 -> 2.44; the kernels in the loop are the same.
//
// rtol is what the iteration works towards; the true residual is judged, and
// a restart decided, by ten times the larger of rtol and asked.
fvs_status bicgstab(cudaStream_t s, Reducer& red, KrylovWork& w, const Ell& A, const double* dextra,
                    Precond& M, const double* b, double* x, double rtol, int maxit,
                    Projector* proj, SolveResult& res, double bnorm_floor = 0.0, IterGraph* graph = nullptr,
                    const std::function<fvs_status()>* tail = nullptr, double asked = 0.0);
fvs_status pcg(cudaStream_t s, Reducer& red, KrylovWork& w, const Ell& A, Precond& M,
               const double* b, double* x, double rtol, int maxit, Projector* proj, SolveResult& res,
               IterGraph* graph = nullptr);

// small vector kernels
fvs_status vcopy(cudaStream_t s, int64_t n, const double* a, double* b);
fvs_status vfill(cudaStream_t s, int64_t n, double v, double* a);

}  // namespace fvs
