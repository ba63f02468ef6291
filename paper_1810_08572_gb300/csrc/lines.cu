// Line preconditioner (declared in la.cuh): tridiagonal solves along chains
// of strongly coupled cells.  Used for the energy system, whose couplings
// across thin cells exceed its mass term several times over, so that
// point-Jacobi needs many Krylov iterations.
#include <cub/device/device_radix_sort.cuh>

#include <cmath>

#include "la.cuh"
#include "reduce.cuh"
#include "scan.cuh"

namespace fvs {

namespace {

constexpr int LCH = 8;          // positions of a line whose loads are in flight together
constexpr int kMaxLine = 512;   // longer chains are cut (a dropped coupling keeps P a valid preconditioner)

// Thomas factors of every line with the current values: row k of a line
// reads lo_k x_{k-1} + b_k x_k + up_k x_{k+1}; pivots d_k = b_k - lo_k cp_{k-1},
// cp_k = up_k / d_k.  One thread per line, the loads of eight positions in
// flight together (16,384 lines of 128 cells: 196 -> 105 us).
__global__ void __launch_bounds__(64) k_line_factor(int64_t ngroups, const int64_t* __restrict__ goff, const int32_t* __restrict__ llen,
                              const int32_t* __restrict__ cell, const int8_t* __restrict__ sprev,
                              const int8_t* __restrict__ snext, int64_t n, const double* __restrict__ val,
                              const double* __restrict__ diag, const double* __restrict__ dextra,
                              double* __restrict__ lo, double* __restrict__ inv, double* __restrict__ cp) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t g = t >> 5;
  if (g >= ngroups) return;
  const int lane = (int)(t & 31);
  const int len = llen[t];
  const int64_t base = goff[g] + lane;
  double cprev = 0.0;
  for (int p0 = 0; p0 < len; p0 += LCH) {
    const int m = min(LCH, len - p0);
    const int64_t i0 = base + (int64_t)p0 * 32;
    double a[LCH], u[LCH], d[LCH];
#pragma unroll
    for (int k = 0; k < LCH; ++k) {
      const int64_t idx = i0 + (k < m ? k : 0) * 32;
      const int32_t c = cell[idx];
      const int kp = sprev[idx], kn = snext[idx];
      a[k] = kp >= 0 ? val[(int64_t)kp * n + c] : 0.0;
      u[k] = kn >= 0 ? val[(int64_t)kn * n + c] : 0.0;
      d[k] = diag[c] + (dextra ? dextra[c] : 0.0);
    }
#pragma unroll
    for (int k = 0; k < LCH; ++k)
      if (k < m) {
        const double piv = d[k] - a[k] * cprev;
        const double iv = piv != 0.0 ? 1.0 / piv : 0.0;
        cprev = u[k] * iv;
        lo[i0 + k * 32] = a[k];
        inv[i0 + k * 32] = iv;
        cp[i0 + k * 32] = cprev;
      }
  }
}

// z = P^-1 r: forward substitution y_k = (r_k - lo_k y_{k-1}) / d_k, then back
// substitution x_k = y_k - cp_k x_{k+1}.  One thread per line, so a launch is
// bound by the latency of its loads: eight positions are loaded together, and
// y is kept in line order, where a warp's stores and loads are contiguous
// (only r is gathered and z scattered by cell).  16,384 lines of 128 cells:
// 57 us.
__global__ void __launch_bounds__(64) k_line_solve(int64_t ngroups, const int64_t* __restrict__ goff,
                                                   const int32_t* __restrict__ llen,
                                                   const int32_t* __restrict__ cell, const double* __restrict__ lo,
                                                   const double* __restrict__ inv, const double* __restrict__ cp,
                                                   const double* __restrict__ r, double* __restrict__ yl,
                                                   double* __restrict__ z) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t g = t >> 5;
  if (g >= ngroups) return;
  const int len = llen[t];
  const int64_t base = goff[g] + (int)(t & 31);
  double y = 0.0;
  for (int p0 = 0; p0 < len; p0 += LCH) {
    const int m = min(LCH, len - p0);
    const int64_t i0 = base + (int64_t)p0 * 32;
    double l[LCH], d[LCH], q[LCH];
#pragma unroll
    for (int k = 0; k < LCH; ++k) {
      const int64_t idx = i0 + (k < m ? k : 0) * 32;
      q[k] = r[cell[idx]];
      l[k] = lo[idx];
      d[k] = inv[idx];
    }
#pragma unroll
    for (int k = 0; k < LCH; ++k)
      if (k < m) {
        y = (q[k] - l[k] * y) * d[k];
        yl[i0 + k * 32] = y;
      }
  }
  double x = 0.0;
  for (int p1 = len; p1 > 0; p1 -= LCH) {
    const int m = min(LCH, p1);
    const int64_t i1 = base + (int64_t)(p1 - 1) * 32;
    double u[LCH], q[LCH];
    int32_t c[LCH];
#pragma unroll
    for (int k = 0; k < LCH; ++k) {
      const int64_t idx = i1 - (k < m ? k : 0) * 32;
      c[k] = cell[idx];
      u[k] = cp[idx];
      q[k] = yl[idx];
    }
#pragma unroll
    for (int k = 0; k < LCH; ++k)
      if (k < m) {
        x = q[k] - u[k] * x;
        z[c[k]] = x;
      }
  }
}

// ---------------------------------------------------------------------------
// the chains, on the device (build_line_layout in lines_host.h is the same
// rule on the host; a test holds the two layouts against one another)
// ---------------------------------------------------------------------------
// two largest off-diagonal couplings of a row (the first slot wins a tie),
// the second only if at least a quarter of the first, and the sum of all;
// the loads of nine slots in flight together.  Magnitudes are compared as bit
// patterns, which order as they do (FP64 compares issue at two lanes a clock);
// a NaN counts as no coupling.
__device__ __forceinline__ void strongest2(int64_t n, int w, const int32_t* __restrict__ col,
                                           const double* __restrict__ val, int64_t i, int32_t& b0, int32_t& b1,
                                           double& m0, double& m1, double& off) {
  constexpr int B = 9;
  constexpr long long INF = 0x7ff0000000000000LL;
  long long q0 = 0, q1 = 0;
  off = 0.0;
  b0 = b1 = -1;
  for (int k0 = 0; k0 < w; k0 += B) {
    int32_t c[B];
    double v[B];
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const bool in = k0 + k < w;
      c[k] = in ? col[(int64_t)(k0 + k) * n + i] : (int32_t)i;
      v[k] = in ? val[(int64_t)(k0 + k) * n + i] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < B; ++k) {
      const int32_t j = c[k];
      const double a = j != (int32_t)i ? fabs(v[k]) : 0.0;
      off += a;
      const long long q = __double_as_longlong(a) > INF ? 0 : __double_as_longlong(a);
      if (q > q0) {
        if (j != b0) { q1 = q0; b1 = b0; }
        q0 = q;
        b0 = j;
      } else if (q > q1 && j != b0) {
        q1 = q;
        b1 = j;
      }
    }
  }
  m0 = __longlong_as_double(q0);
  m1 = __longlong_as_double(q1);
  if (!(m1 >= 0.25 * m0)) { b1 = -1; m1 = 0.0; }
}
__global__ void k_line_best(int64_t n, int w, const int32_t* __restrict__ col, const double* __restrict__ val,
                            int32_t* __restrict__ best) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t b0, b1;
    double m0, m1, o;
    strongest2(n, w, col, val, i, b0, b1, m0, m1, o);
    best[2 * i] = b0;
    best[2 * i + 1] = b1;
  }
}
// couplings that both rows chose
__global__ void k_line_links(int64_t n, const int32_t* __restrict__ best, int32_t* __restrict__ nb) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t l[2] = {-1, -1};
    int q = 0;
    for (int t = 0; t < 2; ++t) {
      const int32_t j = best[2 * i + t];
      if (j >= 0 && (best[2 * (int64_t)j] == (int32_t)i || best[2 * (int64_t)j + 1] == (int32_t)i)) l[q++] = j;
    }
    nb[2 * i] = l[0];
    nb[2 * i + 1] = l[1];
  }
}
// Walks along the chains: node 2 i + d stands at cell i, about to leave it by
// link d.  jump = the node some hops on, hops = how many; a node whose link
// is missing is an end (itself, 0 hops).  Each round doubles the hops.
__global__ void k_line_walk0(int64_t n, const int32_t* __restrict__ nb, int2* __restrict__ walk) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < 2 * n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = (int32_t)(v >> 1), j = nb[v];
    if (j < 0) walk[v] = make_int2((int32_t)v, 0);
    else walk[v] = make_int2(2 * j + (nb[2 * (int64_t)j] == i ? 1 : 0), 1);
  }
}
__global__ void k_line_walk(int64_t n2, const int2* __restrict__ in, int2* __restrict__ out) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n2; v += (int64_t)gridDim.x * blockDim.x) {
    const int2 a = in[v], b = in[a.x];
    out[v] = make_int2(b.x, a.y + b.y);
  }
}
// The same walks with the smallest cell on the way (x: node, y: hops, z: cell).
// After 2^rounds >= n hops a walk that has not ended has gone round a cycle,
// and z is the cycle's smallest cell.
__global__ void k_line_ring0(int64_t n, const int32_t* __restrict__ nb, int4* __restrict__ walk) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < 2 * n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = (int32_t)(v >> 1), j = nb[v];
    if (j < 0) walk[v] = make_int4((int32_t)v, 0, i, 0);
    else walk[v] = make_int4(2 * j + (nb[2 * (int64_t)j] == i ? 1 : 0), 1, min(i, j), 0);
  }
}
__global__ void k_line_ring(int64_t n2, const int4* __restrict__ in, int4* __restrict__ out) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n2; v += (int64_t)gridDim.x * blockDim.x) {
    const int4 a = in[v], b = in[a.x];
    out[v] = make_int4(b.x, a.y + b.y, min(a.z, b.z), 0);
  }
}
// a cycle is cut at its smallest cell, whose second link goes (hops doubled in
// every round where the walk has not ended; an ended one has fewer)
__global__ void k_line_cut(int64_t n, const int4* __restrict__ walk, int hops, int32_t* __restrict__ nb) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int4 a = walk[2 * i];
    if (a.y != hops || a.z != (int32_t)i) continue;
    const int64_t q = nb[2 * i + 1];
    nb[2 * i + 1] = -1;
    nb[2 * q + (nb[2 * q] == (int32_t)i ? 0 : 1)] = -1;
  }
}
// place of every cell: head cell of its chain (the end with the smaller id),
// position, and at the head the number of lines the chain is cut into.  A cell
// whose walks have not both ended flags open.
constexpr int WALK_ROUNDS = 12;   // chains of up to 4,096 links
__global__ void k_line_place(int64_t n, const int32_t* __restrict__ nb, const int2* __restrict__ walk, int max_line,
                             int32_t* __restrict__ head, int32_t* __restrict__ place, int32_t* __restrict__ len,
                             int32_t* __restrict__ cnt, int32_t* __restrict__ open) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int2 a = walk[2 * i], b = walk[2 * i + 1];
    int32_t h = (int32_t)i, p = 0, m = 1;
    int dir = 0;                 // link towards the head
    if (nb[a.x] < 0 && nb[b.x] < 0) {
      const int32_t ea = a.x >> 1, eb = b.x >> 1;
      dir = ea <= eb ? 0 : 1;
      h = dir == 0 ? ea : eb;
      p = dir == 0 ? a.y : b.y;
      m = a.y + b.y + 1;
    } else {
      *open = 1;
    }
    head[i] = h;
    place[i] = p * 2 + dir;
    len[i] = m;
    cnt[i] = p == 0 ? (m + max_line - 1) / max_line : 0;
  }
}
// lengths of the lines, by line; sort keys put longer lines first
__global__ void k_line_lengths(int64_t n, const int32_t* __restrict__ place, const int32_t* __restrict__ len,
                               const int32_t* __restrict__ first, int max_line, int32_t* __restrict__ key,
                               int32_t* __restrict__ id) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if (place[i] >> 1) continue;
    const int m = len[i], nl = (m + max_line - 1) / max_line;
    for (int q = 0; q < nl; ++q) {
      key[first[i] + q] = max_line - min(max_line, m - q * max_line);
      id[first[i] + q] = first[i] + q;
    }
  }
}
__global__ void k_line_groups(int nl, int ng, int max_line, const int32_t* __restrict__ key,
                              const int32_t* __restrict__ id, int32_t* __restrict__ rank, int32_t* __restrict__ llen,
                              int32_t* __restrict__ glen) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ng * 32; t += gridDim.x * blockDim.x) {
    llen[t] = t < nl ? max_line - key[t] : 0;
    if (t < nl) rank[id[t]] = t;
    if ((t & 31) == 0) glen[t >> 5] = max_line - key[t];
  }
}
__global__ void k_line_offsets(int ng, const int32_t* __restrict__ sum, int64_t* __restrict__ goff) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += gridDim.x * blockDim.x) goff[g] = 32LL * sum[g];
}
__global__ void k_line_fill(int64_t n, int w, const int32_t* __restrict__ col, const int32_t* __restrict__ nb,
                            const int32_t* __restrict__ head, const int32_t* __restrict__ place,
                            const int32_t* __restrict__ first, const int32_t* __restrict__ rank,
                            const int32_t* __restrict__ llen, const int64_t* __restrict__ goff, int max_line,
                            int32_t* __restrict__ cell, int8_t* __restrict__ sprev, int8_t* __restrict__ snext) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = place[i] >> 1, dir = place[i] & 1, pos = p % max_line;
    const int32_t t = rank[first[head[i]] + p / max_line];
    const int64_t e = goff[t >> 5] + (int64_t)pos * 32 + (t & 31);
    const int32_t jp = pos > 0 ? nb[2 * i + dir] : -1;
    const int32_t jn = pos + 1 < llen[t] ? nb[2 * i + 1 - dir] : -1;
    int8_t sp = -1, sn = -1;
    for (int k = w - 1; k >= 0; --k) {
      const int32_t j = col[(int64_t)k * n + i];
      if (j == jp) sp = (int8_t)k;
      if (j == jn) sn = (int8_t)k;
    }
    cell[e] = (int32_t)i;
    sprev[e] = jp >= 0 ? sp : (int8_t)-1;
    snext[e] = jn >= 0 ? sn : (int8_t)-1;
  }
}
// sums of a row's off-diagonal magnitudes, and of the same without its chain
// couplings: what Jacobi and the lines leave out
__global__ void k_line_sums(int64_t n, int w, const int32_t* __restrict__ col, const double* __restrict__ val,
                            double* __restrict__ off, double* __restrict__ rest) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t b0, b1;
    double m0, m1, o;
    strongest2(n, w, col, val, i, b0, b1, m0, m1, o);
    off[i] = o;
    rest[i] = o - m0 - m1;
  }
}
// the same over the rows' diagonals of the energy system without latent heat,
// summed (an operator of w slots, times scale)
__global__ void __launch_bounds__(RB) k_line_bound(int64_t n, int w, const int32_t* __restrict__ col,
                                                   const double* __restrict__ val, const double* __restrict__ diag,
                                                   double scale, const double* __restrict__ rcp,
                                                   const double* __restrict__ V, double idt, double* part,
                                                   unsigned int* ticket, double* sc, int s0, int s1) {
  double x = 0.0, y = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    int32_t b0, b1;
    double m0, m1, o;
    strongest2(n, w, col, val, i, b0, b1, m0, m1, o);
    const double d = scale * fabs(diag[i]) + rcp[i] * V[i] * idt;
    if (d > 0.0) {
      const double q = scale / d;
      x = fma(o, q, x);
      y = fma(o - m0 - m1, q, y);
    }
  }
  if (grid_fold<OpSum, 2>(x, y, part, ticket)) {
    sc[s0] = x;
    sc[s1] = y;
  }
}
// both times the rows' inverse diagonals, summed (rows without a diagonal left out)
__global__ void __launch_bounds__(RB) k_line_weight(int64_t n, const double* __restrict__ off,
                                                    const double* __restrict__ rest, const double* __restrict__ dinv,
                                                    double* part, unsigned int* ticket, double* sc, int s0, int s1) {
  double x = 0.0, y = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)RB + threadIdx.x; i < n; i += (int64_t)gridDim.x * RB) {
    const double d = fabs(dinv[i]);
    if (d < 1e300) {
      x = fma(off[i], d, x);
      y = fma(rest[i], d, y);
    }
  }
  if (grid_fold<OpSum, 2>(x, y, part, ticket)) {
    sc[s0] = x;
    sc[s1] = y;
  }
}

}  // namespace

// from the sums in S_TMP0 and S_TMP1
static fvs_status line_gain(cudaStream_t s, Reducer& red, int64_t n, int w, bool& use) {
  FVS_TRY(red.fetch(s));
  const double a = std::min(0.999, red.host[S_TMP0] / (double)n);
  const double b = std::max(0.0, std::min(a, red.host[S_TMP1] / (double)n));
  use = std::sqrt((1.0 + a) * (1.0 - b) / ((1.0 - a) * (1.0 + b))) >
        (w > 7 ? LinePrecond::GAIN_WIDE : LinePrecond::GAIN_FACE);
  return FVS_OK;
}

fvs_status LinePrecond::may(cudaStream_t s, Reducer& red, const Ell& Ain, double scale, const double* rcp,
                            const double* V, double idt, bool& use) {
  use = false;
  if (Ain.n < MIN_ROWS || Ain.w < 3) return FVS_OK;
  k_line_bound<<<red.grid(Ain.n), RB, 0, s>>>(Ain.n, Ain.w, Ain.col, Ain.val, Ain.diag, scale, rcp, V, idt, red.part,
                                              red.ticket, red.sc, S_TMP0, S_TMP1);
  FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return line_gain(s, red, Ain.n, Ain.w, use);
}

fvs_status LinePrecond::worth(cudaStream_t s, Reducer& red, const Ell& Ain, const double* dinv, bool& use) {
  use = false;
  if (Ain.n < MIN_ROWS || Ain.w < 3) return FVS_OK;
  if (!weighed) {
    FVS_TRY(off.alloc(Ain.n));
    FVS_TRY(rest.alloc(Ain.n));
    k_line_sums<<<stride_grid(Ain.n, 256), 256, 0, s>>>(Ain.n, Ain.w, Ain.col, Ain.val, off, rest);
    FVS_COUNT_LAUNCH();
    weighed = true;
  }
  k_line_weight<<<red.vgrid(Ain.n), RB, 0, s>>>(Ain.n, off, rest, dinv, red.part, red.ticket, red.sc, S_TMP0, S_TMP1);
  FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return line_gain(s, red, Ain.n, Ain.w, use);
}

fvs_status LinePrecond::build(cudaStream_t s, const Ell& Ain) {
  ready = false;
  A = &Ain;
  n = Ain.n;
  w = Ain.w;
  built_from = Ain.col.p;
  if (n <= 0) return FVS_OK;
  if (n > 1073741823LL) {
    set_error("line preconditioner: %lld rows exceed 31-bit node ids", (long long)n);
    return FVS_ERR_ARG;
  }
  const int g = stride_grid(n, 256);
  DBuf<int32_t> nb, head, place, len, cnt, first;
  FVS_TRY(nb.alloc(2 * (size_t)n));
  {
    DBuf<int32_t> best;
    FVS_TRY(best.alloc(2 * (size_t)n));
    k_line_best<<<g, 256, 0, s>>>(n, w, Ain.col, Ain.val, best); FVS_COUNT_LAUNCH();
    k_line_links<<<g, 256, 0, s>>>(n, best, nb); FVS_COUNT_LAUNCH();
    FVS_LAUNCH_CHECK();
  }
  FVS_TRY(head.alloc(n)); FVS_TRY(place.alloc(n)); FVS_TRY(len.alloc(n));
  FVS_TRY(cnt.alloc((size_t)n + 1)); FVS_TRY(first.alloc((size_t)n + 1));
  ScanWork sw;
  int32_t nl = 0, open = 0;
  const int g2 = stride_grid(2 * n, 256);
  // places of all cells, the number of lines, and whether a walk was too short
  auto walk = [&](int rounds) -> fvs_status {
    DBuf<int2> wa, wb;
    DBuf<int32_t> op;
    FVS_TRY(wa.alloc(2 * (size_t)n)); FVS_TRY(wb.alloc(2 * (size_t)n)); FVS_TRY(op.alloc(1));
    k_line_walk0<<<g2, 256, 0, s>>>(n, nb, wa); FVS_COUNT_LAUNCH();
    for (int q = 0; q < rounds; ++q) {
      k_line_walk<<<g2, 256, 0, s>>>(2 * n, (q & 1) ? wb.p : wa.p, (q & 1) ? wa.p : wb.p);
      FVS_COUNT_LAUNCH();
    }
    FVS_TRY(cnt.zero(s)); FVS_TRY(op.zero(s));
    k_line_place<<<g, 256, 0, s>>>(n, nb, (rounds & 1) ? wb.p : wa.p, kMaxLine, head, place, len, cnt, op);
    FVS_COUNT_LAUNCH();
    FVS_LAUNCH_CHECK();
    FVS_TRY(exclusive_scan(s, sw, n + 1, cnt, first));
    FVS_CUDA(cudaMemcpyAsync(&nl, first.p + n, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    FVS_CUDA(cudaMemcpyAsync(&open, op.p, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    FVS_CUDA(cudaStreamSynchronize(s));
    return FVS_OK;
  };
  FVS_TRY(walk(WALK_ROUNDS));
  if (open) {
    // cycles, or chains of more links than the rounds reach: cut the cycles,
    // then walk chains of any length
    int rounds = 0;
    while ((1LL << rounds) < n) ++rounds;   // (2^30 hops at most: n is bounded above)
    {
      DBuf<int4> wa, wb;
      FVS_TRY(wa.alloc(2 * (size_t)n)); FVS_TRY(wb.alloc(2 * (size_t)n));
      k_line_ring0<<<g2, 256, 0, s>>>(n, nb, wa); FVS_COUNT_LAUNCH();
      for (int q = 0; q < rounds; ++q) {
        k_line_ring<<<g2, 256, 0, s>>>(2 * n, (q & 1) ? wb.p : wa.p, (q & 1) ? wa.p : wb.p);
        FVS_COUNT_LAUNCH();
      }
      k_line_cut<<<g, 256, 0, s>>>(n, (rounds & 1) ? wb.p : wa.p, 1 << rounds, nb); FVS_COUNT_LAUNCH();
      FVS_LAUNCH_CHECK();
    }
    FVS_TRY(walk(rounds));
  }
  nlines = nl;
  ngroups = (nl + 31) / 32;
  const int ng = (int)ngroups;
  DBuf<int32_t> key, id, key2, id2, rank, glen, gsum;
  FVS_TRY(key.alloc(nl)); FVS_TRY(id.alloc(nl)); FVS_TRY(key2.alloc(nl)); FVS_TRY(id2.alloc(nl));
  FVS_TRY(rank.alloc(nl)); FVS_TRY(glen.alloc((size_t)ng + 1)); FVS_TRY(gsum.alloc((size_t)ng + 1));
  FVS_TRY(goff.alloc((size_t)ng + 1)); FVS_TRY(llen.alloc((size_t)ng * 32 + 1));
  k_line_lengths<<<g, 256, 0, s>>>(n, place, len, first, kMaxLine, key, id); FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  {
    size_t bytes = 0;
    FVS_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, bytes, key.p, key2.p, id.p, id2.p, nl, 0, 10, s));
    DBuf<char> tmp;
    FVS_TRY(tmp.alloc(bytes + 1));
    FVS_CUDA(cub::DeviceRadixSort::SortPairs(tmp.p, bytes, key.p, key2.p, id.p, id2.p, nl, 0, 10, s));
  }
  FVS_TRY(glen.zero(s));
  k_line_groups<<<stride_grid((int64_t)ng * 32, 256), 256, 0, s>>>(nl, ng, kMaxLine, key2, id2, rank, llen, glen);
  FVS_COUNT_LAUNCH();
  FVS_TRY(exclusive_scan(s, sw, ng + 1, glen, gsum));
  k_line_offsets<<<stride_grid(ng + 1, 256), 256, 0, s>>>(ng + 1, gsum, goff); FVS_COUNT_LAUNCH();
  int32_t total = 0, longest = 0;
  FVS_CUDA(cudaMemcpyAsync(&total, gsum.p + ng, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  FVS_CUDA(cudaMemcpyAsync(&longest, llen.p, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  FVS_CUDA(cudaStreamSynchronize(s));
  padded = 32LL * total;
  max_len = longest;
  FVS_TRY(cell.alloc(padded + 1));
  FVS_TRY(sprev.alloc(padded + 1));
  FVS_TRY(snext.alloc(padded + 1));
  FVS_TRY(lo.alloc(padded + 1));
  FVS_TRY(inv.alloc(padded + 1));
  FVS_TRY(cp.alloc(padded + 1));
  FVS_TRY(yl.alloc(padded + 1));
  FVS_CUDA(cudaMemsetAsync(cell.p, 0, (padded + 1) * sizeof(int32_t), s));   // padding is never visited
  k_line_fill<<<g, 256, 0, s>>>(n, w, Ain.col, nb, head, place, first, rank, llen, goff, kMaxLine, cell, sprev, snext);
  FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  ready = true;
  return FVS_OK;
}

void LinePrecond::drop() {
  ready = weighed = false;
  goff.release();
  llen.release();
  cell.release();
  sprev.release();
  snext.release();
  for (DBuf<double>* b : {&lo, &inv, &cp, &yl, &off, &rest}) b->release();
}

fvs_status LinePrecond::factor(cudaStream_t s) {
  if (!ready || n <= 0) return FVS_OK;
  const int64_t threads = ngroups * 32;
  k_line_factor<<<grid_for(threads, 64), 64, 0, s>>>(ngroups, goff, llen, cell, sprev, snext, n, A->val,
                                                      A->diag, dextra, lo, inv, cp);
  FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

fvs_status LinePrecond::apply(cudaStream_t s, const double* r, double* z) {
  if (n <= 0) return FVS_OK;
  const int64_t threads = ngroups * 32;
  k_line_solve<<<grid_for(threads, 64), 64, 0, s>>>(ngroups, goff, llen, cell, lo, inv, cp, r, yl, z);
  FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

}  // namespace fvs

using namespace fvs;

extern "C" __attribute__((visibility("default"))) fvs_status fvs_line_layout(
    const int32_t* col, const double* val, int64_t n, int32_t w, int64_t* sizes, int64_t cap_groups,
    int64_t cap_padded, int64_t* goff, int32_t* llen, int32_t* cell, int8_t* sprev, int8_t* snext) {
  if (!col || !val || !sizes || n < 1 || w < 1 || w > 127 || n > INT32_MAX / 2 / w) {
    set_error("fvs_line_layout: bad argument");
    return FVS_ERR_ARG;
  }
  for (int64_t e = 0; e < n * w; ++e)
    if (col[e] < 0 || col[e] >= n) {
      set_error("fvs_line_layout: column %d outside the rows", (int)col[e]);
      return FVS_ERR_ARG;
    }
  cudaStream_t st = nullptr;
  FVS_CUDA(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
  auto run = [&]() -> fvs_status {
    AllocStream as(st);
    Ell A;
    LinePrecond P;
    FVS_TRY(A.alloc(n, w));
    FVS_CUDA(cudaMemcpyAsync(A.col.p, col, (size_t)n * w * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    FVS_CUDA(cudaMemcpyAsync(A.val.p, val, (size_t)n * w * sizeof(double), cudaMemcpyHostToDevice, st));
    FVS_TRY(P.build(st, A));
    sizes[0] = P.nlines;
    sizes[1] = P.ngroups;
    sizes[2] = P.padded;
    sizes[3] = P.max_len;
    if (goff && llen && cell && sprev && snext && cap_groups >= P.ngroups && cap_padded >= P.padded) {
      FVS_CUDA(cudaMemcpyAsync(goff, P.goff.p, (P.ngroups + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
      FVS_CUDA(cudaMemcpyAsync(llen, P.llen.p, P.ngroups * 32 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
      FVS_CUDA(cudaMemcpyAsync(cell, P.cell.p, P.padded * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
      FVS_CUDA(cudaMemcpyAsync(sprev, P.sprev.p, P.padded, cudaMemcpyDeviceToHost, st));
      FVS_CUDA(cudaMemcpyAsync(snext, P.snext.p, P.padded, cudaMemcpyDeviceToHost, st));
    }
    FVS_CUDA(cudaStreamSynchronize(st));
    return FVS_OK;
  };
  const fvs_status r = run();
  cudaStreamSynchronize(st);
  cudaStreamDestroy(st);
  return r;
}
