// Contour integration for many independent problems in one persistent launch.
//
// Every problem p has its own sparse A_p (B = I), its own contour (nodes
// z_pj, weights w_pj, j < ne) and its own subspace size m_p <= m0.  One
// cooperative kernel solves, for every problem, node and column at once,
//     (z_pj I - A_p) X_pj = Y_p           (eq. qr)   and then
//     (z_pj I - A_p)^H Xh_pj = Yh_p       (eq. ql),
// and forms Q_p = sum_j w_pj X_pj and Qh_p = sum_j conj(w_pj) Xh_pj (fixed
// node order).  The shifted systems are solved by iterative refinement:
// the residual R = Y - (z I - A) X in FP64 arithmetic, a correction D from
// Jacobi-preconditioned BiCGStab in T (float: the single-precision sweeps;
// double: the plain form, one refinement step), X += D.  The Krylov scalars
// of every (problem, node, column) system are its own; converged systems
// are frozen.  All phases of all refinement steps and Krylov iterations run
// inside the one launch, separated by a grid barrier with a bounded wait.
//
// An iteration is eight phases, a grid barrier after each: v = (z I - A) y with
// (rh, v); alpha; s and z; t = (z I - A) z with (t, s), (t, t); omega; d and r
// with (r, r), (rh, r); beta and the stopping test; p and y.  ((rh, r) is summed
// itself: from (rh, s) - omega (rh, t) the updates would be one pass over the
// blocks and a barrier less, 1 to 10 % of an iteration on 0.3 to 3.5 million rows,
// but FP32 sums would cancel in it.)  The products read the matrix in the sweeps' precision (values
// converted once, at set-up: an FP64-to-FP32 conversion costs a warp 64 cycles,
// and one for every entry, node and column was most of an iteration), a tile's
// rows padded to one length in shared memory, two rows at a time so that some
// eighteen gathers are in flight; the inverse diagonals come from set-up too.
// Six problems, 15 700 rows, 8 nodes x 32 columns: 895 us an iteration before,
// 388 now; 16 problems, 336 000 rows, 8 nodes x 48 columns: 22.6 and 9.5 ms; 64
// problems, 3.45 million rows: 208 and 85 ms.
//
// Layout.  Rows of all problems are concatenated; problem p owns rows
// [off_p, off_p + n_p).  A right-hand-side / output block (Y, Q) holds
// problem p's n_p x m_p row-major block at element offset off_p * m0.  A
// node-major block (X and the Krylov blocks) holds problem p's ne blocks of
// n_p x m_p at element offset ne * off_p * m0: entry (j, i, c) at
// ne*off_p*m0 + (j*n_p + i)*m_p + c.  Work is cut into tiles of consecutive
// rows of one problem; each CTA takes tiles grid-stride, each thread takes
// systems (j, c) and walks the tile's rows, so that a warp reads consecutive
// columns of one row (coalesced) and keeps its partial dot products in
// registers; per-tile partials are reduced per system in fixed tile order.
#include "kernels.h"

namespace {

template <typename T>
__device__ __forceinline__ cx<T> crecip(cx<T> a) {
  // 1/a with one scaling to keep |a|^2 in range
  const T s = fmax(fabs(a.re), fabs(a.im));
  if (!(s > 0)) return mk<T>(0, 0);
  const T ar = a.re / s, ai = a.im / s;
  const T d = ar * ar + ai * ai;
  return mk<T>(ar / (d * s), -ai / (d * s));
}

// grid barrier: arrival counter + generation word; bounded wait
__device__ bool grid_bar(unsigned *bar, int *abort_flag, int *err, long long limit) {
  __syncthreads();
  __shared__ int ok;
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned *vgen = bar + 1;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u);
    if (arrived == gridDim.x - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == gen) {
        if (*(volatile int *)abort_flag) { ok = 0; break; }
        if (clock64() - t0 > limit) {
          atomicOr(err, DEVERR_TIMEOUT);
          atomicExch(abort_flag, 1);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
    if (*(volatile int *)abort_flag) ok = 0;
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace

template <typename T>
struct BatchKernelArgs {
  int nprob, ne, m0, ntiles, side0, side1;
  const BatchProb *prob;
  const BatchTile *tiles;
  const cxd *Y, *Yh;
  cxd *Q, *Qh;
  const cx<T> *kinv;     // 1 / (z_j - a_ii): problem p's ne x n_p at ne * off_p
  cxd *X;
  cx<T> *r, *rh, *p, *v, *y, *s, *z, *t, *d;
  cx<T> *part;           // ntiles x 2 x PS partial dots
  double *partd;         // ntiles x PS partial |r|^2 (FP64 residual)
  double *partb;         // ntiles x m0 partial |Y_c|^2
  BatchScal sc;
  unsigned *bar;
  int *ctl;              // [0] abort, [1..4] counters
  BatchStats *stats;
  int *err;
  double tol, tau_min;
  int nsteps, kmax;
  long long spin_limit;
};

namespace {

constexpr int kEll = 2304;   // staged entries (256 rows of nine)

// Rows of a tile in shared memory, padded to K entries (own row, value zero).
template <typename T>
struct TileEll {
  int ci[kEll];
  T v[2 * kEll];             // real values, or interleaved complex ones
  int K, tile, side;         // K < 0: the rows do not fit, read the CSR arrays
};

template <typename T>
__device__ void stage_tile(TileEll<T> &e, const BatchTile &tl, int ti, const BatchProb &pr, int side) {
  if (e.tile == ti && e.side == side) return;  // uniform: set before the last barrier
  __syncthreads();
  const CsrView &M = side == 0 ? pr.A : pr.AH;
  const int rows = tl.r1 - tl.r0;
  __shared__ int kmax;
  if (threadIdx.x == 0) kmax = 0;
  __syncthreads();
  for (int r = threadIdx.x; r < rows; r += blockDim.x) atomicMax(&kmax, M.rowptr[tl.r0 + r + 1] - M.rowptr[tl.r0 + r]);
  __syncthreads();
  const int K = kmax;
  const bool fits = rows * K <= kEll;
  if (fits) {
    const T *vals = reinterpret_cast<const T *>(side == 0 ? pr.vA : pr.vAH);
    for (int idx = threadIdx.x; idx < rows * K; idx += blockDim.x) {
      const int r = idx / K, k = idx - r * K;
      const int b = M.rowptr[tl.r0 + r], cnt = M.rowptr[tl.r0 + r + 1] - b;
      e.ci[idx] = k < cnt ? M.colind[b + k] : tl.r0 + r;
      if (M.cplx) {
        e.v[2 * idx] = k < cnt ? vals[2 * ((size_t)b + k)] : T(0);
        e.v[2 * idx + 1] = k < cnt ? vals[2 * ((size_t)b + k) + 1] : T(0);
      } else {
        e.v[idx] = k < cnt ? vals[(size_t)b + k] : T(0);
      }
    }
  }
  if (threadIdx.x == 0) {
    e.K = fits ? K : -1;
    e.tile = ti;
    e.side = side;
  }
  __syncthreads();
}

// acc -= sum_k a_ik x[col_k]
template <typename T, bool CPLX>
__device__ __forceinline__ void row_fms(cx<T> &acc, const TileEll<T> &e, int idx, cx<T> x) {
  if (CPLX) {
    cfms(acc, mk<T>(e.v[2 * idx], e.v[2 * idx + 1]), x);
  } else {
    const T v = e.v[idx];
    acc.re = fma(-v, x.re, acc.re);
    acc.im = fma(-v, x.im, acc.im);
  }
}

// out_i = (z I - A) x for the rows of a tile (system column c, row stride m);
// use(i, out_i) for every row in order
template <typename T, bool CPLX, typename F>
__device__ __forceinline__ void tile_product(const TileEll<T> &e, int r0, int r1, cx<T> zj, const cx<T> *x, int m, int c, F use) {
  const int K = e.K;
  int i = r0;
  for (; i + 1 < r1; i += 2) {
    const int b0 = (i - r0) * K, b1 = b0 + K;
    cx<T> a0 = zj * x[(size_t)i * m + c], a1 = zj * x[(size_t)(i + 1) * m + c];
#pragma unroll 3
    for (int k = 0; k < K; ++k) {
      const cx<T> x0 = x[(size_t)e.ci[b0 + k] * m + c], x1 = x[(size_t)e.ci[b1 + k] * m + c];
      row_fms<T, CPLX>(a0, e, b0 + k, x0);
      row_fms<T, CPLX>(a1, e, b1 + k, x1);
    }
    use(i, a0);
    use(i + 1, a1);
  }
  if (i < r1) {
    const int b0 = (i - r0) * K;
    cx<T> a0 = zj * x[(size_t)i * m + c];
    for (int k = 0; k < K; ++k) row_fms<T, CPLX>(a0, e, b0 + k, x[(size_t)e.ci[b0 + k] * m + c]);
    use(i, a0);
  }
}
template <typename T, typename F>
__device__ __forceinline__ void product(const TileEll<T> &e, const BatchProb &pr, const BatchTile &tl, int side, cx<T> zj,
                                        const cx<T> *x, int m, int c, F use) {
  const CsrView &M = side == 0 ? pr.A : pr.AH;
  if (e.K >= 0) {
    if (M.cplx)
      tile_product<T, true>(e, tl.r0, tl.r1, zj, x, m, c, use);
    else
      tile_product<T, false>(e, tl.r0, tl.r1, zj, x, m, c, use);
    return;
  }
  for (int i = tl.r0; i < tl.r1; ++i) {  // rows too long for the staging area
    cx<T> acc = zj * x[(size_t)i * m + c];
    for (int64_t k = M.rowptr[i]; k < M.rowptr[i + 1]; ++k)
      cfms(acc, ccast<T>(csr_val(M, k)), x[(size_t)M.colind[k] * m + c]);
    use(i, acc);
  }
}

// Every system once: eight lanes of a warp to a system (they share the sums
// over the problem's tiles), four consecutive systems to a warp.
// f(s, p, q, c, sub, problem) with sub the lane of the eight.
template <typename T, typename F>
__device__ void for_systems(const BatchKernelArgs<T> &a, F f) {
  const int PS = a.ne * a.m0;
  const int total = a.nprob * PS;
  const int lane = threadIdx.x & 31;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
  for (int s4 = w * 4; s4 < total; s4 += nw * 4) {
    const int s = s4 + (lane & 3);
    const int p = s < total ? s / PS : 0, q = s - p * PS;
    const BatchProb &pr = a.prob[p];
    const int c = q % a.m0;
    const bool live = s < total && pr.active && c < pr.m;
    f(live, s, p, q, c, lane >> 2, pr);
  }
}
__device__ __forceinline__ double sum8(double v) {
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ cxd sum8(cxd v) { return mk(sum8(v.re), sum8(v.im)); }

// Loop over the tiles of active problems; body(tile index, tile, problem, j, c,
// sys) is called once per (tile, system) for the thread's systems.  STAGE: the
// tile's rows of side `side` are in e.
template <typename T, bool ONLY_ACTIVE, bool STAGE, typename F>
__device__ void for_tile_systems(const BatchKernelArgs<T> &a, TileEll<T> &e, int side, F f) {
  const int PS = a.ne * a.m0;
  for (int ti = blockIdx.x; ti < a.ntiles; ti += gridDim.x) {
    const BatchTile tl = a.tiles[ti];
    const BatchProb &pr = a.prob[tl.p];
    if (!pr.active) continue;
    if (STAGE) stage_tile(e, tl, ti, pr, side);
    const int m = pr.m;
    const int P = a.ne * m;
    for (int q = threadIdx.x; q < P; q += blockDim.x) {
      const int j = q / m, c = q - j * m;
      const int sys = tl.p * PS + j * a.m0 + c;
      if (ONLY_ACTIVE && !a.sc.act[sys]) continue;
      f(ti, tl, pr, j, c, sys);
    }
  }
}

}  // namespace

// LEAN: FP32 in 64 registers (120 bytes of spills), for 1024 threads an SM; else
// CTAs of at most 256 threads with up to 128 (116 used), which the short phases
// of few rows take better.  336 000 rows in 16 problems: 9.5 ms an iteration, 12.2
// without the lean form; a solve of six problems, 13 000 rows: 91 ms, 99 without
// the other.  FP64 takes 128 either way and has one form.
template <typename T, bool LEAN>
__global__ void __launch_bounds__(LEAN ? 512 : 256, LEAN && sizeof(T) == 8 ? 1 : 2) k_batch_filter(BatchKernelArgs<T> a) {
  __shared__ TileEll<T> ell;
  const int PS = a.ne * a.m0;
  int *abort_flag = a.ctl;
  if (threadIdx.x == 0) ell.tile = -1;
  __syncthreads();
  for (int side = a.side0; side <= a.side1; ++side) {
    const cxd *BYb = side == 0 ? a.Y : a.Yh;
    cxd *Qb = side == 0 ? a.Q : a.Qh;
    int kry_total = 0, steps_done = 0;
    for (int step = 0;; ++step) {
      // ---- R = BY - (z I - A) X in FP64; Krylov start r = rh = p = R, y = K^{-1} p, d = 0 ----
      for_tile_systems<T, false, false>(a, ell, side, [&](int ti, const BatchTile &tl, const BatchProb &pr, int j, int c, int sys) {
        const int n = pr.n, m = pr.m;
        const size_t nb = (size_t)a.ne * pr.off * a.m0 + (size_t)j * n * m;
        const cxd zj = side == 0 ? pr.z[j] : conj(pr.z[j]);
        const CsrView &M = side == 0 ? pr.A : pr.AH;
        const cxd *Xb = a.X + nb;
        const cxd *By = BYb + pr.off * a.m0;
        const cx<T> *ki = a.kinv + (size_t)a.ne * pr.off + (size_t)j * n;
        const bool done = step > 0 && !a.sc.act0[sys];
        double acc2 = 0.0, accb = 0.0;
        for (int i = tl.r0; i < tl.r1; ++i) {
          const cxd b = By[(size_t)i * m + c];
          if (step == 0 && j == 0) accb += abs2(b);
          if (done) continue;
          cxd rr = b;
          if (step > 0) {
            cfms(rr, zj, Xb[(size_t)i * m + c]);
            const int kb = M.rowptr[i], ke = M.rowptr[i + 1];
            if (M.cplx) {
              for (int k = kb; k < ke; ++k) cfma(rr, csr_val(M, k), Xb[(size_t)M.colind[k] * m + c]);
            } else {
#pragma unroll 4
              for (int k = kb; k < ke; ++k) {
                const cxd x = Xb[(size_t)M.colind[k] * m + c];
                const double v = M.val[k];
                rr.re = fma(v, x.re, rr.re);
                rr.im = fma(v, x.im, rr.im);
              }
            }
          } else {
            a.X[nb + (size_t)i * m + c] = mk(0.0, 0.0);
          }
          const cx<T> ro = ccast<T>(rr);
          const size_t e = nb + (size_t)i * m + c;
          const cx<T> kv = side == 0 ? ki[i] : conj(ki[i]);
          a.r[e] = ro;
          a.rh[e] = ro;
          a.p[e] = ro;
          a.y[e] = kv * ro;
          a.d[e] = mk<T>(0, 0);
          acc2 += abs2(rr);
        }
        a.partd[(size_t)ti * PS + j * a.m0 + c] = acc2;
        if (step == 0 && j == 0) a.partb[(size_t)ti * a.m0 + c] = accb;
      });
      if (blockIdx.x == 0 && threadIdx.x == 0) a.ctl[1] = a.ctl[2] = a.ctl[3] = 0;
      if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
      // ---- refinement check: relative residual per system ----
      for_systems(a, [&](bool live, int s, int p, int q, int c, int sub, const BatchProb &pr) {
        const bool open = live && (step == 0 || a.sc.act0[s]);
        double b = 0.0, r2 = 0.0;
        if (live && step == 0)
          for (int ti = pr.tb + sub; ti < pr.te; ti += 8) b += a.partb[(size_t)ti * a.m0 + c];
        if (open)
          for (int ti = pr.tb + sub; ti < pr.te; ti += 8) r2 += a.partd[(size_t)ti * PS + q];
        b = sum8(b);
        r2 = sum8(r2);
        if (!live || sub) return;
        if (step == 0) {
          if (q < a.m0) a.sc.bn2[p * a.m0 + c] = b;
          a.sc.act0[s] = 1;
        } else {
          b = a.sc.bn2[p * a.m0 + c];
        }
        if (!open) {
          a.sc.act[s] = 0;
          return;
        }
        const double rel = b > 0 ? sqrt(r2 / b) : sqrt(r2);
        a.sc.rel[s] = rel;
        if (rel <= a.tol || !(rel == rel) || step >= a.nsteps) {
          a.sc.act0[s] = 0;
          a.sc.act[s] = 0;
          return;
        }
        // Krylov start: rho = (rh, r) = |r|^2; tolerance relative to |r0|
        a.sc.rho[s] = mk(r2, 0.0);
        a.sc.alpha[s] = mk(1.0, 0.0);
        a.sc.omega[s] = mk(1.0, 0.0);
        const double want = 0.5 * a.tol * (b > 0 ? sqrt(b) : 1.0);
        const double tau = fmax(a.tau_min, want / sqrt(r2));
        a.sc.stop2[s] = tau * tau * r2;
        a.sc.act[s] = 1;
        atomicAdd(&a.ctl[1], 1);
      });
      if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
      const int nact = *(volatile int *)&a.ctl[1];
      if (nact == 0 || step >= a.nsteps) { steps_done = step; break; }
      // ---- Jacobi-preconditioned BiCGStab on the active systems ----
      int it = 0;
      for (it = 0; it < a.kmax; ++it) {
        // v = (z I - A) y ;  partial (rh, v)
        for_tile_systems<T, true, true>(a, ell, side, [&](int ti, const BatchTile &tl, const BatchProb &pr, int j, int c, int sys) {
          const int n = pr.n, m = pr.m;
          const size_t nb = (size_t)a.ne * pr.off * a.m0 + (size_t)j * n * m;
          const cx<T> zj = ccast<T>(side == 0 ? pr.z[j] : conj(pr.z[j]));
          cx<T> dot = mk<T>(0, 0);
          product(ell, pr, tl, side, zj, a.y + nb, m, c, [&](int i, cx<T> o) {
            const size_t e = nb + (size_t)i * m + c;
            a.v[e] = o;
            cfma_cj(dot, a.rh[e], o);
          });
          a.part[((size_t)ti * 2) * PS + j * a.m0 + c] = dot;
        });
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
        // alpha = rho / (rh, v)
        for_systems(a, [&](bool live, int s, int p, int q, int c, int sub, const BatchProb &pr) {
          const bool go = live && a.sc.act[s];
          cxd den = mk(0.0, 0.0);
          if (go)
            for (int ti = pr.tb + sub; ti < pr.te; ti += 8) den = den + ccast<double>(a.part[((size_t)ti * 2) * PS + q]);
          den = sum8(den);
          if (!go || sub) return;
          if (!(abs2(den) > 0) || !(den.re == den.re)) {
            a.sc.act[s] = 0;  // breakdown: keep the current correction
            return;
          }
          a.sc.alpha[s] = cdiv(a.sc.rho[s], den);
        });
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
        // s = r - alpha v;  z = K^{-1} s
        for_tile_systems<T, true, false>(a, ell, side, [&](int ti, const BatchTile &tl, const BatchProb &pr, int j, int c, int sys) {
          const int n = pr.n, m = pr.m;
          const size_t nb = (size_t)a.ne * pr.off * a.m0 + (size_t)j * n * m;
          const cx<T> al = ccast<T>(a.sc.alpha[sys]);
          const cx<T> *ki = a.kinv + (size_t)a.ne * pr.off + (size_t)j * n;
          const cx<T> *__restrict__ rp = a.r + nb + c, *__restrict__ vp = a.v + nb + c;
          cx<T> *__restrict__ sp = a.s + nb + c, *__restrict__ zp = a.z + nb + c;
#pragma unroll 4
          for (int i = tl.r0; i < tl.r1; ++i) {
            const size_t e = (size_t)i * m;
            cx<T> sv = rp[e];
            cfms(sv, al, vp[e]);
            const cx<T> kv = side == 0 ? ki[i] : conj(ki[i]);
            sp[e] = sv;
            zp[e] = kv * sv;
          }
        });
        if (blockIdx.x == 0 && threadIdx.x == 0) a.ctl[2] = 0;  // counted after this iteration's update
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
        // t = (z I - A) z ;  partial (t, s), (t, t)
        for_tile_systems<T, true, true>(a, ell, side, [&](int ti, const BatchTile &tl, const BatchProb &pr, int j, int c, int sys) {
          const int n = pr.n, m = pr.m;
          const size_t nb = (size_t)a.ne * pr.off * a.m0 + (size_t)j * n * m;
          const cx<T> zj = ccast<T>(side == 0 ? pr.z[j] : conj(pr.z[j]));
          cx<T> ts = mk<T>(0, 0);
          T tt = 0;
          product(ell, pr, tl, side, zj, a.z + nb, m, c, [&](int i, cx<T> o) {
            const size_t e = nb + (size_t)i * m + c;
            a.t[e] = o;
            cfma_cj(ts, o, a.s[e]);
            tt += abs2(o);
          });
          cx<T> *pp = a.part + ((size_t)ti * 2) * PS + j * a.m0 + c;
          pp[0] = ts;
          pp[PS] = mk<T>(tt, 0);
        });
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
        // omega = (t, s) / (t, t).  act = 2: breakdown, the update below is the system's last
        for_systems(a, [&](bool live, int s, int p, int q, int c, int sub, const BatchProb &pr) {
          const bool go = live && a.sc.act[s];
          cxd ts = mk(0.0, 0.0);
          double tt = 0.0;
          if (go)
            for (int ti = pr.tb + sub; ti < pr.te; ti += 8) {
              const cx<T> *pp = a.part + ((size_t)ti * 2) * PS + q;
              ts = ts + ccast<double>(pp[0]);
              tt += (double)pp[PS].re;
            }
          ts = sum8(ts);
          tt = sum8(tt);
          if (!go || sub) return;
          const cxd om = tt > 0 ? (1.0 / tt) * ts : mk(0.0, 0.0);
          a.sc.omega[s] = om;
          if (!(abs2(om) > 0) || !(abs2(a.sc.rho[s]) > 0)) a.sc.act[s] = 2;
        });
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
        // d += alpha y + omega z ; r = s - omega t ; partial (r, r), (rh, r)
        for_tile_systems<T, true, false>(a, ell, side, [&](int ti, const BatchTile &tl, const BatchProb &pr, int j, int c, int sys) {
          const int n = pr.n, m = pr.m;
          const size_t nb = (size_t)a.ne * pr.off * a.m0 + (size_t)j * n * m;
          const cx<T> al = ccast<T>(a.sc.alpha[sys]);
          const cx<T> om = ccast<T>(a.sc.omega[sys]);
          const cx<T> *__restrict__ zp = a.z + nb + c, *__restrict__ sp = a.s + nb + c, *__restrict__ tp = a.t + nb + c,
                      *__restrict__ yp = a.y + nb + c, *__restrict__ hp = a.rh + nb + c;
          cx<T> *__restrict__ dp = a.d + nb + c, *__restrict__ rp = a.r + nb + c;
          T rr2 = 0;
          cx<T> hr = mk<T>(0, 0);
#pragma unroll 4
          for (int i = tl.r0; i < tl.r1; ++i) {
            const size_t e = (size_t)i * m;
            cx<T> dv = dp[e];
            cfma(dv, al, yp[e]);
            cfma(dv, om, zp[e]);
            dp[e] = dv;
            cx<T> rv = sp[e];
            cfms(rv, om, tp[e]);
            rp[e] = rv;
            rr2 += abs2(rv);
            cfma_cj(hr, hp[e], rv);
          }
          cx<T> *pp = a.part + ((size_t)ti * 2) * PS + j * a.m0 + c;
          pp[0] = hr;
          pp[PS] = mk<T>(rr2, 0);
        });
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
        // stop on |r|^2 <= stop2 or breakdown; beta = ((rh, r) / rho)(alpha / omega) of the others
        for_systems(a, [&](bool live, int s, int p, int q, int c, int sub, const BatchProb &pr) {
          const int act = live ? a.sc.act[s] : 0;
          double rr2 = 0.0;
          cxd hr = mk(0.0, 0.0);
          if (act)
            for (int ti = pr.tb + sub; ti < pr.te; ti += 8) {
              const cx<T> *pp = a.part + ((size_t)ti * 2) * PS + q;
              hr = hr + ccast<double>(pp[0]);
              rr2 += (double)pp[PS].re;
            }
          rr2 = sum8(rr2);
          hr = sum8(hr);
          __syncwarp();
          if (!act || sub) return;
          if (act == 2 || !(rr2 > a.sc.stop2[s]) || !(rr2 == rr2)) {
            a.sc.act[s] = 0;
            return;
          }
          a.sc.beta[s] = cdiv(hr, a.sc.rho[s]) * cdiv(a.sc.alpha[s], a.sc.omega[s]);
          a.sc.rho[s] = hr;
          atomicAdd(&a.ctl[2], 1);
        });
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
        if (*(volatile int *)&a.ctl[2] == 0) {  // nobody left
          ++it;
          break;
        }
        // p = r + beta (p - omega v) ;  y = K^{-1} p
        for_tile_systems<T, true, false>(a, ell, side, [&](int ti, const BatchTile &tl, const BatchProb &pr, int j, int c, int sys) {
          const int n = pr.n, m = pr.m;
          const size_t nb = (size_t)a.ne * pr.off * a.m0 + (size_t)j * n * m;
          const cx<T> om = ccast<T>(a.sc.omega[sys]);
          const cx<T> be = ccast<T>(a.sc.beta[sys]);
          const cx<T> *ki = a.kinv + (size_t)a.ne * pr.off + (size_t)j * n;
          const cx<T> *__restrict__ vp = a.v + nb + c, *__restrict__ rp = a.r + nb + c;
          cx<T> *__restrict__ yp = a.y + nb + c, *__restrict__ pp = a.p + nb + c;
#pragma unroll 4
          for (int i = tl.r0; i < tl.r1; ++i) {
            const size_t e = (size_t)i * m;
            cx<T> tmp = pp[e];
            cfms(tmp, om, vp[e]);
            cx<T> pv = rp[e];
            cfma(pv, be, tmp);
            pp[e] = pv;
            const cx<T> kv = side == 0 ? ki[i] : conj(ki[i]);
            yp[e] = kv * pv;
          }
        });
        if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
      }
      kry_total += it;
      // ---- X += D for the systems refined in this step ----
      for_tile_systems<T, false, false>(a, ell, side, [&](int ti, const BatchTile &tl, const BatchProb &pr, int j, int c, int sys) {
        if (!a.sc.act0[sys]) return;
        const int n = pr.n, m = pr.m;
        const size_t nb = (size_t)a.ne * pr.off * a.m0 + (size_t)j * n * m;
        for (int i = tl.r0; i < tl.r1; ++i) {
          const size_t e = nb + (size_t)i * m + c;
          const cx<T> dv = a.d[e];
          cxd x = a.X[e];
          x.re += (double)dv.re;
          x.im += (double)dv.im;
          a.X[e] = x;
        }
      });
      if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
    }
    // ---- Q = sum_j w_j X_j (left: conj(w_j)), fixed node order; stats ----
    for (int ti = blockIdx.x; ti < a.ntiles; ti += gridDim.x) {
      const BatchTile tl = a.tiles[ti];
      const BatchProb &pr = a.prob[tl.p];
      if (!pr.active) continue;
      const int n = pr.n, m = pr.m;
      const size_t xb = (size_t)a.ne * pr.off * a.m0;
      const size_t cnt = (size_t)(tl.r1 - tl.r0) * m;
      for (size_t e = threadIdx.x; e < cnt; e += blockDim.x) {
        const size_t o = (size_t)tl.r0 * m + e;
        cxd qv = mk(0.0, 0.0);
        for (int j = 0; j < a.ne; ++j) {
          const cxd wj = side == 0 ? pr.w[j] : conj(pr.w[j]);
          cfma(qv, wj, a.X[xb + (size_t)j * n * m + o]);
        }
        Qb[pr.off * a.m0 + o] = qv;
      }
    }
    for_systems(a, [&](bool live, int s, int p, int q, int c, int sub, const BatchProb &pr) {
      if (!live || sub) return;
      const double rel = a.sc.rel[s];
      const double v = (rel == rel) ? rel : INFINITY;
      atomicMax(&a.stats->maxrel_bits[side], (unsigned long long)__double_as_longlong(v));
      if (!(rel <= a.tol)) atomicAdd(&a.stats->unconverged[side], 1);
    });
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      a.stats->krylov_its[side] = kry_total;
      a.stats->steps[side] = steps_done;
    }
    if (!grid_bar(a.bar, abort_flag, a.err, a.spin_limit)) return;
  }
}

template <typename T>
static BatchKernelArgs<T> make_args(const BatchLaunch &L) {
  BatchKernelArgs<T> a{};
  a.nprob = L.nprob;
  a.ne = L.ne;
  a.m0 = L.m0;
  a.ntiles = L.ntiles;
  a.side0 = L.side0;
  a.side1 = L.side1;
  a.prob = L.prob;
  a.tiles = L.tiles;
  a.Y = L.Y;
  a.Yh = L.Yh;
  a.Q = L.Q;
  a.Qh = L.Qh;
  a.kinv = reinterpret_cast<const cx<T> *>(L.kinv);
  a.X = L.X;
  cx<T> *const *kb = reinterpret_cast<cx<T> *const *>(L.kblk);
  a.r = kb[0];
  a.rh = kb[1];
  a.p = kb[2];
  a.v = kb[3];
  a.y = kb[4];
  a.s = kb[5];
  a.z = kb[6];
  a.t = kb[7];
  a.d = kb[8];
  a.part = reinterpret_cast<cx<T> *>(L.part);
  a.partd = L.partd;
  a.partb = L.partb;
  a.sc = L.sc;
  a.bar = L.bar;
  a.ctl = L.ctl;
  a.stats = L.stats;
  a.err = L.err;
  a.tol = L.tol;
  a.tau_min = L.tau_min;
  a.nsteps = L.nsteps;
  a.kmax = L.kmax;
  a.spin_limit = L.spin_limit;
  return a;
}

template <typename T>
static const void *batch_kernel(bool lean) {
  if constexpr (sizeof(T) == 4)
    if (!lean) return (const void *)k_batch_filter<T, false>;
  return (const void *)k_batch_filter<T, true>;
}
template <typename T>
int batch_filter_max_ctas_per_sm(int threads, bool lean) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, batch_kernel<T>(lean), threads, 0) != cudaSuccess) nb = 0;
  cudaGetLastError();
  return nb;
}
template int batch_filter_max_ctas_per_sm<float>(int, bool);
template int batch_filter_max_ctas_per_sm<double>(int, bool);

template <typename T>
cudaError_t batch_filter_launch(const BatchLaunch &L, int grid, int threads, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(L.bar, 0, 2 * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(L.ctl, 0, 8 * sizeof(int), s);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(L.stats, 0, sizeof(BatchStats), s);
  if (e != cudaSuccess) return e;
  BatchKernelArgs<T> a = make_args<T>(L);
  void *params[] = {&a};
  e = cudaLaunchCooperativeKernel(batch_kernel<T>(L.lean), dim3(grid), dim3(threads), params, 0, s);
  note_launch();
  return e;
}
template cudaError_t batch_filter_launch<float>(const BatchLaunch &, int, int, cudaStream_t);
template cudaError_t batch_filter_launch<double>(const BatchLaunch &, int, int, cudaStream_t);

// Set-up of a problem for the sweeps of precision T: the values of a CSR matrix
// (conjugated where the view says so) and the inverse diagonals of its nodes.
template <typename T>
__global__ void k_batch_vals(CsrView M, T *v) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < M.nnz; k += (int64_t)gridDim.x * blockDim.x) {
    const cxd x = csr_val(M, k);
    if (M.cplx) {
      v[2 * k] = (T)x.re;
      v[2 * k + 1] = (T)x.im;
    } else {
      v[k] = (T)x.re;
    }
  }
}
struct BatchNodes {
  cxd z[kBatchMaxNe];
};
template <typename T>
__global__ void k_batch_kinv(const cxd *diag, BatchNodes nd, int ne, int n, cx<T> *kinv) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ne * n; e += gridDim.x * blockDim.x) {
    const int j = e / n, i = e - j * n;
    kinv[e] = crecip(ccast<T>(nd.z[j] - diag[i]));
  }
}
template <typename T>
void launch_batch_setup(const CsrView &A, const CsrView &AH, const cxd *diag, const cxd *z, int ne, T *vA, T *vAH,
                        cx<T> *kinv, cudaStream_t s) {
  k_batch_vals<T><<<grid_for((size_t)A.nnz), 256, 0, s>>>(A, vA);
  note_launch();
  k_batch_vals<T><<<grid_for((size_t)AH.nnz), 256, 0, s>>>(AH, vAH);
  note_launch();
  BatchNodes nd;
  for (int j = 0; j < ne; ++j) nd.z[j] = z[j];
  k_batch_kinv<T><<<grid_for((size_t)ne * A.n), 256, 0, s>>>(diag, nd, ne, A.n, kinv);
  note_launch();
}
template void launch_batch_setup<float>(const CsrView &, const CsrView &, const cxd *, const cxd *, int, float *, float *,
                                        cxf *, cudaStream_t);
template void launch_batch_setup<double>(const CsrView &, const CsrView &, const cxd *, const cxd *, int, double *,
                                         double *, cxd *, cudaStream_t);

__global__ void k_csr_diag(CsrView A, cxd *diag) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += gridDim.x * blockDim.x) {
    cxd d = mk(0.0, 0.0);
    for (int64_t k = A.rowptr[i]; k < A.rowptr[i + 1]; ++k)
      if (A.colind[k] == i) d = d + csr_val(A, k);
    diag[i] = d;
  }
}
void launch_csr_diag(const CsrView &A, cxd *diag, cudaStream_t s) {
  k_csr_diag<<<grid_for((size_t)A.n), 256, 0, s>>>(A, diag);
  note_launch();
}
__global__ void k_fill_pattern(cxd *X, size_t count) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    // a fixed integer hash mapped to [-1, 1]
    unsigned long long h = (e + 1) * 0x9E3779B97F4A7C15ull;
    h ^= h >> 31;
    h *= 0xBF58476D1CE4E5B9ull;
    h ^= h >> 29;
    X[e] = mk((double)(h & 0xFFFFF) / 524288.0 - 1.0, (double)((h >> 20) & 0xFFFFF) / 524288.0 - 1.0);
  }
}
void launch_fill_pattern(cxd *X, size_t count, cudaStream_t s) {
  k_fill_pattern<<<grid_for(count), 256, 0, s>>>(X, count);
  note_launch();
}
