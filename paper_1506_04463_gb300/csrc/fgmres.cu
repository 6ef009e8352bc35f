// Batched flexible GMRES (restarted, FGMRES(k)) for the shifted systems of
// the contour integration, (z_j B - A) d_jc = r_jc for every node j and
// column c at once, in complex FP32, with a right preconditioner that may
// change from step to step (the learned network is not a fixed linear map,
// so the flexible form keeps the preconditioned directions Z).
//
// Every (node, column) system has its own Arnoldi basis, Hessenberg matrix
// and Givens rotations; the block kernels below run all systems in one pass:
// node-major blocks ne x n x m (row-major n x m per node, complex float),
// system s = j*m + c.  Orthogonalisation is classical Gram-Schmidt applied
// twice, in three passes over the block: dot products with all previous basis
// vectors; update and dot products again; update and norm.  Scalars and the
// small least-squares problems are FP64.  Converged systems are frozen (their columns are skipped).
#include <algorithm>
#include <vector>

#include "kernels.h"
#include "reduce.cuh"

namespace {
constexpr int kFgMaxK = 64;
constexpr int kFgThreads = 256;
}  // namespace

// One pass over w by row blocks held in registers:
//   UPDATE  w -= sum_l h[l][s] V_l (the coefficients of the pass before),
//   then partial[chunk][l][s] = sum over the chunk's rows of conj(V_l) w, or
//   NORM    partial[chunk][s] = sum of |w|^2.
// V_l = V + l vs.  Bound by reading V twice out of L2 (the second time mostly
// out of L1).  A thread a system, kRB rows at a time: their loads are issued
// together, and their sums enter the FP64 partials as one value, in two FP32
// chains of four (as separate kernels, with as many chunks of rows as fit 8 CTAs
// an SM and each V_l in a loop over single rows, an orthogonalisation with its
// partial sums took 85 us a step at n = 3000, 192 systems, 44 us now).
constexpr int kRB = 8;
template <bool UPDATE, bool NORM>
__global__ void __launch_bounds__(kFgThreads) k_fg_pass(const cxf *__restrict__ V, size_t vs, int nv,
                                                        const cxd *__restrict__ h, cxf *w, int S, int n, int m,
                                                        int rows_per_cta, const int *__restrict__ active,
                                                        cxd *__restrict__ partial) {
  const int s = blockIdx.y * kFgThreads + threadIdx.x;
  if (s >= S || !active[s]) return;
  const int r0 = blockIdx.x * rows_per_cta, r1 = min(n, r0 + rows_per_cta);
  const int j = s / m, c = s - j * m;
  for (int i = r0; i < r1; i += kRB) {
    const size_t base = ((size_t)j * n + i) * m + c;
    const int cnt = min(kRB, r1 - i);
    cxf x[kRB];
#pragma unroll
    for (int r = 0; r < kRB; ++r) x[r] = r < cnt ? w[base + (size_t)r * m] : mk(0.f, 0.f);
    if (UPDATE) {
      for (int l = 0; l < nv; ++l) {
        const cxf hl = ccast<float>(h[(size_t)l * S + s]);
        const cxf *Vl = V + l * vs + base;
        cxf v[kRB];
#pragma unroll
        for (int r = 0; r < kRB; ++r) v[r] = r < cnt ? Vl[(size_t)r * m] : mk(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < kRB; ++r) cfms(x[r], hl, v[r]);
      }
#pragma unroll
      for (int r = 0; r < kRB; ++r)
        if (r < cnt) w[base + (size_t)r * m] = x[r];
    }
    for (int l = 0; l < (NORM ? 1 : nv); ++l) {
      cxf a0 = mk(0.f, 0.f), a1 = a0;
      if (NORM) {
#pragma unroll
        for (int r = 0; r < kRB; r += 2) {
          cfma_cj(a0, x[r], x[r]);
          cfma_cj(a1, x[r + 1], x[r + 1]);
        }
      } else {
        const cxf *Vl = V + l * vs + base;
        cxf v[kRB];
#pragma unroll
        for (int r = 0; r < kRB; ++r) v[r] = r < cnt ? Vl[(size_t)r * m] : mk(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < kRB; r += 2) {
          cfma_cj(a0, v[r], x[r]);
          cfma_cj(a1, v[r + 1], x[r + 1]);
        }
      }
      cxd *o = partial + ((size_t)blockIdx.x * (NORM ? 1 : nv) + l) * S + s;
      const cxd sum = ccast<double>(a0 + a1);
      *o = i == r0 ? sum : *o + sum;
    }
  }
}
// out[l][s] = sum over the chunks of partial (fixed order): one CTA per 8
// outputs, 32 threads each (more threads an output spend the FP64 pipe on the tree).  A thread per output took 167 us at 1000 chunks
// (three quarters of an FGMRES solve).  H (may be NULL): the Gram-Schmidt
// coefficients, H[s][l][col] += out[l][s].
constexpr int kFrC = 8, kFrR = 32;
__global__ void __launch_bounds__(kFrC *kFrR) k_fg_dots_reduce(const cxd *__restrict__ partial, int nchunks, int count,
                                                               cxd *out, int S, const int *active, cxd *H, int kmax,
                                                               int col) {
  __shared__ cxd sm[kFrC * kFrR];
  const int e = blockIdx.x * kFrC + threadIdx.x % kFrC;
  const int l = e / S, s = e - l * S;
  const bool ok = e < count && active[s];
  const cxd v = column_sum<kFrC, kFrR>(partial, nchunks, count, e, ok, sm);
  if (ok && threadIdx.x < kFrC) {
    out[e] = v;
    if (H) {
      cxd &hv = H[((size_t)s * (kmax + 1) + l) * kmax + col];
      hv = hv + v;
    }
  }
}
constexpr int kFdC = 4, kFdR = 64;
// per system: h_{col+1,col} = ||w|| (sum of the partials of |w|^2), v_{col+1} = w / h;
// Givens rotations on column col, residual estimate, convergence
struct FgScal {
  cxd *H;        // S x (kmax+1) x kmax
  cxd *cs, *sn;  // S x kmax (cs real, stored complex)
  cxd *g;        // S x (kmax+1)
  double *beta;  // |r0| per system
  double *resid; // current residual estimate |g_{col+1}|
  int *active;   // still iterating
  int *nact;     // count of active systems after this step
};
__global__ void __launch_bounds__(kFdC *kFdR)
    k_fg_arnoldi_tail(FgScal sc, const cxd *__restrict__ partial, int nchunks, int S, int kmax, int col, double tol,
                      cxf *invh) {
  __shared__ cxd sm[kFdC * kFdR];
  const int s = blockIdx.x * kFdC + threadIdx.x % kFdC;
  const bool ok = s < S && sc.active[s];
  const cxd wn2 = column_sum<kFdC, kFdR>(partial, nchunks, S, s, ok, sm);
  if (threadIdx.x >= kFdC || s >= S) return;
  invh[s] = mk(0.f, 0.f);
  if (!ok) return;
  const double hn = sqrt(fmax(wn2.re, 0.0));
  cxd *Hs = sc.H + (size_t)s * (kmax + 1) * kmax;
  Hs[(size_t)(col + 1) * kmax + col] = mk(hn, 0.0);
  invh[s] = hn > 0 ? mk((float)(1.0 / hn), 0.f) : mk(0.f, 0.f);
  // apply the previous rotations to column col
  for (int l = 0; l < col; ++l) {
    const cxd c = sc.cs[(size_t)s * kmax + l], sn = sc.sn[(size_t)s * kmax + l];
    const cxd a = Hs[(size_t)l * kmax + col], b = Hs[(size_t)(l + 1) * kmax + col];
    Hs[(size_t)l * kmax + col] = c * a + sn * b;
    Hs[(size_t)(l + 1) * kmax + col] = c * b - conj(sn) * a;
  }
  // new rotation zeroing H[col+1][col]
  const cxd a = Hs[(size_t)col * kmax + col], b = Hs[(size_t)(col + 1) * kmax + col];
  const double na = cabs(a), nb = cabs(b);
  cxd c, sn;
  if (nb == 0.0) {
    c = mk(1.0, 0.0);
    sn = mk(0.0, 0.0);
  } else if (na == 0.0) {
    c = mk(0.0, 0.0);
    sn = (1.0 / nb) * conj(b);  // rotates (0, b) to (|b|, 0)
  } else {
    const double r = hypot(na, nb);
    c = mk(na / r, 0.0);
    sn = (1.0 / (na * r)) * (a * conj(b));  // (a / |a|) conj(b) / r
  }
  sc.cs[(size_t)s * kmax + col] = c;
  sc.sn[(size_t)s * kmax + col] = sn;
  Hs[(size_t)col * kmax + col] = c * a + sn * b;
  Hs[(size_t)(col + 1) * kmax + col] = mk(0.0, 0.0);
  cxd *gs = sc.g + (size_t)s * (kmax + 1);
  const cxd gc = gs[col];
  gs[col] = c * gc;
  gs[col + 1] = (-1.0) * conj(sn) * gc;
  const double res = cabs(gs[col + 1]);
  sc.resid[s] = res;
  if (!(res > tol * sc.beta[s]) || !(hn > 0) || !(res == res)) sc.active[s] = 0;
  if (sc.active[s]) atomicAdd(sc.nact, 1);
}
// v = w * invh (per system), only systems that got a new column
__global__ void k_fg_scale(const cxf *w, const cxf *invh, cxf *v, int ne, int n, int m) {
  const size_t count = (size_t)ne * n * m;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    const size_t j = e / ((size_t)n * m), rem = e - j * n * m;
    const int s = (int)j * m + (int)(rem % m);
    v[e] = invh[s] * w[e];
  }
}
// start of a cycle: beta = |r| per system, v0 = r / beta, g = (beta, 0, ...); H and
// g were zeroed
__global__ void k_fg_start(FgScal sc, const cxd *rn2, int S, int kmax, const double *bnorm, double tol, cxf *invh) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  const double b = sqrt(fmax(rn2[s].re, 0.0));
  sc.beta[s] = bnorm ? bnorm[s] : b;
  sc.g[(size_t)s * (kmax + 1)] = mk(b, 0.0);
  sc.resid[s] = b;
  const bool go = b > tol * sc.beta[s] && b == b && b > 0;
  sc.active[s] = go ? 1 : 0;
  invh[s] = go ? mk((float)(1.0 / b), 0.f) : mk(0.f, 0.f);
  if (go) atomicAdd(sc.nact, 1);
}
// y = H^{-1} g (upper triangular, k columns) per system; in FP32 into yf[l][s]
__global__ void k_fg_solve_small(FgScal sc, int S, int kmax, int k, cxd *ycoef, cxf *yf) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  const cxd *Hs = sc.H + (size_t)s * (kmax + 1) * kmax;
  const cxd *gs = sc.g + (size_t)s * (kmax + 1);
  cxd *y = ycoef + (size_t)s * kmax;
  for (int l = k - 1; l >= 0; --l) {
    cxd acc = gs[l];
    for (int q = l + 1; q < k; ++q) cfms(acc, Hs[(size_t)l * kmax + q], y[q]);
    const cxd d = Hs[(size_t)l * kmax + l];
    y[l] = (abs2(d) > 0) ? cdiv(acc, d) : mk(0.0, 0.0);
    yf[(size_t)l * S + s] = ccast<float>(y[l]);
  }
}
// d += sum_l y_l Z_l, Z_l = Z + l vs
__global__ void k_fg_update_x(const cxf *__restrict__ Z, size_t vs, int k, const cxf *__restrict__ yf, int S, cxf *d,
                              int n, int m, size_t count) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    const size_t j = e / ((size_t)n * m), rem = e - j * n * m;
    const int s = (int)j * m + (int)(rem % m);
    cxf acc = d[e];
#pragma unroll 4
    for (int l = 0; l < k; ++l) cfma(acc, yf[(size_t)l * S + s], Z[l * vs + e]);
    d[e] = acc;
  }
}
// r = b - op(d): op output o = (zB - A) d, so r = b - o
__global__ void k_fg_sub(const cxf *b, const cxf *o, cxf *r, size_t count) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
    r[e] = b[e] - o[e];
}
// Jacobi preconditioner: z = v / (z_j b_ii - a_ii).  The FP64 quotient of a
// (node, row) serves its m columns: a CTA forms the quotients of 256 rows of
// one node, a row a thread, and then streams the rows' m columns.  With the
// quotient formed by every element the kernel was bound by the FP64 pipe
// (49 us for 768k elements, of which the data takes 2).
__global__ void __launch_bounds__(256) k_fg_jacobi(const cxf *__restrict__ v, const cxd *__restrict__ zn, int conj_z,
                                                   const cxd *__restrict__ adiag, const cxd *__restrict__ bdiag,
                                                   cxf *__restrict__ z, int n, int m, int rows) {
  __shared__ cxf inv[256];
  const int j = blockIdx.y, i0 = blockIdx.x * rows, cnt = min(rows, n - i0);
  if ((int)threadIdx.x < cnt) {
    const int i = i0 + threadIdx.x;
    cxd zj = zn[j];
    if (conj_z) zj = conj(zj);
    cxd a = adiag[i], bd = bdiag ? bdiag[i] : mk(1.0, 0.0);
    if (conj_z) {
      a = conj(a);
      bd = conj(bd);
    }
    inv[threadIdx.x] = ccast<float>(cdiv(mk(1.0, 0.0), zj * bd - a));
  }
  __syncthreads();
  const size_t base = ((size_t)j * n + i0) * m;
  for (int e = threadIdx.x; e < cnt * m; e += 256) z[base + e] = inv[e / m] * v[base + e];
}

// ---------------------------------------------------------------------------
// host driver
// ---------------------------------------------------------------------------
constexpr int kFgChunks = 1216;
static size_t fg_block_bytes(int n, int m0, int ne) { return ((size_t)ne * n * m0 * sizeof(cxf) + 255) & ~(size_t)255; }

size_t fgmres_work_bytes(int n, int m0, int ne, int kmax) {
  const size_t S = (size_t)ne * m0;
  return (2 * (size_t)kmax + 4) * fg_block_bytes(n, m0, ne) + (size_t)kFgChunks * (kmax + 1) * S * sizeof(cxd) +
         S * ((size_t)(kmax + 1) * kmax + 4 * kmax + 2 * (kmax + 1) + 8) * sizeof(cxd) + (64 << 10);
}

namespace {
struct FgWork {
  cxf *V, *Z;    // kmax + 1 and kmax blocks
  size_t vs;     // entries from one block to the next
  cxf *w, *o, *r;
  cxd *partial, *dots, *ycoef;
  cxf *invh, *yf;
  FgScal sc;
};

FgWork fg_carve(void *work, int n, int m0, int ne, int kmax) {
  FgWork f;
  unsigned char *p = reinterpret_cast<unsigned char *>(work);
  auto take = [&](size_t bytes) {
    unsigned char *q = p;
    p += (bytes + 255) & ~(size_t)255;
    return q;
  };
  const size_t blk = fg_block_bytes(n, m0, ne);
  const size_t S = (size_t)ne * m0;
  f.vs = blk / sizeof(cxf);
  f.V = (cxf *)take((kmax + 1) * blk);
  f.Z = (cxf *)take(kmax * blk);
  f.w = (cxf *)take(blk);
  f.o = (cxf *)take(blk);
  f.r = (cxf *)take(blk);
  f.partial = (cxd *)take((size_t)kFgChunks * (kmax + 1) * S * sizeof(cxd));
  f.dots = (cxd *)take((kmax + 1) * S * sizeof(cxd));
  f.invh = (cxf *)take(S * sizeof(cxf));
  f.ycoef = (cxd *)take(S * kmax * sizeof(cxd));
  f.yf = (cxf *)take(S * kmax * sizeof(cxf));
  f.sc.H = (cxd *)take(S * (kmax + 1) * kmax * sizeof(cxd));
  f.sc.cs = (cxd *)take(S * kmax * sizeof(cxd));
  f.sc.sn = (cxd *)take(S * kmax * sizeof(cxd));
  f.sc.g = (cxd *)take(S * (kmax + 1) * sizeof(cxd));
  f.sc.beta = (double *)take(S * sizeof(double));
  f.sc.resid = (double *)take(S * sizeof(double));
  f.sc.active = (int *)take(S * sizeof(int));
  f.sc.nact = (int *)take(64);
  return f;
}

// Rows of a CTA: one block of kRB where that is no more than kFgChunks chunks.
int fg_rows(int n) { return ceil_div(ceil_div(n, kFgChunks), kRB) * kRB; }

template <bool UPDATE, bool NORM>
int fg_pass(FgWork &f, int nv, cxf *w, int S, int n, int m, cudaStream_t s) {
  const int rpc = fg_rows(n), chunks = ceil_div(n, rpc);
  k_fg_pass<UPDATE, NORM><<<dim3(chunks, ceil_div(S, kFgThreads)), kFgThreads, 0, s>>>(
      f.V, f.vs, nv, f.dots, w, S, n, m, rpc, f.sc.active, f.partial);
  note_launch();
  return chunks;
}
void fg_reduce(FgWork &f, int chunks, int nv, int S, bool coef, int kmax, int col, cudaStream_t s) {
  k_fg_dots_reduce<<<ceil_div(nv * S, kFrC), kFrC * kFrR, 0, s>>>(f.partial, chunks, nv * S, f.dots, S, f.sc.active,
                                                                  coef ? f.sc.H : nullptr, kmax, col);
  note_launch();
}
// |x|^2 of every system into dots (all systems active)
void fg_norms(FgWork &f, const cxf *x, int S, int n, int m, cudaStream_t s) {
  cudaMemsetAsync(f.sc.active, 1, S * sizeof(int), s);  // any non-zero value
  const int chunks = fg_pass<false, true>(f, 1, const_cast<cxf *>(x), S, n, m, s);
  fg_reduce(f, chunks, 1, S, false, 0, 0, s);
}
}  // namespace

int fgmres_solve(const FgmresOp &op, const cxf *b, cxf *d, int n, int m, int ne, int m0, int kmax, int maxit,
                 double tol, void *work, double *maxrel, cudaStream_t s) {
  if (kmax > kFgMaxK) kmax = kFgMaxK;
  FgWork f = fg_carve(work, n, m0, ne, kmax);
  const int S = ne * m;
  const size_t count = (size_t)ne * n * m;
  const unsigned gb = grid_for(count);
  cudaMemsetAsync(d, 0, count * sizeof(cxf), s);
  cudaMemcpyAsync(f.r, b, count * sizeof(cxf), cudaMemcpyDeviceToDevice, s);
  // |b| per system, the convergence reference: beta of the first start
  fg_norms(f, b, S, n, m, s);
  int its = 0;
  int h_nact = 0;
  bool first = true;
  for (int cycle = 0; its < maxit; ++cycle) {
    // r = b - op(d) (d = 0 on the first cycle: r = b)
    if (!first) {
      op.apply(op.ctx, d, f.o, s);
      k_fg_sub<<<gb, 256, 0, s>>>(b, f.o, f.r, count);
      note_launch();
      fg_norms(f, f.r, S, n, m, s);
    }
    cudaMemsetAsync(f.sc.nact, 0, sizeof(int), s);
    cudaMemsetAsync(f.sc.H, 0, (size_t)S * (kmax + 1) * kmax * sizeof(cxd), s);
    cudaMemsetAsync(f.sc.g, 0, (size_t)S * (kmax + 1) * sizeof(cxd), s);
    // beta of the first cycle is |b| itself (kept in sc.beta across cycles)
    k_fg_start<<<ceil_div(S, 128), 128, 0, s>>>(f.sc, f.dots, S, kmax, first ? nullptr : f.sc.beta, tol, f.invh);
    note_launch();
    first = false;
    k_fg_scale<<<gb, 256, 0, s>>>(f.r, f.invh, f.V, ne, n, m);
    note_launch();
    cudaMemcpyAsync(&h_nact, f.sc.nact, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    if (h_nact == 0) break;
    int col = 0;
    for (col = 0; col < kmax && its < maxit; ++col, ++its) {
      op.precond(op.ctx, f.V + col * f.vs, f.Z + col * f.vs, s);
      op.apply(op.ctx, f.Z + col * f.vs, f.w, s);
      // classical Gram-Schmidt, twice
      int chunks = fg_pass<false, false>(f, col + 1, f.w, S, n, m, s);
      fg_reduce(f, chunks, col + 1, S, true, kmax, col, s);
      fg_pass<true, false>(f, col + 1, f.w, S, n, m, s);
      fg_reduce(f, chunks, col + 1, S, true, kmax, col, s);
      fg_pass<true, true>(f, col + 1, f.w, S, n, m, s);
      cudaMemsetAsync(f.sc.nact, 0, sizeof(int), s);
      k_fg_arnoldi_tail<<<ceil_div(S, kFdC), kFdC * kFdR, 0, s>>>(f.sc, f.partial, chunks, S, kmax, col, tol, f.invh);
      note_launch();
      k_fg_scale<<<gb, 256, 0, s>>>(f.w, f.invh, f.V + (col + 1) * f.vs, ne, n, m);
      note_launch();
      // every system uses col + 1 columns this cycle (frozen systems have zero
      // rows in H and g beyond their last column)
      cudaMemcpyAsync(&h_nact, f.sc.nact, sizeof(int), cudaMemcpyDeviceToHost, s);
      cudaStreamSynchronize(s);
      if (h_nact == 0) {
        ++col;
        ++its;
        break;
      }
    }
    // d += Z y with y = H^{-1} g over the columns built in this cycle
    k_fg_solve_small<<<ceil_div(S, 128), 128, 0, s>>>(f.sc, S, kmax, col, f.ycoef, f.yf);
    note_launch();
    k_fg_update_x<<<gb, 256, 0, s>>>(f.Z, f.vs, col, f.yf, S, d, n, m, count);
    note_launch();
    if (h_nact == 0) break;
  }
  // true residual of the result, relative to |b|
  op.apply(op.ctx, d, f.o, s);
  k_fg_sub<<<gb, 256, 0, s>>>(b, f.o, f.r, count);
  note_launch();
  fg_norms(f, f.r, S, n, m, s);
  std::vector<cxd> rr(S);
  std::vector<double> bb(S);
  cudaMemcpyAsync(rr.data(), f.dots, S * sizeof(cxd), cudaMemcpyDeviceToHost, s);
  cudaMemcpyAsync(bb.data(), f.sc.beta, S * sizeof(double), cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  double mx = 0;
  for (int q = 0; q < S; ++q) {
    const double rel = bb[q] > 0 ? sqrt(fmax(rr[q].re, 0.0)) / bb[q] : 0.0;
    mx = (rel > mx || !(rel == rel)) ? rel : mx;
  }
  *maxrel = mx;
  return its;
}

void launch_fg_jacobi(const cxf *v, const cxd *zn, int conj_z, const cxd *adiag, const cxd *bdiag, cxf *z, int ne,
                      int n, int m, cudaStream_t s) {
  // enough CTAs for the chip first, then up to 256 rows of a quotient each
  const int rows = std::max(1, (int)std::min<long long>(256, ((long long)n * ne + 607) / 608));
  k_fg_jacobi<<<dim3(ceil_div(n, rows), ne), 256, 0, s>>>(v, zn, conj_z, adiag, bdiag, z, n, m, rows);
  note_launch();
}

// X (complex double) = d (mode 0) or X += d (mode 1), d complex float
__global__ void k_cxf_accumulate(cxd *X, const cxf *d, size_t count, int mode) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    const cxd v = ccast<double>(d[e]);
    X[e] = mode ? X[e] + v : v;
  }
}
void launch_cxf_accumulate(cxd *X, const cxf *d, size_t count, int mode, cudaStream_t s) {
  k_cxf_accumulate<<<grid_for(count), 256, 0, s>>>(X, d, count, mode);
  note_launch();
}
// out[j] = (complex float) B Y for every node j (node-major copies of one block)
__global__ void k_broadcast_cxf(const cxd *BY, cxf *out, size_t nm, int ne) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nm * ne; e += (size_t)gridDim.x * blockDim.x)
    out[e] = ccast<float>(BY[e % nm]);
}
void launch_broadcast_cxf(const cxd *BY, cxf *out, size_t nm, int ne, cudaStream_t s) {
  k_broadcast_cxf<<<grid_for(nm * ne), 256, 0, s>>>(BY, out, nm, ne);
  note_launch();
}
