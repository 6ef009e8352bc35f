// Control kernels of the Rayleigh-Ritz step and of the convergence test
// (Fig. alg:three steps 2.b, 3.b-3.d, 4.b-4.c, 5).  All run as one CTA on
// the m <= 128 reduced quantities; the n-sized work is in dense.cu / spmm.cu.
#include <float.h>
#include "rr.cuh"

// Steps 2.b and 3.b-3.c: spurious count against the previous Ritz values,
// stable sort of gamma by decreasing modulus, resize (eq. resize) and the
// bi-orthonormalising coefficients of eq. (uu):
//   S  = V[:, ord] Gamma^{-1/2},   Sh = Vh[:, ord] Gamma^{-H/2},  Vh = V^{-H}.
// Complex symmetric: V scaled to v^T v = 1 and Vh = conj(V) (Sec. 2.4).
__global__ void k_gamma_prep(int m, const cxd *BQ, const cxd *gam, const cxd *V, const cxd *Vinv,
                             const cxd *prev_rho, const int *prev_inside, int have_prev, double mu, double eta,
                             int cs, cxd *S, cxd *Sh, int *ord, RRStatus *st) {
  __shared__ int o[kMaxM0];
  __shared__ cxd g[kMaxM0];
  __shared__ cxd tcs[kMaxM0];
  const int tid = threadIdx.x, nt = blockDim.x;
  // moduli once, then every value finds its own place: the number of larger
  // ones, and of equal ones before it (a stable sort, decreasing).  Moduli
  // are compared as integers (the bits of non-negative doubles), since an FP64
  // compare costs a warp 64 cycles; NaN goes last.
  __shared__ long long key[kMaxM0];
  double md = -1.0;
  if (tid < m) {
    md = cabs(gam[tid]);
    key[tid] = md == md ? __double_as_longlong(md) : -1;
  }
  bool spur = false;
  if (tid < m && have_prev && prev_inside[tid]) {
    const cxd r2 = prev_rho[tid] * prev_rho[tid];
    const cxd d = BQ[(size_t)tid * m + tid];
    const double den = cabs(r2);
    const double q = den > 0 ? cabs(r2 - d) / den : INFINITY;
    spur = !(q < mu);
  }
  const int ms = __syncthreads_count(spur);
  if (tid < m) {
    int rank = 0;
    for (int j = 0; j < m; ++j) rank += key[j] > key[tid] || (key[j] == key[tid] && j < tid);
    o[rank] = tid;
  }
  __syncthreads();
  const double gmax = cabs(gam[o[0]]);
  const int mt = __syncthreads_count(tid < m && md >= eta * gmax && gmax > 0);
  if (tid == 0) {
    st->m_s = ms;
    st->m_tilde = mt;
  }
  for (int b = tid; b < m; b += nt) {
    ord[b] = o[b];
    const cxd sq = csqrt(gam[o[b]]);
    g[b] = cdiv(mk(1.0, 0.0), sq);
    if (cs) {
      cxd t = mk(0.0, 0.0);
      for (int a = 0; a < m; ++a) cfma(t, V[(size_t)a * m + o[b]], V[(size_t)a * m + o[b]]);
      tcs[b] = csqrt(t);
    }
  }
  __syncthreads();
  for (int e = tid; e < m * m; e += nt) {
    const int a = e / m, b = e - a * m;
    if (b >= mt) {
      S[e] = mk(0.0, 0.0);
      Sh[e] = mk(0.0, 0.0);
      continue;
    }
    const int src = o[b];
    cxd v = V[(size_t)a * m + src];
    if (cs) {
      v = cdiv(v, tcs[b]);
      S[e] = v * g[b];
      Sh[e] = conj(v) * conj(g[b]);
    } else {
      S[e] = v * g[b];
      Sh[e] = conj(Vinv[(size_t)src * m + a]) * conj(g[b]);
    }
  }
}

// Step 4.c: rho_a(lambda_i) = sum_j w_j / (z_j - lambda_i)   (eq. rational).
// One warp per eigenvalue, a lane per node: the FP64 quotients (some 50
// instructions of 64 cycles each) are formed side by side.
__global__ void __launch_bounds__(32) k_rho(int ne, const cxd *z, const cxd *w, const cxd *lam, cxd *rho) {
  const int i = blockIdx.x, lane = threadIdx.x;
  const cxd l = lam[i];
  cxd s = mk(0.0, 0.0);
  for (int j = lane; j < ne; j += 32) s = s + cdiv(w[j], z[j] - l);
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    s.re += __shfl_down_sync(0xffffffffu, s.re, o);
    s.im += __shfl_down_sync(0xffffffffu, s.im, o);
  }
  if (lane == 0) rho[i] = s;
}

// Y[:, i] /= ||y_i||, Yh[:, i] *= ||y_i|| (column scale of the Ritz vectors).
// The root and the quotient of a column are formed once per CTA: by every
// element they made the kernel FP64-bound (192 us at 90 000 x 64, of which
// moving the 369 MB takes 54).
__global__ void __launch_bounds__(256) k_scale_pairs(cxd *Y, cxd *Yh, const double *nrm2, int m, size_t count) {
  __shared__ double sc[kMaxM0], inv[kMaxM0];
  for (int c = threadIdx.x; c < m; c += blockDim.x) {
    const double s = sqrt(nrm2[c]);
    sc[c] = s > 0 ? s : 1.0;
    inv[c] = s > 0 ? 1.0 / s : 1.0;
  }
  __syncthreads();
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % m);
    Y[e] = inv[c] * Y[e];
    Yh[e] = sc[c] * Yh[e];
  }
}

__device__ __forceinline__ bool inside_contour(cxd l, const RRParams &p) {
  if (!(isfinite(l.re) && isfinite(l.im))) return false;
  if (p.kind == 2) {
    bool in = false;
    for (int k = 0; k < p.ne; ++k) {
      const cxd a = p.cz[k], b = p.cz[(k + 1) % p.ne];
      if ((a.im > l.im) != (b.im > l.im)) {
        double xc = a.re + (l.im - a.im) * (b.re - a.re) / (b.im - a.im);
        if (l.re < xc) in = !in;
      }
    }
    return in;
  }
  const double ca = cos(p.angle), sa = sin(p.angle);
  const double dx = l.re - p.c_re, dy = l.im - p.c_im;
  const double u = ca * dx + sa * dy, v = -sa * dx + ca * dy;
  const double a = p.r, b = p.r * (p.kind == 0 ? 1.0 : p.ratio);
  return (u / a) * (u / a) + (v / b) * (v / b) <= 1.0;
}

// Step 5: inside count m_r, residuals of eq. (res), m = m_r - m_s, converged
// pairs ordered by increasing residual; saves rho and the inside flags for the
// spurious test of the next iteration.
__global__ void k_converge(RRParams p, int mt, const cxd *lam, const cxd *rho, const double *cn, double *res,
                           int *ord, cxd *prev_rho, int *prev_inside, RRStatus *st) {
  __shared__ long long key[kMaxM0];  // bits of the residual (>= 0), or the largest integer outside
  __shared__ double mxs[4];
  const int tid = threadIdx.x, i = tid;  // 128 threads, mt <= 128
  bool in = false;
  double r = INFINITY;
  if (i < mt) {
    in = inside_contour(lam[i], p);
    if (in) {
      const double r1 = cn[i] / (p.alpha * cn[kMaxM0 + i]);
      const double r2 = cn[2 * kMaxM0 + i] / (p.alpha * cn[3 * kMaxM0 + i]);
      r = fmax(r1, r2);
      if (!(r == r)) r = INFINITY;
    }
    res[i] = r;
    prev_rho[i] = rho[i];
    prev_inside[i] = in;
    key[i] = in ? __double_as_longlong(r) : 0x7fffffffffffffffll;
  }
  const int mr = __syncthreads_count(in);
  // inside pairs by increasing residual, then the others by index: every pair
  // counts the ones before it
  const int m = mr - st->m_s;
  int rank = 0;
  if (i < mt) {
    for (int j = 0; j < mt; ++j) rank += key[j] < key[i] || (key[j] == key[i] && j < i);
    ord[rank] = i;
  }
  const bool low = in && rank < m;  // among the m lowest residuals
  const bool bad = __syncthreads_or(low && !(r < p.eps));
  const bool conv = m >= 1 && !bad;
  const int below = __syncthreads_count(in && r < p.eps);
  double mx = low ? r : 0.0;
#pragma unroll
  for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((tid & 31) == 0) mxs[tid >> 5] = mx;
  __syncthreads();
  if (tid == 0) {
    // 5.d: on convergence every inside pair below eps is returned (at least m)
    st->m_r = mr;
    st->m = conv ? below : (m > 0 ? m : 0);
    st->conv = conv ? 1 : 0;
    st->max_res = m >= 1 ? fmax(fmax(mxs[0], mxs[1]), fmax(mxs[2], mxs[3])) : INFINITY;
  }
}

// Column statistics for the output normalisation: ||y||^2, the entry of
// largest modulus (first index on ties) and y^^H (B y).
__global__ void k_colstats(const cxd *Y, const cxd *Yh, const cxd *BY, int m, int n, int rows_per_cta,
                           double *pn, double *pmax, int *pidx, cxd *pval, cxd *pdot) {
  const int c = threadIdx.x;
  if (c >= m) return;
  const int rbeg = blockIdx.x * rows_per_cta, rend = min(n, rbeg + rows_per_cta);
  double s = 0.0, best = -1.0;
  int bi = 0;
  cxd bv = mk(0.0, 0.0), d = mk(0.0, 0.0);
  for (int i = rbeg; i < rend; ++i) {
    const cxd y = Y[(size_t)i * m + c];
    const double a2 = abs2(y);
    s += a2;
    if (a2 > best) {
      best = a2;
      bi = i;
      bv = y;
    }
    cfma_cj(d, Yh[(size_t)i * m + c], BY[(size_t)i * m + c]);
  }
  const size_t o = (size_t)blockIdx.x * m + c;
  pn[o] = s;
  pmax[o] = best;
  pidx[o] = bi;
  pval[o] = bv;
  pdot[o] = d;
}

__global__ void k_finalize_coeffs(int m, int nparts, const double *pn, const double *pmax, const int *pidx,
                                  const cxd *pval, const cxd *pdot, cxd *sx, cxd *sxh) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= m) return;
  double s = 0.0, best = -1.0;
  int bi = 0x7fffffff;
  cxd bv = mk(1.0, 0.0), d = mk(0.0, 0.0);
  for (int p = 0; p < nparts; ++p) {
    const size_t o = (size_t)p * m + c;
    s += pn[o];
    if (pmax[o] > best || (pmax[o] == best && pidx[o] < bi)) {
      best = pmax[o];
      bi = pidx[o];
      bv = pval[o];
    }
    d = d + pdot[o];
  }
  const double nrm = sqrt(s);
  const double av = cabs(bv);
  cxd ph = av > 0 ? mk(bv.re / av, -bv.im / av) : mk(1.0, 0.0);  // conj(phase)
  const cxd scale = (nrm > 0 ? 1.0 / nrm : 1.0) * ph;
  const cxd t = scale * d;  // x^^H B x after scaling x
  sx[c] = scale;
  sxh[c] = cdiv(mk(1.0, 0.0), conj(t));
}

// X[:, k] = sx[src] Y[:, src], Xh[:, k] = sxh[src] Yh[:, src], src = ord[k].
__global__ void k_gather_out(const cxd *Y, const cxd *Yh, int m, int n, const int *ord, int mout, const cxd *sx,
                             const cxd *sxh, cxd *X, cxd *Xh, int ldo) {
  const size_t count = (size_t)n * mout;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    const size_t i = e / mout;
    const int k = (int)(e - i * mout);
    const int src = ord[k];
    X[i * ldo + k] = sx[src] * Y[i * m + src];
    Xh[i * ldo + k] = sxh[src] * Yh[i * m + src];
  }
}
__global__ void k_gather_small(const cxd *lam, const double *res, const int *ord, int mout, double *lam_out,
                               double *res_out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= mout) return;
  lam_out[2 * k] = lam[ord[k]].re;
  lam_out[2 * k + 1] = lam[ord[k]].im;
  if (res_out) res_out[k] = res[ord[k]];
}

// ---------------------------------------------------------------------------
void launch_gamma_prep(int m, const cxd *BQ, const cxd *gam, const cxd *V, const cxd *Vinv, const cxd *prev_rho,
                       const int *prev_inside, int have_prev, double mu, double eta, int cs, cxd *S, cxd *Sh,
                       int *ord, RRStatus *st, cudaStream_t s) {
  k_gamma_prep<<<1, 256, 0, s>>>(m, BQ, gam, V, Vinv, prev_rho, prev_inside, have_prev, mu, eta, cs, S, Sh, ord,
                                 st);
  note_launch();
}
void launch_rho(int m, int ne, const cxd *z, const cxd *w, const cxd *lam, cxd *rho, cudaStream_t s) {
  k_rho<<<m, 32, 0, s>>>(ne, z, w, lam, rho);
  note_launch();
}
void launch_scale_pairs(cxd *Y, cxd *Yh, const double *nrm2, int m, int n, cudaStream_t s) {
  size_t count = (size_t)n * m;
  k_scale_pairs<<<grid_for(count), 256, 0, s>>>(Y, Yh, nrm2, m, count);
  note_launch();
}
void launch_converge(const RRParams &p, int mt, const cxd *lam, const cxd *rho, const double *cn, double *res,
                     int *ord, cxd *prev_rho, int *prev_inside, RRStatus *st, cudaStream_t s) {
  k_converge<<<1, 128, 0, s>>>(p, mt, lam, rho, cn, res, ord, prev_rho, prev_inside, st);
  note_launch();
}
int launch_colstats(const cxd *Y, const cxd *Yh, const cxd *BY, int m, int n, double *pn, double *pmax, int *pidx,
                    cxd *pval, cxd *pdot, cudaStream_t s) {
  int g = min(304, ceil_div(n, 64));
  int rpc = ceil_div(n, g);
  g = ceil_div(n, rpc);
  k_colstats<<<g, 128, 0, s>>>(Y, Yh, BY, m, n, rpc, pn, pmax, pidx, pval, pdot);
  note_launch();
  return g;
}
void launch_finalize(int m, int nparts, const double *pn, const double *pmax, const int *pidx, const cxd *pval,
                     const cxd *pdot, cxd *sx, cxd *sxh, const cxd *Y, const cxd *Yh, int n, const int *ord, int mout,
                     cxd *X, cxd *Xh, int ldo, const cxd *lam, const double *res, double *lam_out, double *res_out,
                     cudaStream_t s) {
  k_finalize_coeffs<<<1, 128, 0, s>>>(m, nparts, pn, pmax, pidx, pval, pdot, sx, sxh);
  note_launch();
  size_t count = (size_t)n * mout;
  if (count) {
    k_gather_out<<<grid_for(count), 256, 0, s>>>(Y, Yh, m, n, ord, mout, sx, sxh, X,
                                                                                 Xh, ldo);
    note_launch();
  }
  if (mout) {
    k_gather_small<<<1, 128, 0, s>>>(lam, res, ord, mout, lam_out, res_out);
    note_launch();
  }
}
