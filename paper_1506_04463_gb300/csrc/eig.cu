// Small dense work of the Rayleigh-Ritz step (m <= 128), spread over the chip.
//
// The part's FP64 pipe takes 64 cycles for a warp instruction whether one lane
// or 32 are active, and a dependent chain costs the same 64 cycles a link.  So
// a sequential FP64 algorithm on one CTA (k_small_eig, dense.cu: some 30
// dependent instructions for each of 9000 rotations at m = 64) is 10 ms of
// waiting, while an FP64 product of two 64 x 64 complex matrices on 128 CTAs
// takes 3 us.  The kernels here do the sequential part in FP32 (4.5 cycles a
// link) and get FP64 accuracy back with products:
//
//  * small_eig: eigenpairs of a general complex matrix.  k_eig32 computes an
//    FP32 eigendecomposition (X, W = X^{-1}, d) of the shifted, scaled and
//    balanced matrix on one CTA; Newton's method then refines all pairs at
//    once in FP64: with R = M X - X diag(d) and E = W R, a first-order
//    correction is X <- X (I + F), F_ij = E_ij / (d_j - d_i), d_j += E_jj, and
//    W follows by W <- (I - F) W and Newton-Schulz steps W <- (2 I - W X) W.
//    These are formed from the left defect I - W X because W X is what has to
//    be the identity (Yh^H B Y = W X): in rounding the right defect differs
//    from it by the condition number (X of condition 1e4, m = 32: |W X - I| of
//    9e-14, of 4e-11 from the right defect, 7e-13 with an FP64 inverse).
//    It converges quadratically where the eigenvalues are separated by more
//    than the FP32 errors; three iterations are usual.  Where it does not get
//    below kFTol in kMaxIt iterations (clustered or graded spectra), the FP64
//    QR kernel computes the pairs from scratch: it is always launched and
//    returns at once when the refinement has converged.
//  * small_inv_near: inverse of a matrix close to the identity (B_U of step
//    4.b) by Newton-Schulz products, the FP64 Gauss-Jordan kernel otherwise.
//  * biorth: coefficients S, Sh with Sh^H B_Q S = I (eq. uu) by elimination
//    with complete pivoting on one cluster, where the resize (eq. resize)
//    provably keeps every column.  That takes a B_Q of condition below 1e13:
//    both of the 10 x 10 and 100 x 100 grids' solves and the second of the 40 x
//    40 one have it, the graded ones of the 300 x 300 benchmark do not.
#include <cooperative_groups.h>
#include <float.h>
#include <algorithm>
#include "rr.cuh"

namespace {

constexpr int kMaxIt = 5;            // Newton iterations launched
constexpr float kFTol = 3.7e-9f;     // stop: the next correction would be of order m F^2 < 2e-15

}  // namespace

// Workspace of small_eig: status words, then m x m blocks.
struct EigState {
  int failed;            // the FP32 eigendecomposition did not converge
  int done;              // refinement converged (set by k_eig_finish)
  int expo, pad;         // M = 2^-expo D^{-1} (A - mu I) D
  cxd mu;
  unsigned fmax[8];      // bits of max |F_ij| of each iteration
  double dsc[kMaxM0];    // D
  cxd d[2][kMaxM0];      // eigenvalues of M, ping-pong
  int near;              // small_inv_near: the matrix was close to the identity
};

size_t small_eig_state_bytes() { return (sizeof(EigState) + 255) & ~(size_t)255; }

namespace {

// z != 0 by its bits (an FP64 compare costs a warp 64 cycles)
__device__ __forceinline__ bool nonzero(cxd z) {
  return (((__double2hiint(z.re) | __double2hiint(z.im)) & 0x7fffffff) | __double2loint(z.re) | __double2loint(z.im)) !=
         0;
}
__device__ __forceinline__ float cabs1f(cxf a) { return fabsf(a.re) + fabsf(a.im); }

// Iteration `it` has nothing left to do: the seed failed or an earlier
// iteration's correction was below the tolerance.
__device__ __forceinline__ bool eig_over(const EigState *st, int it) {
  if (st->failed) return true;
  for (int k = 0; k < it; ++k)
    if (!(__uint_as_float(st->fmax[k]) > kFTol)) return true;
  return false;
}

// principal square root
__device__ __forceinline__ cxf csqrtf_(cxf a) {
  const float r = sqrtf(a.re * a.re + a.im * a.im);
  if (!(r > 0.f)) return mk(0.f, 0.f);
  const float t = sqrtf(0.5f * (r + fabsf(a.re)));
  const float u = a.im / (2.f * t);
  if (a.re >= 0.f) return mk(t, u);
  return mk(fabsf(u), a.im >= 0.f ? t : -t);
}

__device__ __forceinline__ cxf crecipf(cxf d) {
  const float sc = fmaxf(fabsf(d.re), fabsf(d.im));
  const float is = 1.f / sc;
  const float a = d.re * is, b = d.im * is;
  const float r = is / (a * a + b * b);
  return mk(a * r, -b * r);
}

// right rotation of a row's pair (h1, h2): o = c h1 + conj(s) h2, h1 = c h2 - s h1
__device__ __forceinline__ void rotate(float4 g, cxf &h1, cxf h2, cxf &o) {
  o.re = fmaf(g.y, h2.re, fmaf(g.z, h2.im, g.x * h1.re));
  o.im = fmaf(g.y, h2.im, fmaf(-g.z, h2.re, g.x * h1.im));
  cxf n;
  n.re = fmaf(-g.y, h1.re, fmaf(g.z, h1.im, g.x * h2.re));
  n.im = fmaf(-g.y, h1.im, fmaf(-g.z, h1.re, g.x * h2.im));
  h1 = n;
}

}  // namespace

// FP32 eigendecomposition of M = 2^-e D^{-1} (A - mu I) D on one CTA: mu is
// the mean of the diagonal (so that FP32 resolves the spectrum's spread and
// not its position), e the exponent of the largest entry, D the powers of two
// of the Parlett-Reinsch balancing.  Householder reduction, explicit
// single-shift QR, back-substitution.  H (and Z for m <= zmax) in shared
// memory with an odd row length.  Writes M (FP64), X, W (FP64 copies of the
// FP32 values), d and D.  One warp carries the chain of left rotations, its
// lanes on the columns: the next rotation waits for a complex update, a
// reciprocal square root and four shuffles, some 130 cycles, against 2000 for
// an FP64 rotation; the right rotations of a sweep are a row a thread.
template <int Q>  // ceil(m / 32): columns of a lane
__global__ void __launch_bounds__(256, 1) k_eig32(const cxd *__restrict__ A, int m, cxd *__restrict__ Mout,
                                                  cxd *__restrict__ X, cxd *__restrict__ W, cxf *__restrict__ zglob,
                                                  int zsm, EigState *st) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ cxf v[kMaxM0];
  __shared__ float4 rot[kMaxM0];  // (c, s.re, s.im, -) of the current sweep
  __shared__ float dsc[kMaxM0];
  __shared__ double red[256];
  __shared__ int redi[8];
  __shared__ int sh_l, sh_hi, sh_done, hskip_s;
  __shared__ cxf sh_mu, hbeta_s;
  __shared__ float hsc_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ld = m | 1;
  cxf *H = reinterpret_cast<cxf *>(dsm);
  cxf *Z = zsm ? H + (size_t)m * ld : zglob;
  // ---- mean of the diagonal, exponent of the largest entry ----
  if (tid < 64) {
    double s = 0.0;
    for (int i = lane; i < m; i += 32) s += tid < 32 ? A[(size_t)i * m + i].re : A[(size_t)i * m + i].im;
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp] = s / m;
  }
  __syncthreads();
  const cxd mu = mk(red[0], red[1]);
  int em = 0;
  for (int e = tid; e < m * m; e += 256) {
    cxd a = A[e];
    if (e / m == e % m) a = a - mu;
    em = max(em, max(__double2hiint(a.re) & 0x7fffffff, __double2hiint(a.im) & 0x7fffffff));
  }
  em = __reduce_max_sync(0xffffffffu, em);
  if (lane == 0) redi[warp] = em;
  __syncthreads();
  for (int w = 0; w < 8; ++w) em = max(em, redi[w]);
  const int ef = em >> 20;  // exponent field of the largest component
  const bool bad = ef >= 2046 || ef < 64;  // overflow, NaN, or all (nearly) zero: left to the FP64 kernel
  if (bad) {
    if (tid == 0) st->failed = 1;
    return;
  }
  const double scale = __hiloint2double((2046 - ef) << 20, 0);  // 2^(1023 - ef)
  for (int e = tid; e < m * m; e += 256) {
    const int i = e / m, j = e - i * m;
    cxd a = A[e];
    if (i == j) a = a - mu;
    H[(size_t)i * ld + j] = mk((float)(scale * a.re), (float)(scale * a.im));
  }
  if (tid < m) dsc[tid] = 1.f;
  __syncthreads();
  // ---- balancing by one warp, powers of two (see k_small_eig) ----
  if (tid < 32) {
    for (int pass = 0; pass < 16; ++pass) {
      bool changed = false;
      for (int i = 0; i < m; ++i) {
        float c = 0.f, r = 0.f;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const int j = lane + 32 * q;
          if (j < m && j != i) {
            c += cabs1f(H[(size_t)j * ld + i]);
            r += cabs1f(H[(size_t)i * ld + j]);
          }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          c += __shfl_xor_sync(0xffffffffu, c, o);
          r += __shfl_xor_sync(0xffffffffu, r, o);
        }
        if (!(c > 0.f) || !(r > 0.f) || (c >= 0.5f * r && c < 2.f * r)) continue;
        const float s = c + r;
        float f = 1.f;
        for (int q = 0; q < 40 && c < 0.5f * r; ++q) {
          c *= 2.f;
          r *= 0.5f;
          f *= 2.f;
        }
        for (int q = 0; q < 40 && c >= 2.f * r; ++q) {
          c *= 0.5f;
          r *= 2.f;
          f *= 0.5f;
        }
        if (c + r >= 0.95f * s) continue;
        changed = true;
        const float fi = 1.f / f;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const int j = lane + 32 * q;
          if (j < m) {
            H[(size_t)j * ld + i] = f * H[(size_t)j * ld + i];
            H[(size_t)i * ld + j] = fi * H[(size_t)i * ld + j];
          }
        }
        if (lane == 0) dsc[i] *= f;
        __syncwarp();
      }
      if (!changed) break;
    }
  }
  __syncthreads();
  // balancing can shrink the matrix by many orders: scale it to size one again
  int eb = 0;
  for (int e = tid; e < m * m; e += 256) {
    const cxf h = H[(size_t)(e / m) * ld + e % m];
    eb = max(eb, max(__float_as_int(h.re) & 0x7fffffff, __float_as_int(h.im) & 0x7fffffff));
  }
  eb = __reduce_max_sync(0xffffffffu, eb);
  if (lane == 0) redi[warp] = eb;
  __syncthreads();
  for (int w = 0; w < 8; ++w) eb = max(eb, redi[w]);
  const int e2 = (eb >> 23) - 127;  // exponent of the balanced matrix
  if (e2 > 100 || e2 < -100) {
    if (tid == 0) st->failed = 1;
    return;
  }
  const float s2 = __int_as_float((127 - e2) << 23);
  const double scale2 = scale * (double)s2;
  for (int e = tid; e < m * m; e += 256) {
    const int i = e / m, j = e - i * m;
    cxd a = A[e];
    if (i == j) a = a - mu;
    const double f = scale2 * ((double)dsc[j] / (double)dsc[i]);  // a power of two
    Mout[e] = mk(f * a.re, f * a.im);
    H[(size_t)i * ld + j] = s2 * H[(size_t)i * ld + j];
    Z[(size_t)i * ld + j] = mk(i == j ? 1.f : 0.f, 0.f);
  }
  if (tid < m) st->dsc[tid] = dsc[tid];
  if (tid == 0) {
    st->mu = mu;
    st->expo = ef - 1023 + e2;
  }
  __syncthreads();
  // ---- Householder reduction to Hessenberg form ----
  for (int k = 0; k + 2 < m; ++k) {
    const int L = m - k - 1;
    if (tid < 32) {
      float n2 = 0.f;
      for (int i = lane; i < L; i += 32) n2 += abs2(H[(size_t)(k + 1 + i) * ld + k]);
#pragma unroll
      for (int o = 16; o; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      if (lane == 0) {
        int skip = !(n2 > 1e-36f);
        cxf beta = mk(0.f, 0.f);
        float sc = 0.f;
        if (!skip) {
          const float nrm = sqrtf(n2);
          const cxf x0 = H[(size_t)(k + 1) * ld + k];
          const float ax0 = sqrtf(abs2(x0));
          const cxf ph = ax0 > 0.f ? mk(x0.re / ax0, x0.im / ax0) : mk(1.f, 0.f);
          beta = mk(-ph.re * nrm, -ph.im * nrm);
          const float vn2 = n2 - abs2(x0) + abs2(x0 - beta);
          skip = !(vn2 > 0.f);
          if (!skip) sc = 2.f / vn2;
        }
        hskip_s = skip;
        hsc_s = sc;
        hbeta_s = beta;
      }
    }
    for (int i = tid; i < L; i += 256) v[i] = H[(size_t)(k + 1 + i) * ld + k];
    __syncthreads();
    if (hskip_s) {
      __syncthreads();
      for (int i = 1 + tid; i < L; i += 256) H[(size_t)(k + 1 + i) * ld + k] = mk(0.f, 0.f);
      __syncthreads();
      continue;
    }
    const cxf beta = hbeta_s;
    const float sc = hsc_s;
    if (tid == 0) v[0] = v[0] - beta;
    __syncthreads();
    for (int base = 0; base < m - k; base += 64) {  // four threads a column
      const int jj = base + (tid >> 2), j = k + jj, part = tid & 3;
      const bool act = jj < m - k;
      cxf w = mk(0.f, 0.f);
      if (act)
        for (int i = part; i < L; i += 4) cfma_cj(w, v[i], H[(size_t)(k + 1 + i) * ld + j]);
      w.re += __shfl_xor_sync(0xffffffffu, w.re, 1);
      w.im += __shfl_xor_sync(0xffffffffu, w.im, 1);
      w.re += __shfl_xor_sync(0xffffffffu, w.re, 2);
      w.im += __shfl_xor_sync(0xffffffffu, w.im, 2);
      w = sc * w;
      if (act)
        for (int i = part; i < L; i += 4) cfms(H[(size_t)(k + 1 + i) * ld + j], v[i], w);
    }
    __syncthreads();
    for (int r = tid; r < 2 * m; r += 256) {
      cxf *M = r < m ? H + (size_t)r * ld : Z + (size_t)(r - m) * ld;
      cxf s = mk(0.f, 0.f);
#pragma unroll 4
      for (int i = 0; i < L; ++i) cfma(s, M[k + 1 + i], v[i]);
      s = sc * s;
#pragma unroll 4
      for (int i = 0; i < L; ++i) {  // row -= s v^H
        cxf h = M[k + 1 + i];
        const cxf vi = v[i];
        h.re -= s.re * vi.re + s.im * vi.im;
        h.im -= s.im * vi.re - s.re * vi.im;
        M[k + 1 + i] = h;
      }
    }
    __syncthreads();
    for (int i = 1 + tid; i < L; i += 256) H[(size_t)(k + 1 + i) * ld + k] = mk(0.f, 0.f);
    if (tid == 0) H[(size_t)(k + 1) * ld + k] = beta;
    __syncthreads();
  }
  // ---- QR iteration ----
  if (tid == 0) {
    sh_hi = m - 1;
    sh_done = 0;
  }
  __syncthreads();
  int its = 0, total = 0;
  const float floor_ = (float)m * FLT_EPSILON;  // the largest entry of M is about one
  while (true) {
    if (tid < 32) {
      int hi = sh_hi, l = 0, done = 0;
      while (true) {
        l = 0;
        for (int base = hi; base >= 1; base -= 32) {
          const int lc = base - lane;
          bool neg = false;
          if (lc >= 1) {
            const float s = cabs1f(H[(size_t)(lc - 1) * ld + lc - 1]) + cabs1f(H[(size_t)lc * ld + lc]);
            const float sub = cabs1f(H[(size_t)lc * ld + lc - 1]);
            neg = sub <= 2.f * FLT_EPSILON * s || (its >= 20 && sub <= floor_) || sub < 1e-30f;
          }
          const unsigned vote = __ballot_sync(0xffffffffu, neg);
          if (vote) {
            l = base - (__ffs(vote) - 1);
            break;
          }
        }
        __syncwarp();
        if (lane == 0 && l > 0) H[(size_t)l * ld + l - 1] = mk(0.f, 0.f);
        __syncwarp();
        if (l < hi) break;
        --hi;  // one eigenvalue found: look at the next block at once
        its = 0;
        if (hi < 1) {
          done = 1;
          break;
        }
      }
      if (!done) {
        ++its;
        if (++total > 10 * m) {  // three sweeps an eigenvalue are usual
          done = 2;
        } else {
          const cxf a = H[(size_t)(hi - 1) * ld + hi - 1], b = H[(size_t)(hi - 1) * ld + hi];
          const cxf c = H[(size_t)hi * ld + hi - 1], d = H[(size_t)hi * ld + hi];
          cxf sft;
          if (its % 11 == 10) {
            sft = d + mk(0.75f * cabs1f(c), 0.f);
          } else {
            const cxf half = mk(0.5f * (a.re - d.re), 0.5f * (a.im - d.im));
            const cxf disc = csqrtf_(half * half + b * c);
            const cxf mid = mk(0.5f * (a.re + d.re), 0.5f * (a.im + d.im));
            const cxf m1 = mid + disc, m2 = mid - disc;
            sft = abs2(m1 - d) < abs2(m2 - d) ? m1 : m2;
          }
          if (!(cabs1f(sft) < 1e18f)) done = 2;  // overflow or NaN
          // left rotations: lane owns columns lane + 32 q; cur: row k of its
          // columns, nxt: row k + 1
          cxf cur[Q], nxt[Q];
          auto own = [&](const cxf (&row)[Q], int j) {  // column j's entry, in every lane
            cxf x = row[0];
#pragma unroll
            for (int q = 1; q < Q; ++q)
              if ((j >> 5) == q) x = row[q];
            return mk(__shfl_sync(0xffffffffu, x.re, j & 31), __shfl_sync(0xffffffffu, x.im, j & 31));
          };
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const int j = lane + 32 * q;
            cur[q] = j < m ? H[(size_t)l * ld + j] : mk(0.f, 0.f);
            if (j == l) cur[q] = cur[q] - sft;
            nxt[q] = j < m ? H[(size_t)(l + 1) * ld + j] : mk(0.f, 0.f);
            if (j == l + 1) nxt[q] = nxt[q] - sft;
          }
          // sub: the subdiagonal entry H[k+1][k], known a step ahead of its rotation
          cxf sub = own(nxt, l);
          for (int k = l; k < hi && done == 0; ++k) {
            // prefetch row k + 2
            cxf pre[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              const int j = lane + 32 * q;
              pre[q] = (j < m && k + 2 <= hi) ? H[(size_t)(k + 2) * ld + j] : mk(0.f, 0.f);
              if (j == k + 2) pre[q] = pre[q] - sft;
            }
            const cxf a = own(cur, k), b = sub;
            sub = own(pre, k + 1);
            // c = |a| / rho, s = a conj(b) / (|a| rho), rho^2 = |a|^2 + |b|^2
            const float a2 = abs2(a), t = a2 + abs2(b);
            float c;
            cxf s;
            if (a2 > 1e-16f && t < 1e16f) {
              float r1;
              asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(a2 * t));
              c = a2 * r1;
              s = r1 * (a * conj(b));
            } else {
              const float mx = fmaxf(fmaxf(fabsf(a.re), fabsf(a.im)), fmaxf(fabsf(b.re), fabsf(b.im)));
              if (!(mx > 0.f)) {
                c = 1.f;
                s = mk(0.f, 0.f);
              } else {
                const cxf an = mk(a.re / mx, a.im / mx), bn = mk(b.re / mx, b.im / mx);
                const float na = sqrtf(abs2(an)), rho = sqrtf(abs2(an) + abs2(bn));
                c = na / rho;
                s = na > 0.f ? (1.f / (na * rho)) * (an * conj(bn)) : (1.f / rho) * conj(bn);
              }
            }
            if (lane == 0) rot[k] = make_float4(c, s.re, s.im, 0.f);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
              const int j = lane + 32 * q;
              cxf p1, p2;
              p1.re = fmaf(s.re, nxt[q].re, fmaf(-s.im, nxt[q].im, c * cur[q].re));
              p1.im = fmaf(s.re, nxt[q].im, fmaf(s.im, nxt[q].re, c * cur[q].im));
              p2.re = fmaf(-s.re, cur[q].re, fmaf(-s.im, cur[q].im, c * nxt[q].re));
              p2.im = fmaf(-s.re, cur[q].im, fmaf(s.im, cur[q].re, c * nxt[q].im));
              if (j < m && j >= k) H[(size_t)k * ld + j] = p1;
              cur[q] = j <= k ? mk(0.f, 0.f) : p2;
              nxt[q] = pre[q];
            }
          }
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            const int j = lane + 32 * q;
            // row hi, and the annihilated subdiagonal entries
            if (done == 0 && j < m && j >= hi) H[(size_t)hi * ld + j] = cur[q];
            if (done == 0 && j >= l && j < hi) H[(size_t)(j + 1) * ld + j] = mk(0.f, 0.f);
          }
          if (lane == 0) sh_mu = sft;
        }
      }
      if (lane == 0) {
        sh_hi = hi;
        sh_l = l;
        sh_done = done;
      }
    }
    __syncthreads();
    if (sh_done) break;
    const int l = sh_l, hi = sh_hi;
    // right rotations: rows 0..hi of H and every row of Z, a row a thread
    for (int r = tid; r <= hi + m; r += 256) {
      cxf *M = r <= hi ? H + (size_t)r * ld : Z + (size_t)(r - hi - 1) * ld;
      cxf h1 = M[l];
      int k = l;
      for (; k + 4 <= hi; k += 4) {  // four rotations' operands before the first store
        float4 g[4];
        cxf h2[4], o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          g[u] = rot[k + u];
          h2[u] = M[k + u + 1];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) rotate(g[u], h1, h2[u], o[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) M[k + u] = o[u];
      }
      for (; k < hi; ++k) {
        cxf o;
        rotate(rot[k], h1, M[k + 1], o);
        M[k] = o;
      }
      M[hi] = h1;
      if (r >= l && r <= hi) M[r] = M[r] + sh_mu;
    }
    __syncthreads();
  }
  if (sh_done == 2) {
    if (tid == 0) st->failed = 1;
    return;
  }
  // ---- eigenvectors of the triangular T: E (unit upper triangular), kept
  // transposed in the strictly lower part of H: E(j, k) at H[k][j], j < k ----
  const float small = 1e-6f;
  for (int k = tid; k < m; k += 256) {
    const cxf tk = H[(size_t)k * ld + k];
    for (int j = k - 1; j >= 0; --j) {
      cxf s = H[(size_t)j * ld + k];
      for (int q = j + 1; q < k; ++q) cfma(s, H[(size_t)j * ld + q], H[(size_t)k * ld + q]);
      cxf d = H[(size_t)j * ld + j] - tk;
      if (cabs1f(d) < small * FLT_EPSILON) d = mk(small * FLT_EPSILON, 0.f);
      H[(size_t)k * ld + j] = -(s * crecipf(d));
    }
    st->d[0][k] = ccast<double>(tk);
    // ||x_k|| = ||E(:, k)|| (Z is unitary): scaled to about one by a power of two
    float n2 = 1.f;
    for (int j = 0; j < k; ++j) n2 += abs2(H[(size_t)k * ld + j]);
    const int eh = min(max((((__float_as_int(n2) >> 23) & 0xff) - 127) / 2, 0), 60);
    v[k] = mk(__int_as_float((127 - eh) << 23), __int_as_float((127 + eh) << 23));
  }
  __syncthreads();
  // X = Z E, a warp per row of Z in turn
  for (int i = warp; i < m; i += 8) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int k = lane + 32 * q;
      if (k < m) {
        cxf s = Z[(size_t)i * ld + k];
        for (int j = 0; j < k; ++j) cfma(s, Z[(size_t)i * ld + j], H[(size_t)k * ld + j]);
        X[(size_t)i * m + k] = ccast<double>(v[k].re * s);
      }
    }
  }
  __syncthreads();
  // W = E^{-1} Z^H: column c of W solves E w = conj(row c of Z), in place of that row
  for (int c = tid; c < m; c += 256) {
    cxf *zr = Z + (size_t)c * ld;
    for (int k = m - 1; k >= 0; --k) {
      cxf s = conj(zr[k]);
      for (int j = k + 1; j < m; ++j) cfms(s, H[(size_t)j * ld + k], zr[j]);
      zr[k] = s;
      W[(size_t)k * m + c] = ccast<double>(v[k].im * s);
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 products C = A B of m x m complex matrices with an epilogue.  A CTA of
// four warps (one to each sub-partition's FP64 pipe) forms a 4 x 8 tile, a
// lane an entry, the four warps a quarter of the sum each: at m = 64 128 CTAs,
// 16 complex FMAs a thread.
// ---------------------------------------------------------------------------
constexpr int kGm = 4, kGn = 8;

__device__ __forceinline__ cxd tile_dot(const cxd *__restrict__ A, const cxd *__restrict__ B, int m, int i, int j,
                                        bool ok, cxd *sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cxd s = mk(0.0, 0.0);
  if (ok) {
#pragma unroll 8
    for (int k = warp; k < m; k += 4) cfma(s, A[(size_t)i * m + k], B[(size_t)k * m + j]);
  }
  if (warp) sm[(warp - 1) * 32 + lane] = s;
  __syncthreads();
  if (warp == 0) s = (s + sm[lane]) + (sm[32 + lane] + sm[64 + lane]);
  return s;  // valid in warp 0
}

static dim3 tile_grid(int m, int nz = 1) { return dim3(ceil_div(m, kGn), ceil_div(m, kGm), nz); }

// z = 0: R = M X - X diag(d);  z = 1: C = 2 I - W X
__global__ void __launch_bounds__(128) k_eig_resid(int m, const cxd *M, const cxd *X, const cxd *W, cxd *R, cxd *C,
                                                   const EigState *st, int it) {
  __shared__ cxd sm[96];
  if (eig_over(st, it)) return;
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.y * kGm + (lane >> 3), j = blockIdx.x * kGn + (lane & 7);
  const bool ok = i < m && j < m;
  if (blockIdx.z == 0) {
    cxd s = tile_dot(M, X, m, i, j, ok, sm);
    if (threadIdx.x < 32 && ok) {
      cfms(s, X[(size_t)i * m + j], st->d[it & 1][j]);
      R[(size_t)i * m + j] = s;
    }
  } else {
    const cxd s = tile_dot(W, X, m, i, j, ok, sm);
    if (threadIdx.x < 32 && ok) C[(size_t)i * m + j] = mk((i == j ? 2.0 : 0.0) - s.re, -s.im);
  }
}
// z = 0: E = W R -> F_ij = E_ij / (d_j - d_i), d_j += E_jj;  z = 1: W1 = C W
__global__ void __launch_bounds__(128) k_eig_corr(int m, const cxd *W, const cxd *R, const cxd *C, cxd *Fm, cxd *W1,
                                                  EigState *st, int it) {
  __shared__ cxd sm[96];
  if (eig_over(st, it)) return;
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.y * kGm + (lane >> 3), j = blockIdx.x * kGn + (lane & 7);
  const bool ok = i < m && j < m;
  if (blockIdx.z == 0) {
    const cxd e = tile_dot(W, R, m, i, j, ok, sm);
    if (threadIdx.x < 32) {
      float mag = 0.f;
      if (ok) {
        const cxd dj = st->d[it & 1][j];
        cxd f = mk(0.0, 0.0);
        if (i == j) {
          st->d[(it + 1) & 1][j] = dj + e;
        } else if (nonzero(e)) {
          f = e * crecip64(dj - st->d[it & 1][i]);
        }
        Fm[(size_t)i * m + j] = f;
        const cxd chk = i == j ? e : f;  // |E_jj| is small too when it converges
        mag = fmaxf(fabsf((float)chk.re), fabsf((float)chk.im));
        // equal eigenvalues, overflow or NaN: does not converge
        if (!(mag < 1e30f) || chk.re != chk.re || chk.im != chk.im) mag = 1e30f;
        if (i == j && mag < 1e30f) mag = 0.f;
      }
      const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(mag));
      if (lane == 0) atomicMax(&st->fmax[it], mx);
    }
  } else {
    const cxd s = tile_dot(C, W, m, i, j, ok, sm);
    if (threadIdx.x < 32 && ok) W1[(size_t)i * m + j] = s;
  }
}
// z = 0: X1 = X + X F;  z = 1: W2 = W1 - F W1
__global__ void __launch_bounds__(128) k_eig_apply(int m, const cxd *X, const cxd *Fm, const cxd *W1, cxd *X1, cxd *W2,
                                                   const EigState *st, int it) {
  __shared__ cxd sm[96];
  if (eig_over(st, it)) return;
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.y * kGm + (lane >> 3), j = blockIdx.x * kGn + (lane & 7);
  const bool ok = i < m && j < m;
  if (blockIdx.z == 0) {
    const cxd s = tile_dot(X, Fm, m, i, j, ok, sm);
    if (threadIdx.x < 32 && ok) X1[(size_t)i * m + j] = X[(size_t)i * m + j] + s;
  } else {
    const cxd s = tile_dot(Fm, W1, m, i, j, ok, sm);
    if (threadIdx.x < 32 && ok) W2[(size_t)i * m + j] = W1[(size_t)i * m + j] - s;
  }
}
// Eigenpairs of A from those of M, a warp a column: lambda = mu + 2^e d,
// V = D X with unit columns, Vinv = V^{-1} = (norm) W D^{-1}.
__global__ void __launch_bounds__(32) k_eig_finish(int m, const cxd *X0, const cxd *X1, const cxd *W0, const cxd *W1,
                                                   EigState *st, cxd *lam, cxd *V, cxd *Vinv) {
  const int k = blockIdx.x, lane = threadIdx.x;
  int it = -1;
  if (!st->failed)
    for (int q = 0; q < kMaxIt && it < 0; ++q)
      if (!(__uint_as_float(st->fmax[q]) > kFTol)) it = q;
  if (k == 0 && lane == 0) st->done = it >= 0;
  if (it < 0) return;
  const cxd *X = (it & 1) ? X0 : X1, *W = (it & 1) ? W0 : W1;  // iteration `it` wrote the other buffer
  double s = 0.0;
  for (int i = lane; i < m; i += 32) s += abs2(st->dsc[i] * X[(size_t)i * m + k]);
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const double nrm = sqrt(s), inv = s > 0 ? 1.0 / nrm : 1.0;
  for (int i = lane; i < m; i += 32) {
    V[(size_t)i * m + k] = (inv * st->dsc[i]) * X[(size_t)i * m + k];
    if (Vinv) Vinv[(size_t)k * m + i] = (nrm / st->dsc[i]) * W[(size_t)k * m + i];
  }
  if (lane == 0) {
    const cxd d = st->d[(it + 1) & 1][k];
    lam[k] = mk(st->mu.re + scalbn(d.re, st->expo), st->mu.im + scalbn(d.im, st->expo));
  }
}

// Eigenvalues, unit right eigenvectors V and (if Vinv) V^{-1} of the m x m
// matrix A.  work: at least small_eig_work_bytes(); swork: 3 m^2 of the FP64
// kernels.
size_t small_eig_work_bytes() {
  return small_eig_state_bytes() + 9 * (size_t)kMaxM0 * kMaxM0 * sizeof(cxd);
}
void small_eig(const cxd *A, int m, cxd *lam, cxd *V, cxd *Vinv, cxd *swork, void *work, int *d_err, cudaStream_t s) {
  if (m < 4) {  // one QR launch is shorter than the chain below (m = 3: 95 us against 120)
    cudaMemsetAsync(work, 0, offsetof(EigState, dsc), s);
    small_eig_qr(A, m, lam, V, swork, d_err, nullptr, s);
    if (Vinv) small_inv(V, m, Vinv, swork, d_err, nullptr, s);
    return;
  }
  EigState *st = reinterpret_cast<EigState *>(work);
  const size_t mm = (size_t)m * m;
  cxd *b = reinterpret_cast<cxd *>(reinterpret_cast<unsigned char *>(work) + small_eig_state_bytes());
  cxd *M = b, *X[2] = {b + mm, b + 2 * mm}, *W[2] = {b + 3 * mm, b + 4 * mm}, *R = b + 5 * mm, *C = b + 6 * mm,
      *Fm = b + 7 * mm, *W1 = b + 8 * mm;
  cudaMemsetAsync(st, 0, offsetof(EigState, dsc), s);
  const size_t hb = (size_t)m * (m | 1) * sizeof(cxf);
  const int zsm = 2 * hb <= 200 * 1024;
  const size_t smem = zsm ? 2 * hb : hb;
  const int Q = ceil_div(m, 32);
#define EIG32(q)                                                                                                   \
  do {                                                                                                             \
    cudaFuncSetAttribute(k_eig32<q>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);                     \
    k_eig32<q><<<1, 256, smem, s>>>(A, m, M, X[0], W[0], reinterpret_cast<cxf *>(W1), zsm, st);                    \
  } while (0)
  if (Q == 1) EIG32(1);
  else if (Q == 2) EIG32(2);
  else if (Q == 3) EIG32(3);
  else EIG32(4);
#undef EIG32
  note_launch();
  const dim3 grid = tile_grid(m, 2);
  for (int it = 0; it < kMaxIt; ++it) {
    const int a = it & 1;
    k_eig_resid<<<grid, 128, 0, s>>>(m, M, X[a], W[a], R, C, st, it);
    note_launch();
    k_eig_corr<<<grid, 128, 0, s>>>(m, W[a], R, C, Fm, W1, st, it);
    note_launch();
    k_eig_apply<<<grid, 128, 0, s>>>(m, X[a], Fm, W1, X[a ^ 1], W[a ^ 1], st, it);
    note_launch();
  }
  k_eig_finish<<<m, 32, 0, s>>>(m, X[0], X[1], W[0], W[1], st, lam, V, Vinv);
  note_launch();
  small_eig_qr(A, m, lam, V, swork, d_err, &st->done, s);
  if (Vinv) small_inv(V, m, Vinv, swork, d_err, &st->done, s);
}

// ---------------------------------------------------------------------------
// products and inverses of the reduced problem
// ---------------------------------------------------------------------------
// C = A B (herm: C = (A B)^H)
__global__ void __launch_bounds__(128) k_small_prod(int m, const cxd *A, const cxd *B, cxd *C, int herm) {
  __shared__ cxd sm[96];
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.y * kGm + (lane >> 3), j = blockIdx.x * kGn + (lane & 7);
  const bool ok = i < m && j < m;
  const cxd s = tile_dot(A, B, m, i, j, ok, sm);
  if (threadIdx.x < 32 && ok) {
    if (herm)
      C[(size_t)j * m + i] = conj(s);
    else
      C[(size_t)i * m + j] = s;
  }
}
void small_prod(int m, const cxd *A, const cxd *B, cxd *C, int herm, cudaStream_t s) {
  k_small_prod<<<tile_grid(m), 128, 0, s>>>(m, A, B, C, herm);
  note_launch();
}

// X0 = 2 I - B and *near = 1 when m max|B - I| <= 1e-3, so that ||I - B X0||
// <= 1e-6 and two Newton-Schulz steps end at 1e-24 (one CTA).
__global__ void __launch_bounds__(512) k_inv_start(int m, const cxd *B, cxd *X0, int *near) {
  __shared__ int far;
  if (threadIdx.x == 0) far = 0;
  __syncthreads();
  bool f = false;
  const double lim = 1e-3 / m;
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
    const cxd b = B[e];
    const double one = e / m == e % m ? 1.0 : 0.0;
    if (!(fabs(b.re - one) + fabs(b.im) <= lim)) f = true;
    X0[e] = mk(2.0 * one - b.re, -b.im);
  }
  if (f) far = 1;
  __syncthreads();
  if (threadIdx.x == 0) *near = far ? 0 : 1;
}
// mode 0: C = 2 I - A B;  mode 1: C = A B
__global__ void __launch_bounds__(128) k_inv_step(int m, const cxd *A, const cxd *B, cxd *C, int mode,
                                                  const int *near) {
  __shared__ cxd sm[96];
  if (!*near) return;
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.y * kGm + (lane >> 3), j = blockIdx.x * kGn + (lane & 7);
  const bool ok = i < m && j < m;
  const cxd s = tile_dot(A, B, m, i, j, ok, sm);
  if (threadIdx.x < 32 && ok)
    C[(size_t)i * m + j] = mode ? s : mk((i == j ? 2.0 : 0.0) - s.re, -s.im);
}
// Binv = B^{-1} for a matrix that is usually within 1e-3 of the identity.
// work as for small_eig.
void small_inv_near(const cxd *B, int m, cxd *Binv, cxd *swork, void *work, int *d_err, cudaStream_t s) {
  EigState *st = reinterpret_cast<EigState *>(work);
  cxd *b = reinterpret_cast<cxd *>(reinterpret_cast<unsigned char *>(work) + small_eig_state_bytes());
  const size_t mm = (size_t)m * m;
  cxd *X0 = b, *C = b + mm, *X1 = b + 2 * mm;
  k_inv_start<<<1, 512, 0, s>>>(m, B, X0, &st->near);
  note_launch();
  k_inv_step<<<tile_grid(m), 128, 0, s>>>(m, B, X0, C, 0, &st->near);
  k_inv_step<<<tile_grid(m), 128, 0, s>>>(m, X0, C, X1, 1, &st->near);
  k_inv_step<<<tile_grid(m), 128, 0, s>>>(m, B, X1, C, 0, &st->near);
  k_inv_step<<<tile_grid(m), 128, 0, s>>>(m, X1, C, Binv, 1, &st->near);
  for (int k = 0; k < 4; ++k) note_launch();
  small_inv(B, m, Binv, swork, d_err, &st->near, s);
}

cudaError_t small_forms(const void *work, int *refined, int *near, cudaStream_t s) {
  const EigState *st = reinterpret_cast<const EigState *>(work);
  cudaError_t e = cudaMemcpyAsync(refined, &st->done, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(near, &st->near, sizeof(int), cudaMemcpyDeviceToHost, s);
  return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}

// Complex symmetric reduced problem (Sec. 2.4): W scaled so that w^T B_U w = 1,
// Wh = conj(W).  BW = B_U W (small_prod); a warp a column.
__global__ void __launch_bounds__(32) k_cs_wnorm(int m, const cxd *BW, cxd *W, cxd *Wh) {
  const int k = blockIdx.x, lane = threadIdx.x;
  cxd s = mk(0.0, 0.0);
  for (int a = lane; a < m; a += 32) cfma(s, W[(size_t)a * m + k], BW[(size_t)a * m + k]);
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
    s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
  }
  const cxd t = csqrt(s);
  for (int a = lane; a < m; a += 32) {
    const cxd v = cdiv(W[(size_t)a * m + k], t);
    W[(size_t)a * m + k] = v;
    Wh[(size_t)a * m + k] = conj(v);
  }
}
void launch_cs_wnorm(int m, const cxd *BU, cxd *W, cxd *Wh, cxd *BW, cudaStream_t s) {
  small_prod(m, BU, W, BW, 0, s);
  k_cs_wnorm<<<m, 32, 0, s>>>(m, BW, W, Wh);
  note_launch();
}

// ---------------------------------------------------------------------------
// Bi-orthonormalising coefficients without the eigendecomposition of B_Q.
//
// The paper forms U = Q V Gamma^{-1/2}, Uh = Qh Vh Gamma^{-H/2} from B_Q = V
// Gamma Vh^H (eq. uu); any S, Sh with Sh^H B_Q S = I give blocks of the same
// spans with Uh^H B U = I, and the reduced problem's pairs depend on the spans
// alone.  The eigenvalues themselves are needed only for the resize (eq.
// resize), which drops columns with |gamma_i| < eta max|gamma|.  Elimination
// with complete pivoting, Lacc B_Q Uacc = diag(p) (up to the order), gives S =
// Uacc p^{-1/2}, Sh^H = p^{-1/2} Lacc, and with them a bound on every
// eigenvalue: |gamma| <= ||B_Q||_F and |gamma| >= 1 / ||B_Q^{-1}||_F >=
// 1 / (||S||_F ||Sh||_F).  If eta ||B_Q|| ||S|| ||Sh|| <= 0.01 and eta >= 1e-17
// decides nothing closer than FP64 resolves (||B_Q|| ||S|| ||Sh|| <= 1e13), no
// column can be dropped and *ok = 1; otherwise the caller takes the
// eigendecomposition.
//
// One cluster of 8 CTAs, columns dealt out cyclically, in shared memory.  A
// step is: each CTA's largest unpivoted entry (by the high word of its larger
// component: integer compares); exchange; the winner's CTA forms the
// multipliers and sends them with its column of Uacc to the others; everyone
// updates its columns.  Two cluster barriers a step.  m = 64: the eigen-
// decomposition (8.8 ms on the graded B_Q of a solve) and the inverse of V
// (0.75 ms) are not needed any more.
// ---------------------------------------------------------------------------
namespace cg = cooperative_groups;
constexpr int kBoC = 8, kBoT = 256, kBoCols = kMaxM0 / kBoC;
struct BiorthSmem {
  cxd B[kMaxM0][kBoCols], L[kMaxM0][kBoCols], U[kMaxM0][kBoCols];
  cxd lc[2][kMaxM0], uc[2][kMaxM0];  // multipliers and pivot column of Uacc over the pivot, by step parity
  unsigned long long cand[2][kBoC];
  unsigned long long wred[kBoT / 32];
  double nrm[kBoC][3];
  double dred[kBoT / 32];
  cxd piv[kMaxM0];
  short prow[kMaxM0], pcol[kMaxM0];
  unsigned char rdone[kMaxM0], cdone[kMaxM0];
};
__global__ void __cluster_dims__(kBoC, 1, 1) __launch_bounds__(kBoT)
    k_biorth(int m, const cxd *__restrict__ BQ, const cxd *__restrict__ prev_rho, const int *__restrict__ prev_inside,
             int have_prev, double mu, double eta, cxd *__restrict__ S, cxd *__restrict__ Sh, RRStatus *st) {
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  extern __shared__ __align__(16) unsigned char dsm[];
  BiorthSmem &sm = *reinterpret_cast<BiorthSmem *>(dsm);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nc = (m - rank + kBoC - 1) / kBoC;  // own columns rank, rank + 8, ...
  double b2 = 0.0;
  for (int e = tid; e < m * nc; e += kBoT) {
    const int i = e / nc, jl = e - i * nc, j = rank + kBoC * jl;
    const cxd b = BQ[(size_t)i * m + j];
    b2 += abs2(b);
    sm.B[i][jl] = b;
    sm.L[i][jl] = sm.U[i][jl] = mk(i == j ? 1.0 : 0.0, 0.0);
  }
  if (tid < m) sm.rdone[tid] = sm.cdone[tid] = 0;
  cl.sync();
  for (int k = 0; k < m; ++k) {
    const int par = k & 1;
    // own largest entry: key = high word of max(|re|, |im|), then position
    unsigned long long best = 0;
    for (int e = tid; e < m * nc; e += kBoT) {
      const int i = e / nc, jl = e - i * nc;
      if (sm.rdone[i] || sm.cdone[rank + kBoC * jl]) continue;
      const cxd b = sm.B[i][jl];
      const unsigned h = (unsigned)max(__double2hiint(b.re) & 0x7fffffff, __double2hiint(b.im) & 0x7fffffff);
      const unsigned long long key = ((unsigned long long)h << 32) | (unsigned)(0xffff - (i * kMaxM0 + rank + kBoC * jl)) | 0x10000u;
      best = key > best ? key : best;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const unsigned long long other = __shfl_xor_sync(0xffffffffu, best, o);
      best = other > best ? other : best;
    }
    if (lane == 0) sm.wred[warp] = best;
    __syncthreads();
    if (tid < kBoC) {
      unsigned long long b = 0;
      for (int w = 0; w < kBoT / 32; ++w) b = sm.wred[w] > b ? sm.wred[w] : b;
      cl.map_shared_rank(&sm.cand[par][0], tid)[rank] = b;
    }
    cl.sync();
    unsigned long long win = 0;
    for (int r = 0; r < kBoC; ++r) win = sm.cand[par][r] > win ? sm.cand[par][r] : win;
    const int at = 0xffff - (int)(win & 0xffff), pr = at / kMaxM0, pc = at - pr * kMaxM0;
    if (pc % kBoC == rank) {
      const int jl = pc / kBoC;
      const cxd p = sm.B[pr][jl];
      if (tid < m) {
        const int i = tid;
        const cxd pi = crecip64(p);
        const cxd l = (i == pr || sm.rdone[i]) ? mk(0.0, 0.0) : sm.B[i][jl] * pi;
        const cxd u = nonzero(sm.U[i][jl]) ? sm.U[i][jl] * pi : mk(0.0, 0.0);
#pragma unroll
        for (int r = 0; r < kBoC; ++r) {
          BiorthSmem *o = cl.map_shared_rank(&sm, r);
          o->lc[par][i] = l;
          o->uc[par][i] = u;
        }
      }
      if (tid < kBoC) {
        BiorthSmem *o = cl.map_shared_rank(&sm, tid);
        o->piv[k] = p;
      }
    }
    cl.sync();
    // own columns: B[i][j] -= l_i B[pr][j]; L[i][j] -= l_i L[pr][j];
    // U[i][j] -= B[pr][j] (U[i][pc] / p) for the unpivoted columns j != pc
    for (int e = tid; e < m * nc; e += kBoT) {
      const int i = e / nc, jl = e - i * nc, j = rank + kBoC * jl;
      const bool open = !sm.cdone[j] && j != pc;
      const cxd l = sm.lc[par][i];
      const bool row = nonzero(l);
      const cxd lp = sm.L[pr][jl];
      if (row && nonzero(lp)) cfms(sm.L[i][jl], l, lp);
      if (open) {
        const cxd bp = sm.B[pr][jl];
        const cxd u = sm.uc[par][i];
        if (row) cfms(sm.B[i][jl], l, bp);
        if (nonzero(u)) cfms(sm.U[i][jl], bp, u);
      }
    }
    __syncthreads();  // row pr is read above by every thread and never written
    if (tid == 0) {
      sm.rdone[pr] = 1;
      sm.cdone[pc] = 1;
      sm.prow[k] = (short)pr;
      sm.pcol[k] = (short)pc;
    }
    __syncthreads();
  }
  // S[:, k] = U[:, pc_k] / sqrt(p_k), Sh[:, k] = conj(L[pr_k, :] / sqrt(p_k)); norms
  double s2 = 0.0, h2 = 0.0;
  for (int k = warp; k < m; k += kBoT / 32) {
    const int pr = sm.prow[k], pc = sm.pcol[k];
    const cxd ri = cdiv(mk(1.0, 0.0), csqrt(sm.piv[k]));
    if (pc % kBoC == rank)
      for (int i = lane; i < m; i += 32) {
        const cxd v = sm.U[i][pc / kBoC] * ri;
        S[(size_t)i * m + k] = v;
        s2 += abs2(v);
      }
    for (int jl = lane; jl < nc; jl += 32) {
      const cxd v = conj(sm.L[pr][jl] * ri);
      Sh[(size_t)(rank + kBoC * jl) * m + k] = v;
      h2 += abs2(v);
    }
  }
  double tot[3] = {b2, s2, h2};
  for (int q = 0; q < 3; ++q) {
    double t = tot[q];
#pragma unroll
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    __syncthreads();
    if (lane == 0) sm.dred[warp] = t;
    __syncthreads();
    if (tid == 0) {
      t = 0.0;
      for (int w = 0; w < kBoT / 32; ++w) t += sm.dred[w];
      cl.map_shared_rank(&sm.nrm[0][0], 0)[rank * 3 + q] = t;
    }
  }
  cl.sync();
  if (rank == 0) {
    // spurious test of Sec. 2.7 against the previous Ritz values
    bool spur = false;
    if (tid < m && have_prev && prev_inside[tid]) {
      const cxd r2 = prev_rho[tid] * prev_rho[tid];
      const double den = cabs(r2);
      const double q = den > 0 ? cabs(r2 - BQ[(size_t)tid * m + tid]) / den : INFINITY;
      spur = !(q < mu);
    }
    const int ms = __syncthreads_count(spur);
    if (tid == 0) {
      double t[3] = {0.0, 0.0, 0.0};
      for (int r = 0; r < kBoC; ++r)
        for (int q = 0; q < 3; ++q) t[q] += sm.nrm[r][q];
      const double cond = sqrt(t[0]) * sqrt(t[1]) * sqrt(t[2]);
      const bool ok = cond <= 1e13 && eta * cond <= 0.01;
      st->m_s = ms;
      st->m_tilde = ok ? m : 0;
      st->biorth = ok ? 1 : 0;
    }
  }
}
cudaError_t launch_biorth(int m, const cxd *BQ, const cxd *prev_rho, const int *prev_inside, int have_prev, double mu,
                          double eta, cxd *S, cxd *Sh, RRStatus *st, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_biorth, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(BiorthSmem));
  if (e != cudaSuccess) return e;
  k_biorth<<<kBoC, kBoT, sizeof(BiorthSmem), s>>>(m, BQ, prev_rho, prev_inside, have_prev, mu, eta, S, Sh, st);
  note_launch();
  return cudaGetLastError();
}
