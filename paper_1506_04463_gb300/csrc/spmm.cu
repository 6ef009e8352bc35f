// Sparse products of the contour filter and of the Rayleigh-Ritz step.
//
//  * k_multishift_residual: one pass over A (and B) applies every shift z_j
//    to every column: R_j = B Y - (z_j B - A) X_j, the residual of the shifted
//    systems of eq. (qr) for all quadrature nodes at once, and optionally
//    the filtered block Q = sum_j w_j X_j (eq. qr) in fixed node order.
//  * k_node_sum: Q = sum_j w_j X_j alone, once per filter in the refined form.
//  * k_spmm: Out = M1 X - s_c M2 X with a per-column shift, used for B Q,
//    A U, B U and the eigen-residuals of eq. (res).
//  * csr transpose for the conjugate-transpose products A^H, B^H (eq. ql and
//    the left residual of eq. res).
#include <algorithm>
#include <type_traits>
#include "kernels.h"
#include "reduce.cuh"

template <bool CPLX>
__device__ __forceinline__ void csr_fma(cxd &acc, const CsrView &M, int64_t k, const cxd &x) {
  if (CPLX) {
    cxd v = reinterpret_cast<const cxd *>(M.val)[k];
    if (M.conj_vals) v.im = -v.im;
    cfma(acc, v, x);
  } else {
    const double v = M.val[k];
    acc.re = fma(v, x.re, acc.re);
    acc.im = fma(v, x.im, acc.im);
  }
}

// ---------------------------------------------------------------------------
// multi-shift residual + node accumulation
// ---------------------------------------------------------------------------
// Bound by the FP64 pipe, which a warp instruction takes for 64 cycles whatever
// the lanes it serves, so FP64 instructions are what counts: without B the
// diagonal entries of A are folded into the shifts (z_j - a_ii, once a row and
// node instead of once a column), the squares go into their sum as two FMAs,
// and Q is formed for eight rows at a time with full warps.  The rows' other
// entries are staged, so that the gathers of a row are issued together; four
// CTAs an SM, since fewer registers spill.  n = 44521, 15 nodes, 45 columns,
// 5 entries a row, with Q: 1348 -> 989 us; n = 90000, 16 nodes, 62 columns,
// FP32 residual without Q: 2.95 -> 2.66 ms (bound by the conversions to and
// from FP32 and 12 FMAs, 2.5 ms).
constexpr int kMsThreads = 256;
constexpr int kMsMaxPairs = 8;  // ne*m <= 2048
constexpr int kMsRows = 8;      // rows between two barriers
constexpr int kMsStage = 160;   // entries of A they may have to be staged

// LONG: rows of more than 128 entries on average, nothing staged or folded, since
// the search for the diagonal takes more than it saves there (600 full rows, 8
// nodes, 1, 13 and 32 columns 170, 226 and 384 us folded, 142, 175 and 335 so).
template <typename Tout, bool ACPLX, bool BCPLX, bool HASB, bool LONG = false>
__global__ void __launch_bounds__(kMsThreads, 4)
    k_multishift_residual(CsrView A, CsrView B, int ne, const cxd *__restrict__ z,
                          const cxd *__restrict__ w, const cxd *__restrict__ X, size_t xns,
                          const cxd *__restrict__ BY, cx<Tout> *__restrict__ R, cxd *__restrict__ Q,
                          double *__restrict__ partial, int m, int rows_per_cta, const int *skip) {
  if (skip && *skip) return;
  using Val = typename std::conditional<ACPLX, cxd, double>::type;
  constexpr bool FOLD = !HASB && !LONG;
  __shared__ cxd ws[kMaxNe], zs[FOLD ? kMsRows : 1][kMaxNe];
  __shared__ Val sval[kMsStage];
  __shared__ int scol[kMsStage], sbeg[kMsRows], send[kMsRows];
  const int tid = threadIdx.x;
  if (tid < ne) {
    ws[tid] = w[tid];
    if (!FOLD) zs[0][tid] = z[tid];
  }
  const int P = ne * m;
  const int n = A.n;
  const int rbeg = blockIdx.x * rows_per_cta;
  const int rend = min(n, rbeg + rows_per_cta);
  double nacc[kMsMaxPairs];
#pragma unroll
  for (int q = 0; q < kMsMaxPairs; ++q) nacc[q] = 0.0;

  for (int i0 = rbeg; i0 < rend; i0 += kMsRows) {
    const int rows = min(kMsRows, rend - i0);
    const int64_t k0 = A.rowptr[i0];
    const bool staged = !LONG && A.rowptr[i0 + rows] - k0 <= kMsStage;
    __syncthreads();
    if (FOLD) {
      // z_j - a_ii of the chunk's rows (entries of one position add up)
      for (int e = tid; e < rows * ne; e += kMsThreads) {
        const int r = e / ne, j = e - r * ne, i = i0 + r;
        cxd d = z[j];
        for (int64_t k = A.rowptr[i]; k < A.rowptr[i + 1]; ++k)
          if (A.colind[k] == i) d = d - csr_val(A, k);
        zs[r][j] = d;
      }
    }
    if (staged && tid < 32 * rows && (tid & 31) == 0) {
      const int r = tid >> 5, i = i0 + r;
      int o = (int)(A.rowptr[i] - k0);
      sbeg[r] = o;
      for (int64_t k = A.rowptr[i]; k < A.rowptr[i + 1]; ++k) {
        const int col = A.colind[k];
        if (FOLD && col == i) continue;
        scol[o] = col;
        if constexpr (ACPLX) sval[o] = csr_val(A, k); else sval[o] = A.val[k];
        ++o;
      }
      send[r] = o;
    }
    __syncthreads();
    for (int r = 0; r < rows; ++r) {
      const int i = i0 + r;
#pragma unroll
      for (int q = 0; q < kMsMaxPairs; ++q) {
        const int pair = tid + kMsThreads * q;
        if (pair < P) {
          const int j = pair / m, c = pair - j * m;
          const cxd *Xj = X + (size_t)j * xns + c;
          cxd acc = BY ? BY[(size_t)i * m + c] : mk(0.0, 0.0);
          if (HASB) {
            cxd bx = mk(0.0, 0.0);
            for (int64_t k = B.rowptr[i]; k < B.rowptr[i + 1]; ++k)
              csr_fma<BCPLX>(bx, B, k, Xj[(size_t)B.colind[k] * m]);
            cfms(acc, zs[0][j], bx);
          } else {
            cfms(acc, zs[FOLD ? r : 0][j], Xj[(size_t)i * m]);
          }
          if (staged) {
            const int ke = send[r];
#pragma unroll 4
            for (int k = sbeg[r]; k < ke; ++k) {
              const cxd x = Xj[(size_t)scol[k] * m];
              if constexpr (ACPLX) {
                cfma(acc, sval[k], x);
              } else {
                acc.re = fma(sval[k], x.re, acc.re);
                acc.im = fma(sval[k], x.im, acc.im);
              }
            }
          } else {
            for (int64_t k = A.rowptr[i]; k < A.rowptr[i + 1]; ++k) {
              const int col = A.colind[k];
              if (!FOLD || col != i) csr_fma<ACPLX>(acc, A, k, Xj[(size_t)col * m]);
            }
          }
          const cx<Tout> ro = ccast<Tout>(acc);
          if (R) R[(size_t)j * xns + (size_t)i * m + c] = ro;
          // the norm of the stored residual, squared in its own precision
          if constexpr (sizeof(Tout) == 8)
            nacc[q] = fma(ro.re, ro.re, fma(ro.im, ro.im, nacc[q]));
          else
            nacc[q] += (double)(ro.re * ro.re + ro.im * ro.im);
        }
      }
    }
    if (Q) {
      for (int e = tid; e < rows * m; e += kMsThreads) {
        const size_t o = (size_t)i0 * m + e;
        cxd qv = mk(0.0, 0.0);
#pragma unroll 4
        for (int j = 0; j < ne; ++j) cfma(qv, ws[j], X[(size_t)j * xns + o]);
        Q[o] = qv;
      }
    }
  }
  if (partial) {
#pragma unroll
    for (int q = 0; q < kMsMaxPairs; ++q) {
      const int pair = tid + kMsThreads * q;
      if (pair < P) partial[(size_t)blockIdx.x * P + pair] = nacc[q];
    }
  }
}

// Q = sum_j w_j X_j (eq. q00 with the nodes' solutions), row-major n x m,
// nodes summed in fixed order
__global__ void k_node_sum(int ne, const cxd *__restrict__ w, const cxd *__restrict__ X, size_t xns, size_t nm,
                           cxd *__restrict__ Q) {
  __shared__ cxd ws[kMaxNe];
  if (threadIdx.x < ne) ws[threadIdx.x] = w[threadIdx.x];
  __syncthreads();
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nm; e += (size_t)gridDim.x * blockDim.x) {
    cxd q = mk(0.0, 0.0);
    for (int j = 0; j < ne; ++j) cfma(q, ws[j], X[(size_t)j * xns + e]);
    Q[e] = q;
  }
}
void launch_node_sum(int ne, const cxd *d_w, const cxd *X, size_t xns, int n, int m, cxd *Q, cudaStream_t s) {
  const size_t nm = (size_t)n * m;
  k_node_sum<<<grid_for(nm), 256, 0, s>>>(ne, d_w, X, xns, nm, Q);
  note_launch();
}
// complex128 -> complex64 copy (single-precision right-hand sides)
__global__ void k_to_cxf(const cxd *__restrict__ X, cxf *__restrict__ Y, size_t count) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
    Y[e] = ccast<float>(X[e]);
}
void launch_to_cxf(const cxd *X, cxf *Y, size_t count, cudaStream_t s) {
  k_to_cxf<<<grid_for(count), 256, 0, s>>>(X, Y, count);
  note_launch();
}

int spmm_max_grid() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms * 8;
}

static int ms_grid(int n) {
  int g = spmm_max_grid();
  if (g > n) g = n;
  return g < 1 ? 1 : g;
}

#define MS_LAUNCH(AC, BC, HB, LG, SKIP)                                                                     \
  k_multishift_residual<Tout, AC, BC, HB, LG><<<g, kMsThreads, 0, s>>>(A, Bv, ne, d_z, d_w, X, xns, BY, R, Q, \
                                                                       partial, m, rpc, SKIP)
#define MS_CALL(SKIP)                                                                                       \
  do {                                                                                                      \
    if (!B && A.nnz > 128 * (int64_t)A.n) {                                                                 \
      if (A.cplx) MS_LAUNCH(true, false, false, true, SKIP); else MS_LAUNCH(false, false, false, true, SKIP); \
    } else if (!B) {                                                                                        \
      if (A.cplx) MS_LAUNCH(true, false, false, false, SKIP); else MS_LAUNCH(false, false, false, false, SKIP); \
    } else if (A.cplx) {                                                                                    \
      if (bc) MS_LAUNCH(true, true, true, false, SKIP); else MS_LAUNCH(true, false, true, false, SKIP);     \
    } else {                                                                                                \
      if (bc) MS_LAUNCH(false, true, true, false, SKIP); else MS_LAUNCH(false, false, true, false, SKIP);   \
    }                                                                                                       \
  } while (0)

template <typename Tout>
int launch_multishift_residual(const CsrView &A, const CsrView *B, int ne, const cxd *d_z, const cxd *d_w,
                               const cxd *X, const cxd *BY, cx<Tout> *R, cxd *Q, double *partial, int m,
                               const int *d_skip, cudaStream_t s) {
  const int grid = ms_grid(A.n);
  const int rpc = ceil_div(A.n, grid);
  const int g = ceil_div(A.n, rpc);
  const size_t xns = (size_t)A.n * m;
  CsrView Bv = B ? *B : A;
  const bool bc = B ? B->cplx : false;
  MS_CALL(d_skip);
  note_launch();
  return g;
}
template int launch_multishift_residual<double>(const CsrView &, const CsrView *, int, const cxd *, const cxd *,
                                                const cxd *, const cxd *, cxd *, cxd *, double *, int, const int *,
                                                cudaStream_t);
template int launch_multishift_residual<float>(const CsrView &, const CsrView *, int, const cxd *, const cxd *,
                                               const cxd *, const cxd *, cxf *, cxd *, double *, int, const int *,
                                               cudaStream_t);

// Relative residual of every (side, node, column): ||R||_2 / ||B Y||_2, summed
// over the per-CTA partials in fixed order; the maximum is folded in with an
// integer atomicMax on the bits of the (non-negative) double, which is
// order-independent.
// Same product with the grid capped at max_grid CTAs, so that the partial
// sums fit a caller-provided buffer of max_grid * ne * m doubles.
template <typename Tout>
int launch_multishift_residual_capped(const CsrView &A, const CsrView *B, int ne, const cxd *d_z, const cxd *d_w,
                                      const cxd *X, const cxd *BY, cx<Tout> *R, cxd *Q, double *partial, int m,
                                      int max_grid, cudaStream_t s) {
  int grid = ms_grid(A.n);
  if (grid > max_grid) grid = max_grid;
  const int rpc = ceil_div(A.n, grid);
  const int g = ceil_div(A.n, rpc);
  const size_t xns = (size_t)A.n * m;
  CsrView Bv = B ? *B : A;
  const bool bc = B ? B->cplx : false;
  MS_CALL(nullptr);
  note_launch();
  return g;
}
template int launch_multishift_residual_capped<double>(const CsrView &, const CsrView *, int, const cxd *,
                                                       const cxd *, const cxd *, const cxd *, cxd *, cxd *, double *,
                                                       int, int, cudaStream_t);
#undef MS_CALL
#undef MS_LAUNCH

// One CTA per 4 (node, column) pairs, 64 threads a pair: at 1216 partials and
// 2048 pairs this took 179 us with a thread per pair (a chain of 1216 loads);
// spread out it is bound by reading the 20 MB of partials from L2.
constexpr int kRelC = 4, kRelR = 64;
__global__ void __launch_bounds__(kRelC *kRelR) k_residual_rel(const double *__restrict__ partial, int nparts, int P,
                                                               int m, const double *bynorm2, int nsides,
                                                               unsigned long long *maxbits) {
  __shared__ double sm[kRelC * kRelR];
  const int sp = blockIdx.x * kRelC + threadIdx.x % kRelC;
  const bool ok = sp < nsides * P;
  const int side = ok ? sp / P : 0, pair = ok ? sp - side * P : 0;
  const double s = column_sum<kRelC, kRelR>(partial + (size_t)side * nparts * P, nparts, P, pair, ok, sm);
  if (ok && threadIdx.x < kRelC) {
    const double d = bynorm2[side * m + pair % m];
    const double rel = d > 0 ? sqrt(s / d) : sqrt(s);
    const double mx = (rel == rel) ? rel : INFINITY;
    atomicMax(maxbits, (unsigned long long)__double_as_longlong(mx));
  }
}

void launch_residual_check(const double *partial, int nparts, int ne, int m, const double *bynorm2, int nsides,
                           double *d_maxrel, cudaStream_t s) {
  // d_maxrel doubles as the atomic accumulator (bits of a non-negative double)
  unsigned long long *bits = reinterpret_cast<unsigned long long *>(d_maxrel);
  cudaMemsetAsync(bits, 0, sizeof(unsigned long long), s);
  const int total = nsides * ne * m;
  k_residual_rel<<<ceil_div(total, kRelC), kRelC * kRelR, 0, s>>>(partial, nparts, ne * m, m, bynorm2, nsides, bits);
  note_launch();
}

// ---------------------------------------------------------------------------
// single-shift products with per-column shift and column 1-norms
// ---------------------------------------------------------------------------
// |z|: the square root of |z|^2 where that neither over- nor underflows (by the
// exponent field of the larger component, an integer test), else hypot, which
// takes three times the FP64 instructions.
__device__ __forceinline__ double modulus(cxd z) {
  const int e = max(__double2hiint(z.re) & 0x7fffffff, __double2hiint(z.im) & 0x7fffffff) >> 20;
  if (e > 1023 - 400 && e < 1023 + 400) return sqrt(fma(z.re, z.re, z.im * z.im));
  return hypot(z.re, z.im);
}

// NORMS: also the per-CTA column 1-norms of Out and of M2 X (the residuals of
// eq. res); the FP64 pipe bounds them, so products that don't need them (A U,
// B Q) leave them out: 90 000 x 64, 5 entries a row, 490 us with both norms
// by hypot.
template <bool C1, bool C2, bool NORMS>
__global__ void __launch_bounds__(256) k_spmm(CsrView M1, CsrView M2, int hasM2, const cxd *__restrict__ shift,
                                              const cxd *__restrict__ X, cxd *__restrict__ Out, int m,
                                              int rows_per_cta, double *p1, double *p2) {
  __shared__ double r1[256], r2[256];
  const int tid = threadIdx.x;
  const int lanes = 256 / m;  // m <= 128 -> lanes >= 2
  const int c = tid % m, lr = tid / m;
  const bool active = lr < lanes;
  const int n = M1.n;
  const int rbeg = blockIdx.x * rows_per_cta, rend = min(n, rbeg + rows_per_cta);
  double a1 = 0.0, a2 = 0.0;
  const cxd sh = (shift && active) ? shift[c] : mk(0.0, 0.0);
  if (active) {
    for (int i = rbeg + lr; i < rend; i += lanes) {
      cxd acc = mk(0.0, 0.0);
      for (int64_t k = M1.rowptr[i]; k < M1.rowptr[i + 1]; ++k)
        csr_fma<C1>(acc, M1, k, X[(size_t)M1.colind[k] * m + c]);
      cxd bx;
      if (hasM2) {
        bx = mk(0.0, 0.0);
        for (int64_t k = M2.rowptr[i]; k < M2.rowptr[i + 1]; ++k)
          csr_fma<C2>(bx, M2, k, X[(size_t)M2.colind[k] * m + c]);
      } else {
        bx = X[(size_t)i * m + c];
      }
      if (shift) cfms(acc, sh, bx);
      Out[(size_t)i * m + c] = acc;
      if (NORMS) {
        a1 += modulus(acc);
        a2 += modulus(bx);
      }
    }
  }
  if (!NORMS) return;
  r1[tid] = a1;
  r2[tid] = a2;
  __syncthreads();
  if (tid < m) {
    double s1 = 0.0, s2 = 0.0;
    for (int l = 0; l < lanes; ++l) {
      s1 += r1[l * m + tid];
      s2 += r2[l * m + tid];
    }
    p1[(size_t)blockIdx.x * m + tid] = s1;
    if (p2) p2[(size_t)blockIdx.x * m + tid] = s2;
  }
}

int launch_spmm(const CsrView &M1, const CsrView *M2, const cxd *shift, const cxd *X, cxd *Out, int m, double *p1,
                double *p2, cudaStream_t s) {
  const int grid = ms_grid(M1.n);
  const int rpc = ceil_div(M1.n, grid);
  const int g = ceil_div(M1.n, rpc);
  CsrView M2v = M2 ? *M2 : M1;
  const bool c2 = M2 ? M2->cplx : false;
#define SP_LAUNCH(A1, A2)                                                                                        \
  do {                                                                                                           \
    if (p1)                                                                                                      \
      k_spmm<A1, A2, true><<<g, 256, 0, s>>>(M1, M2v, M2 != nullptr, shift, X, Out, m, rpc, p1, p2);             \
    else                                                                                                         \
      k_spmm<A1, A2, false><<<g, 256, 0, s>>>(M1, M2v, M2 != nullptr, shift, X, Out, m, rpc, nullptr, nullptr);  \
  } while (0)
  if (M1.cplx) {
    if (c2) SP_LAUNCH(true, true); else SP_LAUNCH(true, false);
  } else {
    if (c2) SP_LAUNCH(false, true); else SP_LAUNCH(false, false);
  }
  note_launch();
#undef SP_LAUNCH
  return g;
}

// out[c] = sum of the partials of column c: one CTA per 4 columns.  1216
// partials of 64 columns: 100 us with a thread per column.
constexpr int kRpC = 4, kRpR = 64;
__global__ void __launch_bounds__(kRpC *kRpR) k_reduce_parts(const double *__restrict__ parts, int nparts, int m,
                                                             double *out) {
  __shared__ double sm[kRpC * kRpR];
  const int c = blockIdx.x * kRpC + threadIdx.x % kRpC;
  const double s = column_sum<kRpC, kRpR>(parts, nparts, m, c, c < m, sm);
  if (c < m && threadIdx.x < kRpC) out[c] = s;
}
void launch_reduce_parts(const double *parts, int nparts, int m, double *out, cudaStream_t s) {
  k_reduce_parts<<<ceil_div(m, kRpC), kRpC * kRpR, 0, s>>>(parts, nparts, m, out);
  note_launch();
}

// ---------------------------------------------------------------------------
// deterministic CSR transpose
// ---------------------------------------------------------------------------
__global__ void k_count_cols(CsrView A, int32_t *cnt) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += gridDim.x * blockDim.x)
    for (int64_t k = A.rowptr[i]; k < A.rowptr[i + 1]; ++k) atomicAdd(&cnt[A.colind[k]], 1);
}
// exclusive scan of cnt[0..n) into out[0..n], single CTA
__global__ void k_scan(const int32_t *cnt, int n, int32_t *out) {
  __shared__ int32_t part[1024];
  const int t = threadIdx.x, nt = blockDim.x;
  const int chunk = ceil_div(n, nt);
  const int b = t * chunk, e = min(n, b + chunk);
  int32_t s = 0;
  for (int i = b; i < e; ++i) s += cnt[i];
  part[t] = s;
  __syncthreads();
  if (t == 0) {
    int32_t run = 0;
    for (int i = 0; i < nt; ++i) {
      int32_t v = part[i];
      part[i] = run;
      run += v;
    }
    out[n] = run;
  }
  __syncthreads();
  int32_t run = part[t];
  for (int i = b; i < e; ++i) {
    out[i] = run;
    run += cnt[i];
  }
}
__global__ void k_fill_t(CsrView A, const int32_t *rowptr_t, int32_t *cursor, int32_t *colind_t, double *val_t) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += gridDim.x * blockDim.x)
    for (int64_t k = A.rowptr[i]; k < A.rowptr[i + 1]; ++k) {
      int c = A.colind[k];
      int pos = rowptr_t[c] + atomicAdd(&cursor[c], 1);
      colind_t[pos] = i;
      if (A.cplx) {
        val_t[2 * (size_t)pos] = A.val[2 * k];
        val_t[2 * (size_t)pos + 1] = A.val[2 * k + 1];
      } else {
        val_t[pos] = A.val[k];
      }
    }
}
__global__ void k_sort_rows(int n, const int32_t *rowptr, int32_t *colind, double *val, int cplx) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    const int b = rowptr[r], e = rowptr[r + 1];
    for (int i = b + 1; i < e; ++i) {
      int key = colind[i];
      double v0 = cplx ? val[2 * (size_t)i] : val[i];
      double v1 = cplx ? val[2 * (size_t)i + 1] : 0.0;
      int j = i - 1;
      while (j >= b && colind[j] > key) {
        colind[j + 1] = colind[j];
        if (cplx) {
          val[2 * (size_t)(j + 1)] = val[2 * (size_t)j];
          val[2 * (size_t)(j + 1) + 1] = val[2 * (size_t)j + 1];
        } else {
          val[j + 1] = val[j];
        }
        --j;
      }
      colind[j + 1] = key;
      if (cplx) {
        val[2 * (size_t)(j + 1)] = v0;
        val[2 * (size_t)(j + 1) + 1] = v1;
      } else {
        val[j + 1] = v0;
      }
    }
  }
}

cudaError_t csr_transpose(const CsrView &A, int32_t *rowptr_t, int32_t *colind_t, double *val_t, int32_t *work,
                          cudaStream_t s) {
  const int n = A.n;
  const int grid = min(4096, ceil_div(n, 256));
  cudaMemsetAsync(work, 0, (size_t)n * sizeof(int32_t), s);
  k_count_cols<<<grid, 256, 0, s>>>(A, work);
  note_launch();
  k_scan<<<1, 1024, 0, s>>>(work, n, rowptr_t);
  note_launch();
  cudaMemsetAsync(work, 0, (size_t)n * sizeof(int32_t), s);
  k_fill_t<<<grid, 256, 0, s>>>(A, rowptr_t, work, colind_t, val_t);
  note_launch();
  k_sort_rows<<<grid, 256, 0, s>>>(n, rowptr_t, colind_t, val_t, A.cplx);
  note_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP32 multi-shift operator of the Krylov sweeps: V_j = (z_j B - A) P_j for
// every node j and column c (left side: the conjugate-transpose CSR with
// conj(z_j)).  P, V: node-major ne blocks of n x m complex float, row-major.
// Bound by the gathers of P's rows out of L2.  G lanes a row, two columns a
// lane (one 16-byte load per gathered row where m is even), so that narrow
// blocks fill their warps with several rows.  A lane loads and converts one
// entry of the row, which the group's lanes then read by shuffles: converting
// in every lane took the FP64 pipe 64 cycles a warp and entry.
// The rows are walked for ng nodes at a time, as many as keep what the rows in
// flight reach (their number plus the band's width) within kGatherBytes, a
// third of L2.  Rows of up to U entries keep them in registers for all nodes.
// 8 nodes of 50021 rows, 9 random entries each, 48 columns of P (154 MB):
// 203 us with all nodes at once and a warp a row, 185 without the registers,
// 141 us (the gathers are 1.5 GB, 11 TB/s out of L2); its transpose, with rows
// of up to 25 entries, 352 -> 248 us; 200000 rows, 16 columns 654 -> 330; on the
// 300 x 300 grid, 16 columns 124 -> 50, 63 columns 281 -> 175.
// ---------------------------------------------------------------------------
// Two columns a lane: neighbours (PAIR, rows start on 16 bytes), or G apart
// where m is odd.
template <bool PAIR, int G> __device__ __forceinline__ float4 load2(const cxf *p, bool second) {
  if constexpr (PAIR) return *reinterpret_cast<const float4 *>(p);
  const float2 a = *reinterpret_cast<const float2 *>(p);
  float2 b = make_float2(0.f, 0.f);
  if (second) b = *reinterpret_cast<const float2 *>(p + G);
  return make_float4(a.x, a.y, b.x, b.y);
}
template <bool PAIR, int G> __device__ __forceinline__ void store2(cxf *p, float4 v, bool second) {
  if constexpr (PAIR) {
    *reinterpret_cast<float4 *>(p) = v;
  } else {
    *reinterpret_cast<float2 *>(p) = make_float2(v.x, v.y);
    if (second) *reinterpret_cast<float2 *>(p + G) = make_float2(v.z, v.w);
  }
}

// acc += a * x (two complex lanes)
template <bool CPLX> __device__ __forceinline__ void vfma(float4 &acc, cxf a, const float4 &x) {
  acc.x = fmaf(a.re, x.x, acc.x);
  acc.y = fmaf(a.re, x.y, acc.y);
  acc.z = fmaf(a.re, x.z, acc.z);
  acc.w = fmaf(a.re, x.w, acc.w);
  if constexpr (CPLX) {
    acc.x = fmaf(-a.im, x.y, acc.x);
    acc.y = fmaf(a.im, x.x, acc.y);
    acc.z = fmaf(-a.im, x.w, acc.z);
    acc.w = fmaf(a.im, x.z, acc.w);
  }
}

// A row's entries in the lanes of its group, G at a time
template <bool CPLX, int G> struct RowPart {
  int col;
  cxf val;
  __device__ __forceinline__ void load(const CsrView &M, int64_t beg, int cnt, int base, float sign) {
    const int k = base + (threadIdx.x & (G - 1));
    col = 0;
    val = mk(0.f, 0.f);
    if (k < cnt) {
      col = M.colind[beg + k];
      if constexpr (CPLX) {
        const cxd v = reinterpret_cast<const cxd *>(M.val)[beg + k];
        val = mk(sign * (float)v.re, (M.conj_vals ? -sign : sign) * (float)v.im);
      } else {
        val = mk(sign * (float)M.val[beg + k], 0.f);
      }
    }
  }
  // acc += the product of entries base .. of a row of cnt (most: of the warp's
  // rows), the gathers of U entries issued together
  template <int U, bool PAIR>
  __device__ __forceinline__ void apply(float4 &acc, int base, int cnt, int most, const cxf *Pc, int m,
                                        bool ok, bool second) const {
    const int nb = min(G, most - base), left = ok ? min(G, cnt - base) : 0;
    for (int k = 0; k < nb; k += U) {
      float4 x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int cu = __shfl_sync(0xffffffffu, col, k + u, G);
        x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k + u < left) x[u] = load2<PAIR, G>(Pc + (size_t)cu * m, second);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        cxf v;
        v.re = __shfl_sync(0xffffffffu, val.re, k + u, G);
        v.im = CPLX ? __shfl_sync(0xffffffffu, val.im, k + u, G) : 0.f;
        if (k + u < left) vfma<CPLX>(acc, v, x[u]);
      }
    }
  }
};

constexpr int kSpThreads = 256;
template <bool ACPLX, bool BCPLX, bool HASB, bool PAIR, int G, int U>
__global__ void __launch_bounds__(kSpThreads, U == 5 ? 4 : PAIR ? 3 : 2)
    k_multishift_spmm_f32(CsrView A, CsrView B, int ne, const cxd *__restrict__ z, int conj_z,
                          const cxf *__restrict__ P, cxf *__restrict__ V, int n, int m, int ng) {
  __shared__ cxf zs[kMaxNe];
  if (threadIdx.x < ne) {
    const cxd zz = z[threadIdx.x];
    zs[threadIdx.x] = mk((float)zz.re, conj_z ? -(float)zz.im : (float)zz.im);
  }
  __syncthreads();
  constexpr int RPW = 32 / G, kShort = U < G ? U : G;
  const int lane = threadIdx.x & 31, gl = lane & (G - 1);
  const int warp = (int)(((long long)blockIdx.x * kSpThreads + threadIdx.x) >> 5);
  const int nwarps = (int)(((long long)gridDim.x * kSpThreads) >> 5);
  const size_t xns = (size_t)n * m;
  for (int j0 = 0; j0 < ne; j0 += ng) {
    const int j1 = min(ne, j0 + ng);
    for (int ib = warp * RPW; ib < n; ib += nwarps * RPW) {
      const int i = ib + lane / G;
      const bool row = i < n;
      const int64_t ka = row ? A.rowptr[i] : 0, kb = HASB && row ? B.rowptr[i] : 0;
      const int na = row ? (int)(A.rowptr[i + 1] - ka) : 0, nb = HASB && row ? (int)(B.rowptr[i + 1] - kb) : 0;
      const int ma = G == 32 ? na : __reduce_max_sync(0xffffffffu, na);
      const int mb = !HASB || G == 32 ? nb : __reduce_max_sync(0xffffffffu, nb);
      RowPart<ACPLX, G> ra;  // -A
      RowPart<BCPLX, G> rb;
      ra.load(A, ka, na, 0, -1.f);
      if (HASB) rb.load(B, kb, nb, 0, 1.f);
      for (int c0 = 0; c0 < m; c0 += 2 * G) {
        const int c = c0 + (PAIR ? 2 * gl : gl);
        const bool ok = row && c < m, second = !PAIR && c + G < m;
        if (!HASB && ma <= kShort) {
          // short rows, the usual case: their entries in registers for all nodes
          int col[kShort];
          cxf v[kShort];
#pragma unroll
          for (int u = 0; u < kShort; ++u) {
            col[u] = __shfl_sync(0xffffffffu, ra.col, u, G);
            if (u >= na) col[u] = i;  // value zero
            v[u].re = __shfl_sync(0xffffffffu, ra.val.re, u, G);
            v[u].im = ACPLX ? __shfl_sync(0xffffffffu, ra.val.im, u, G) : 0.f;
          }
          if (!ok) continue;
#pragma unroll 2
          for (int j = j0; j < j1; ++j) {
            const cxf *Pc = P + (size_t)j * xns + c;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), x[kShort];
#pragma unroll
            for (int u = 0; u < kShort; ++u) x[u] = load2<PAIR, G>(Pc + (size_t)col[u] * m, second);
            const float4 own = load2<PAIR, G>(Pc + (size_t)i * m, second);
#pragma unroll
            for (int u = 0; u < kShort; ++u) vfma<ACPLX>(acc, v[u], x[u]);
            vfma<true>(acc, zs[j], own);
            store2<PAIR, G>(V + (size_t)j * xns + (size_t)i * m + c, acc, second);
          }
          continue;
        }
        for (int j = j0; j < j1; ++j) {
          const cxf *Pc = P + (size_t)j * xns + c;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f), bx = acc;
          if (HASB) {
            rb.template apply<U, PAIR>(bx, 0, nb, mb, Pc, m, ok, second);
            for (int base = G; base < mb; base += G) {
              RowPart<BCPLX, G> more;
              more.load(B, kb, nb, base, 1.f);
              more.template apply<U, PAIR>(bx, base, nb, mb, Pc, m, ok, second);
            }
          } else if (ok) {
            bx = load2<PAIR, G>(Pc + (size_t)i * m, second);
          }
          ra.template apply<U, PAIR>(acc, 0, na, ma, Pc, m, ok, second);
          for (int base = G; base < ma; base += G) {
            RowPart<ACPLX, G> more;
            more.load(A, ka, na, base, -1.f);
            more.template apply<U, PAIR>(acc, base, na, ma, Pc, m, ok, second);
          }
          vfma<true>(acc, zs[j], bx);
          if (ok) store2<PAIR, G>(V + (size_t)j * xns + (size_t)i * m + c, acc, second);
        }
      }
    }
  }
}


// VW columns of a lane: neighbours (VW = 2, rows start on 16 bytes) or one.
template <int VW> __device__ __forceinline__ float4 loadw(const cxf *p) {
  if constexpr (VW == 2) return *reinterpret_cast<const float4 *>(p);
  const float2 a = *reinterpret_cast<const float2 *>(p);
  return make_float4(a.x, a.y, 0.f, 0.f);
}
template <int VW> __device__ __forceinline__ void storew(cxf *p, float4 v) {
  if constexpr (VW == 2)
    *reinterpret_cast<float4 *>(p) = v;
  else
    *reinterpret_cast<float2 *>(p) = make_float2(v.x, v.y);
}

// More than 32 columns, no B, rows of up to K entries (longer ones take a
// loop): a warp a row, whose entries every lane reads and keeps itself, for ng
// nodes at a time.  Bound by the gathers out of L2, K + 1 in flight
// a lane; the group kernel above spends as many issue slots on its shuffles,
// and past nine entries it has no row in registers.  What each K measured
// against it stands with the rule below.  Real rows of five (all nodes at once)
// take complex products and the column in each row's address, which the compiler
// schedules better there: 300 x 300 grid, 64 columns, 16 nodes 298 us, 302 in the
// other form; complex ones 253 and 234.
template <bool ACPLX, int VW, int K>
__global__ void __launch_bounds__(kSpThreads) k_multishift_spmm_f32_wide(CsrView A, int ne, const cxd *__restrict__ z,
                                                                         int conj_z, const cxf *__restrict__ P,
                                                                         cxf *__restrict__ V, int n, int m, int ng) {
  __shared__ cxf zs[kMaxNe];
  if (threadIdx.x < ne) {
    const cxd zz = z[threadIdx.x];
    zs[threadIdx.x] = mk((float)zz.re, conj_z ? -(float)zz.im : (float)zz.im);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int warp = (int)(((long long)blockIdx.x * kSpThreads + threadIdx.x) >> 5);
  const int nwarps = (int)(((long long)gridDim.x * kSpThreads) >> 5);
  const size_t xns = (size_t)n * m;
  auto entry = [&](int64_t k) {  // of -A
    if constexpr (ACPLX) {
      const cxd v = reinterpret_cast<const cxd *>(A.val)[k];
      return mk(-(float)v.re, A.conj_vals ? (float)v.im : -(float)v.im);
    }
    return mk(-(float)A.val[k], 0.f);
  };
  constexpr bool FIVE = K == 5 && !ACPLX;
  for (int j0 = 0; j0 < ne; j0 += FIVE ? ne : ng) {
    const int j1 = FIVE ? ne : min(ne, j0 + ng);
    for (int i = warp; i < n; i += nwarps) {
      const int64_t ka = A.rowptr[i];
      const int nk = (int)(A.rowptr[i + 1] - ka);
      int col[K];
      cxf av[K];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        col[k] = k < nk ? A.colind[ka + k] : i;
        av[k] = k < nk ? entry(ka + k) : mk(0.f, 0.f);
      }
      const bool fast = nk <= K;
      for (int c = lane * VW; c < m; c += 32 * VW) {
#pragma unroll 2
        for (int j = j0; j < j1; ++j) {
          const cxf *Pj = P + (size_t)j * xns + (FIVE ? 0 : c);
          const int cj = FIVE ? c : 0;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
          if (fast) {
            float4 xs[K];
#pragma unroll
            for (int k = 0; k < K; ++k) xs[k] = loadw<VW>(Pj + (size_t)col[k] * m + cj);
            vfma<true>(acc, zs[j], loadw<VW>(Pj + (size_t)i * m + cj));
#pragma unroll
            for (int k = 0; k < K; ++k) vfma<ACPLX || FIVE>(acc, av[k], xs[k]);
          } else {
            vfma<true>(acc, zs[j], loadw<VW>(Pj + (size_t)i * m + cj));
            for (int k = 0; k < nk; ++k)
              vfma<ACPLX || FIVE>(acc, entry(ka + k), loadw<VW>(Pj + (size_t)A.colind[ka + k] * m + cj));
          }
          storew<VW>(V + (size_t)j * xns + (size_t)i * m + c, acc);
        }
      }
    }
  }
}

// Longest row of A and of A^H.
__global__ void k_longest_rows(CsrView A, CsrView AH, int *out) {
  int mx[2] = {0, 0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += gridDim.x * blockDim.x) {
    mx[0] = max(mx[0], (int)(A.rowptr[i + 1] - A.rowptr[i]));
    mx[1] = max(mx[1], (int)(AH.rowptr[i + 1] - AH.rowptr[i]));
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int v = __reduce_max_sync(0xffffffffu, mx[q]);
    if ((threadIdx.x & 31) == 0) atomicMax(out + q, v);
  }
}
void launch_longest_rows(const CsrView &A, const CsrView &AH, int *d_out, cudaStream_t s) {
  cudaMemsetAsync(d_out, 0, 2 * sizeof(int), s);
  k_longest_rows<<<std::min(1024, ceil_div(A.n, 256)), 256, 0, s>>>(A, AH, d_out);
  note_launch();
}

constexpr size_t kGatherBytes = 48u << 20;

template <bool PAIR, int G>
static void spmm_f32_launch(const CsrView &A, const CsrView *B, int bw, int longest, int ne, const cxd *d_z, int conj_z,
                            const cxf *P, cxf *V, int m, cudaStream_t s) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const CsrView Bv = B ? *B : A;
  const int rows = kSpThreads / G;  // of a CTA
  const int need = std::max(1, ceil_div(A.n, rows));
  const size_t window = std::min<size_t>(A.n, (size_t)bw + (size_t)4 * sms * rows) * m * sizeof(cxf);
  const int ng = (int)std::min<size_t>(ne, std::max<size_t>(1, kGatherBytes / window));
  const bool few = A.nnz <= 5 * (int64_t)A.n;
  if constexpr (G == 32) {
    // A warp a row against the group kernel, us, 8 nodes, 64000 rows of a stencil
    // (50000 random ones), 48 columns, 33 where the number is odd.  Rows of five:
    // 109 and 119, odd 115 and 109, so even numbers only.  Seven: 134 and 154 (132
    // and 144), odd 132 and 167; complex odd the same, and beyond 48 columns slower
    // (212 and 183).  Nine: 177 and 158, odd 173 and 171: never.  Thirteen: 232 and
    // 314 (271 and 279), odd 249 and 390 (253 and 335).  Where nodes go in turns the
    // row is read again in every turn, which pays from 96 columns a turn, or two
    // passes over the row's columns (random rows of 13, a node a turn: 64 columns
    // 804 and 656, 96 columns 513 and 591).
    const bool turns = ng < ne && ng * m < 96 && m <= 64;
    int K = 0;
    if (!B && few && PAIR && ng == ne) K = 5;
    else if (!B && !few && !turns && longest <= 7 && (PAIR || !A.cplx)) K = 7;
    else if (!B && !turns && longest > 9 && longest <= 16 && A.nnz > 9 * (int64_t)A.n) K = 16;
    if (K) {
      constexpr int VW = PAIR ? 2 : 1;
      auto launch = [&](auto kern) {
        int occ = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kSpThreads, 0);
        kern<<<std::min(occ * sms, need), kSpThreads, 0, s>>>(A, ne, d_z, conj_z, P, V, A.n, m, ng);
      };
      auto pick = [&](auto cplx) {
        constexpr bool AC = decltype(cplx)::value;
        if constexpr (PAIR)
          if (K == 5) return launch(k_multishift_spmm_f32_wide<AC, VW, 5>);
        if constexpr (PAIR || !AC)
          if (K == 7) return launch(k_multishift_spmm_f32_wide<AC, VW, 7>);
        launch(k_multishift_spmm_f32_wide<AC, VW, 16>);
      };
      if (A.cplx)
        pick(std::true_type{});
      else
        pick(std::false_type{});
      note_launch();
      return;
    }
  }
#define SPF(AC, BC, HB, U)                                                                              \
  do {                                                                                                  \
    auto kern = k_multishift_spmm_f32<AC, BC, HB, PAIR, G, U>;                                          \
    int occ = 1;                                                                                        \
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kSpThreads, 0);                           \
    kern<<<std::min(occ * sms, need), kSpThreads, 0, s>>>(A, Bv, ne, d_z, conj_z, P, V, A.n, m, ng);    \
  } while (0)
  if (!B) {
    if (A.cplx) {
      if (few) SPF(true, false, false, 5); else SPF(true, false, false, 9);
    } else {
      if (few) SPF(false, false, false, 5); else SPF(false, false, false, 9);
    }
  } else if (B->cplx) {
    if (A.cplx) SPF(true, true, true, 5); else SPF(false, true, true, 5);
  } else {
    if (A.cplx) SPF(true, false, true, 5); else SPF(false, false, true, 5);
  }
#undef SPF
  note_launch();
}

void launch_multishift_spmm_f32(const CsrView &A, const CsrView *B, int bw, int longest, int ne, const cxd *d_z,
                                int conj_z, const cxf *P, cxf *V, int m, cudaStream_t s) {
  // the fewest lanes a row that cover it in one pass; where long rows are too few
  // to fill the chip, sixteen, which gather more of a row at once (us, 8 nodes,
  // 600 rows of 600: 1 column 668 -> 447, 8 columns 793 -> 404; 3000 rows of 100, 8
  // columns 152 -> 87; 6000 rows of 60 the other way, 103 -> 70 for 70 -> 111)
  const bool few_long = A.nnz > 16 * (int64_t)A.n && A.n <= 3648;
  const int cols = few_long ? std::max(9, ceil_div(m, 2)) : ceil_div(m, 2);
#define SPG(PAIR)                                                                                     \
  do {                                                                                                \
    if (cols <= 4) return spmm_f32_launch<PAIR, 4>(A, B, bw, longest, ne, d_z, conj_z, P, V, m, s);   \
    if (cols <= 8) return spmm_f32_launch<PAIR, 8>(A, B, bw, longest, ne, d_z, conj_z, P, V, m, s);   \
    if (cols <= 16) return spmm_f32_launch<PAIR, 16>(A, B, bw, longest, ne, d_z, conj_z, P, V, m, s); \
    return spmm_f32_launch<PAIR, 32>(A, B, bw, longest, ne, d_z, conj_z, P, V, m, s);                 \
  } while (0)
  if (m % 2 == 0) SPG(true);
  SPG(false);
#undef SPG
}
