// Tridiagonal shifted solves, (z B - A) x = r and its conjugate transpose, from
// the band factors L D U' (U' = D^{-1} U with unit diagonal), one warp a
// right-hand side with the rows in 32 chunks, a lane each.
//
// The recurrences y_r = b_r - a_r y_{r-1} and x_r = s_r - c_r x_{r+1} are run
// in every chunk at once from zero; the values entering the chunks follow from
// a scan over the lanes of the chunks' affine maps, and are then carried into
// the rows with the products P_r of the coefficients (formed with the factors).
// Twenty FP64 FMAs a row and column in three passes, n / 32 steps each, instead
// of a chain of 2 n steps: 1000 rows, 40 columns, 8 nodes, both sides in FP64,
// 2940 us with the general band solver, 67 us.  Bound by the FP64 pipe (a warp
// instruction takes it 64 cycles): with 640 columns, about one warp for each
// of the chip's 608 sub-partitions.  Taken for every pencil with kl, ku <= 1.
#include "kernels.h"

namespace {
constexpr int kWarps = 4;  // columns of a CTA

template <typename T> __device__ __forceinline__ cx<T> cj_if(cx<T> v, bool c) {
  if (c) v.im = -v.im;
  return v;
}
// (g, t) <- (g, t) o (g1, t1): v -> t + g (t1 + g1 v)
template <typename T> __device__ __forceinline__ void compose(cx<T> &g, cx<T> &t, cx<T> g1, cx<T> t1) {
  cfma(t, g, t1);
  g = g * g1;
}
template <typename T> __device__ __forceinline__ cx<T> shfl_up(cx<T> v, int d) {
  return mk<T>(__shfl_up_sync(0xffffffffu, v.re, d), __shfl_up_sync(0xffffffffu, v.im, d));
}
template <typename T> __device__ __forceinline__ cx<T> shfl_down(cx<T> v, int d) {
  return mk<T>(__shfl_down_sync(0xffffffffu, v.re, d), __shfl_down_sync(0xffffffffu, v.im, d));
}
}  // namespace

// Coefficient arrays of a slot and side, element [k * 32 + lane] for row
// lane * len + k: a, P (forward), d (1 / pivot), c, Pb (backward).
enum { kA = 0, kP = 1, kD = 2, kC = 3, kPb = 4, kArrays = 5 };
size_t tri_elems(int n, int nf) { return (size_t)nf * 2 * kArrays * 32 * ceil_div(n, 32); }

template <typename T>
__global__ void __launch_bounds__(32) k_tri_setup(int n, int kl, int ku, const cx<T> *__restrict__ band, cx<T> *__restrict__ co) {
  const int slot = blockIdx.x, side = blockIdx.y, lane = threadIdx.x, len = ceil_div(n, 32), W = kl + ku + 1;
  const cx<T> *Bd = band + (size_t)slot * n * W;
  cx<T> *o = co + ((size_t)slot * 2 + side) * kArrays * 32 * len;
  const size_t st = (size_t)32 * len;
  auto pivot = [&](int r) { return Bd[(size_t)r * W + kl]; };
  auto low = [&](int r) { return kl > 0 && r >= 1 && r < n ? Bd[(size_t)r * W + kl - 1] : mk<T>(0, 0); };  // L(r, r-1)
  auto up = [&](int r) { return ku > 0 && r >= 0 && r + 1 < n ? Bd[(size_t)r * W + kl + 1] : mk<T>(0, 0); };  // U(r, r+1)
  cx<T> P = mk<T>(1, 0);
  for (int k = 0; k < len; ++k) {
    const int r = lane * len + k;
    cx<T> a = mk<T>(0, 0), d = mk<T>(0, 0), c = mk<T>(0, 0);
    if (r < n) {
      d = cdiv(mk<T>(1, 0), pivot(r));
      if (side == 0) {
        a = low(r);
        c = up(r) * d;
      } else {
        a = r >= 1 ? conj(cdiv(up(r - 1), pivot(r - 1))) : mk<T>(0, 0);
        c = conj(low(r + 1));
        d = conj(d);
      }
    }
    P = -(a * P);
    o[kA * st + k * 32 + lane] = a;
    o[kP * st + k * 32 + lane] = P;
    o[kD * st + k * 32 + lane] = d;
    o[kC * st + k * 32 + lane] = c;
  }
  P = mk<T>(1, 0);
  for (int k = len - 1; k >= 0; --k) {
    P = -(o[kC * st + k * 32 + lane] * P);
    o[kPb * st + k * 32 + lane] = P;
  }
}

template <typename T>
__global__ void __launch_bounds__(32 * kWarps) k_tri_solve(int n, const cx<T> *__restrict__ co, SolveMap map,
                                                           const cx<T> *rhs0, const cx<T> *rhs1, cxd *X0, cxd *X1,
                                                           size_t rns, int m, size_t xns, int mode, cx<T> *__restrict__ ys) {
  const int side = blockIdx.z, node = blockIdx.y, lane = threadIdx.x & 31;
  const int c = blockIdx.x * kWarps + (threadIdx.x >> 5);
  if (c >= m) return;
  const int len = ceil_div(n, 32), slot = map.f[node] & 0xffff;
  const bool cj = (map.f[node] >> 16) & 1;
  const size_t st = (size_t)32 * len;
  const cx<T> *o = co + ((size_t)slot * 2 + side) * kArrays * st + lane;
  const cx<T> *b = (side ? rhs1 : rhs0) + (size_t)node * rns + c;
  cxd *X = (side ? X1 : X0) + (size_t)node * xns + c;
  cx<T> *v = ys + (((size_t)side * gridDim.y + node) * m + c) * st + lane;
  const int r0 = lane * len, cnt = max(0, min(len, n - r0));
  // forward, every chunk from zero
  cx<T> y = mk<T>(0, 0);
#pragma unroll 4
  for (int k = 0; k < cnt; ++k) {
    cx<T> t = b[(size_t)(r0 + k) * m];
    cfms(t, cj_if(o[kA * st + k * 32], cj), y);
    y = t;
    v[k * 32] = y;
  }
  // the value entering each chunk: scan of y_out = y + g y_in
  cx<T> g = cnt > 0 ? cj_if(o[kP * st + (cnt - 1) * 32], cj) : mk<T>(1, 0);
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const cx<T> g1 = shfl_up(g, d), t1 = shfl_up(y, d);
    if (lane >= d) compose(g, y, g1, t1);
  }
  cx<T> in = shfl_up(y, 1);
  if (lane == 0) in = mk<T>(0, 0);
  // backward, every chunk from zero, on the corrected and scaled values
  cx<T> x = mk<T>(0, 0);
#pragma unroll 4
  for (int k = cnt - 1; k >= 0; --k) {
    cx<T> t = v[k * 32];
    cfma(t, cj_if(o[kP * st + k * 32], cj), in);
    t = cj_if(o[kD * st + k * 32], cj) * t;
    cfms(t, cj_if(o[kC * st + k * 32], cj), x);
    x = t;
    v[k * 32] = x;
  }
  g = cnt > 0 ? cj_if(o[kPb * st], cj) : mk<T>(1, 0);
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const cx<T> g1 = shfl_down(g, d), t1 = shfl_down(x, d);
    if (lane + d < 32) compose(g, x, g1, t1);
  }
  in = shfl_down(x, 1);
  if (lane == 31) in = mk<T>(0, 0);
#pragma unroll 4
  for (int k = 0; k < cnt; ++k) {
    cx<T> t = v[k * 32];
    cfma(t, cj_if(o[kPb * st + k * 32], cj), in);
    cxd *xp = X + (size_t)(r0 + k) * m;
    const cxd td = ccast<double>(t);
    *xp = mode ? (*xp + td) : td;
  }
}

template <typename T>
void launch_tri_setup(int n, int klp, int kup, int nf, const cx<T> *band, cx<T> *co, cudaStream_t s) {
  k_tri_setup<T><<<dim3(nf, 2), 32, 0, s>>>(n, klp, kup, band, co);
  note_launch();
}
template void launch_tri_setup<float>(int, int, int, int, const cxf *, cxf *, cudaStream_t);
template void launch_tri_setup<double>(int, int, int, int, const cxd *, cxd *, cudaStream_t);

size_t tri_scratch_elems(int n, int m, int ne) { return (size_t)2 * ne * m * 32 * ceil_div(n, 32); }

template <typename T>
cudaError_t tri_solve_sides(int n, int ne, const int *fmap, const cx<T> *co, const cx<T> *rhsR, const cx<T> *rhsL,
                            size_t rns, int m, cxd *XR, cxd *XL, size_t xns, int mode, cx<T> *ys, cudaStream_t s) {
  SolveMap map;
  for (int j = 0; j < kMaxNe; ++j) map.f[j] = j < ne ? fmap[j] : 0;
  const int nsides = (rhsL && XL) ? 2 : 1;
  k_tri_solve<T><<<dim3(ceil_div(m, kWarps), ne, nsides), 32 * kWarps, 0, s>>>(
      n, co, map, rhsR, rhsL ? rhsL : rhsR, XR, XL ? XL : XR, rns, m, xns, mode, ys);
  note_launch();
  return cudaGetLastError();
}
template cudaError_t tri_solve_sides<float>(int, int, const int *, const cxf *, const cxf *, const cxf *, size_t, int,
                                            cxd *, cxd *, size_t, int, cxf *, cudaStream_t);
template cudaError_t tri_solve_sides<double>(int, int, const int *, const cxd *, const cxd *, const cxd *, size_t, int,
                                             cxd *, cxd *, size_t, int, cxd *, cudaStream_t);
