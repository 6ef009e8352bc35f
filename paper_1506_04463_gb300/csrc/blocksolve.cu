// Shifted solves by block substitution with inverted diagonal blocks.
//
// A band of half-width bw cut into blocks of b >= bw rows is block tridiagonal,
// M = z B - A.  With S_i = L_ii U_ii the diagonal blocks of its LU factors
// (the Schur complements of block elimination) and T_i = S_i^{-1}, a system
// M x = r is
//     z_i = T_i (r_i - M_{i,i-1} z_{i-1}),      i = 1, 2, ...
//     x_i = z_i - T_i (M_{i,i+1} x_{i+1}),      i = ..., 2, 1,
// and M^H x = r the same with T_i^H and the blocks of M^H.  The off-diagonal
// blocks are those of the matrix itself, a few entries a row, so a solve is
// 2 n / b dependent steps of one b x b product instead of 2 n / 16 steps of a
// 16-row window product and a small triangular solve (band.cu), which are bound
// by the latency of their serial part.  One sweep, both sides: FP32, n = 10000,
// band 100, 16 nodes, 40 columns 2.9 -> 2.1 ms; n = 4096, band 256, 8 nodes,
// 20 columns 1.6 -> 0.43 ms; FP64, n = 1600, band 40, 16 nodes, 48 columns
// 5.3 -> 2.2 ms.
//
// The explicit inverses cost some accuracy: the FP64 refinement contracts by
// two to four times less a step than with the triangular factors, and needs one
// step more now and then.  If it does not contract, the caller goes back to the
// triangular solves, which remain for that, for wider bands and for matrices
// with many entries a row.
#include <algorithm>
#include "kernels.h"
#include "mbar.cuh"

namespace {

constexpr int kGroup = 256;       // threads that cover a product's rows and columns
constexpr int kCons = 512;        // consumer threads: two such groups, on alternate stages
constexpr int kGroups = 4;        // column groups; a CTA takes kGroups * C columns
constexpr long long kSpin = 1ll << 22;
constexpr int kMaxStages = 6;
// columns of T per stage
template <typename T> struct Chunk { static constexpr int KC = 8; };

// asynchronous copy of one value to shared memory (zeros when !ok)
__device__ __forceinline__ void cp_async(cxf *dst, const cxf *src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 8 : 0));
}
__device__ __forceinline__ void cp_async(cxd *dst, const cxd *src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 16 : 0));
}
__device__ __forceinline__ void cp_async(int *dst, const int *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ void cons_bar() { asm volatile("bar.sync 1, 512;\n" ::: "memory"); }

// C consecutive complex values as wide loads (aligned to C values)
template <int C> __device__ __forceinline__ void load_row(cxf (&v)[C], const cxf *p) {
  if constexpr (C == 1) {
    v[0] = *p;
  } else {
#pragma unroll
    for (int c = 0; c < C; c += 2) {
      const float4 w = *reinterpret_cast<const float4 *>(p + c);
      v[c] = mk(w.x, w.y);
      v[c + 1] = mk(w.z, w.w);
    }
  }
}
template <int C> __device__ __forceinline__ void load_row(cxd (&v)[C], const cxd *p) {
#pragma unroll
  for (int c = 0; c < C; ++c) v[c] = p[c];
}

// Product of a b x b tile with b x C columns, U row groups a thread.
// FP64: rows rg + RG u, complex entries T[k][r].
template <typename T, int C, int U> struct Product {
  cxd acc[U][C];
  static constexpr int kRowsPer = 1;
  using Rhs = cxd;  // stored entry of the right-hand side
  static __device__ __forceinline__ Rhs rhs(cxd v) { return v; }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < C; ++c) acc[u][c] = mk(0.0, 0.0);
  }
  // one stage: kc columns of T (stage) times rows of t (row stride R)
  __device__ __forceinline__ void stage(const cxd *Ts, const Rhs *ts, int b, int R, int rg, int RG) {
#pragma unroll 4
    for (int k = 0; k < Chunk<T>::KC; ++k) {
      cxd tv[C];
      load_row(tv, ts + k * R);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const cxd a = Ts[(size_t)k * b + rg + RG * u];
#pragma unroll
        for (int c = 0; c < C; ++c) cfma(acc[u][c], a, tv[c]);
      }
    }
  }
  template <typename F> __device__ __forceinline__ void each(int rg, int RG, F f) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < C; ++c) f(rg + RG * u, c, acc[u][c]);
  }
};
// FP32: pairs of rows 2 (rg + RG u), + 1 as packed operands (a stage's column
// holds b real parts, then b imaginary parts): fma.rn.f32x2 runs at 124 FMAs a
// clock and SM where the scalar form reached 104, with half the instructions.
// The right-hand side is stored with both parts doubled, so that no register
// moves (which run on the FMA pipe) are needed: half as many as FMAs before.
struct __align__(16) Dup {
  unsigned long long re, im;
};
__device__ __forceinline__ void ffma2(unsigned long long &d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long dup(float x) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
  return d;
}
__device__ __forceinline__ float2 unpack(unsigned long long d) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(d));
  return v;
}
template <int C, int U> struct Product<float, C, U> {
  unsigned long long re[U][C], im[U][C];
  static constexpr int kRowsPer = 2;
  using Rhs = Dup;
  static __device__ __forceinline__ Rhs rhs(cxf v) { return Dup{dup(v.re), dup(v.im)}; }
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < C; ++c) re[u][c] = im[u][c] = 0ull;
  }
  __device__ __forceinline__ void stage(const cxf *Tst, const Rhs *ts, int b, int R, int rg, int RG) {
    const float *Ts = reinterpret_cast<const float *>(Tst) + 2 * rg;
#pragma unroll 4
    for (int k = 0; k < Chunk<float>::KC; ++k) {
      unsigned long long ar[U], ai[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float *p = Ts + (size_t)k * 2 * b + 2 * RG * u;
        ar[u] = *reinterpret_cast<const unsigned long long *>(p);
        ai[u] = *reinterpret_cast<const unsigned long long *>(p + b);
      }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(ts + k * R + c);
        const unsigned long long tn = t.y ^ 0x8000000080000000ull;  // -Im t (integer pipe)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          ffma2(re[u][c], ar[u], t.x);
          ffma2(im[u][c], ar[u], t.y);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          ffma2(re[u][c], ai[u], tn);
          ffma2(im[u][c], ai[u], t.x);
        }
      }
    }
  }
  template <typename F> __device__ __forceinline__ void each(int rg, int RG, F f) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const float2 x = unpack(re[u][c]), y = unpack(im[u][c]);
        const int r = 2 * (rg + RG * u);
        f(r, c, mk(x.x, y.x));
        f(r + 1, c, mk(x.y, y.y));
      }
  }
};

// entry (line, x) of a tile: lines are columns (Tc) or rows (Tr); FP32 keeps
// the real and imaginary parts of a line apart
__device__ __forceinline__ void put(cxd *t, int b, int line, int x, cxd v) { t[(size_t)line * b + x] = v; }
__device__ __forceinline__ void put(cxf *t, int b, int line, int x, cxf v) {
  float *f = reinterpret_cast<float *>(t) + (size_t)line * 2 * b;
  f[x] = v.re;
  f[b + x] = v.im;
}

}  // namespace

// ---------------------------------------------------------------------------
// off-diagonal entries: row r's entries of M = z B - A in the block before
// (dir 0) and after (dir 1) its own, K a row (local column; rows with fewer are
// filled up with zeros at column 0), values of A and of B apart since z differs
// by node
// ---------------------------------------------------------------------------
__global__ void k_block_count(CsrView A, CsrView B, int hasB, int b, int *kmax) {
  int mx = 0;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < A.n; r += gridDim.x * blockDim.x) {
    const int lo = (r / b) * b;
    int cnt[2] = {0, 0};
    for (int k = A.rowptr[r]; k < A.rowptr[r + 1]; ++k) {
      const int c = A.colind[k];
      if (c < lo) ++cnt[0];
      if (c >= lo + b) ++cnt[1];
    }
    if (hasB)
      for (int k = B.rowptr[r]; k < B.rowptr[r + 1]; ++k) {
        const int c = B.colind[k];
        if (c < lo) ++cnt[0];
        if (c >= lo + b) ++cnt[1];
      }
    mx = max(mx, max(cnt[0], cnt[1]));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) atomicMax(kmax, mx);
}
template <typename T>
__global__ void k_block_entries(CsrView A, CsrView B, int hasB, int b, int K, int nrows, int *idx, cx<T> *va, cx<T> *vb) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += gridDim.x * blockDim.x) {
    const int lo = (r / b) * b;
    for (int dir = 0; dir < 2; ++dir) {
      const size_t base = ((size_t)dir * nrows + r) * K;
      const int first = dir ? lo + b : lo - b;  // first row of the neighbouring block
      int q = 0;
      auto add = [&](const CsrView &M, bool isB) {
        for (int k = M.rowptr[r]; k < M.rowptr[r + 1]; ++k) {
          const int c = M.colind[k];
          if (dir ? c < lo + b : c >= lo) continue;
          idx[base + q] = c - first;
          const cx<T> v = ccast<T>(csr_val(M, k));
          va[base + q] = isB ? mk<T>(0, 0) : v;
          if (vb) vb[base + q] = isB ? v : mk<T>(0, 0);
          ++q;
        }
      };
      if (r < A.n) {
        add(A, false);
        if (hasB) add(B, true);
      }
      for (; q < K; ++q) {
        idx[base + q] = 0;
        va[base + q] = mk<T>(0, 0);
        if (vb) vb[base + q] = mk<T>(0, 0);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// T_i = U_ii^{-1} L_ii^{-1} from the band factors, 32 columns a CTA: forward
// and backward substitution on 16-row blocks, whose diagonal inverses are
// there already (k_band_diag_inv).  Y (b x 32) stays in shared memory; a
// 16-row strip of the factor is staged for each block; four rows a warp, the
// sum over k in two halves.  FP arithmetic of the factors' precision, 2/3 b^3
// complex FMAs a block (11 M at b = 256), all blocks of all factors independent.
// Output: column-major (Tc, for M) and row-major (Tr, for M^H) copies.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_block_inv(int n, int kl, int ku, int b, const cx<T> *__restrict__ band,
                                                   size_t ns, const cx<T> *__restrict__ dinv, cx<T> *__restrict__ Tc,
                                                   cx<T> *__restrict__ Tr) {  // grid (blocks, column strips, slots)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int LDY = 33;
  cx<T> *Y = reinterpret_cast<cx<T> *>(smem_raw);  // b x LDY
  cx<T> *F = Y + (size_t)b * LDY;                  // 16 x (b + 2) factor strip
  cx<T> *P = F + (size_t)16 * (b + 2);             // 2 x 16 x 32 partial sums
  cx<T> *D = P + 2 * 16 * 32;                      // 16 x 17
  const int ldf = b + 2;
  const int c0 = blockIdx.y * 32, blk = blockIdx.x, slot = blockIdx.z;
  const int W = kl + ku + 1, r0 = blk * b;
  const cx<T> *Bd = band + (size_t)slot * ns;
  const cx<T> *Dv = dinv + (size_t)slot * ceil_div(n, 16) * 1024;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nq = min(b, n - r0 + 15) / 16;  // 16-row blocks that hold rows of the matrix
  const int half = warp >> 2, rg = (warp & 3) * 4;
  for (int e = tid; e < b * 32; e += 256) {
    const int r = e >> 5, c = e & 31;
    Y[r * LDY + c] = mk<T>(r == c0 + c ? 1 : 0, 0);
  }
  __syncthreads();
  for (int phase = 0; phase < 2; ++phase) {
    for (int s = 0; s < nq; ++s) {
      const int q = phase ? nq - 1 - s : s;
      if (!phase && q * 16 + 16 <= c0) continue;  // rows above the unit entries stay zero
      const int klo = phase ? 16 * (q + 1) : c0, khi = phase ? 16 * nq : 16 * q;
      // factor strip: rows 16q.., columns [klo, khi) of the block
      for (int rr = warp; rr < 16; rr += 8) {
        const int r = r0 + 16 * q + rr;
        for (int k = klo + lane; k < khi; k += 32) {
          const int d = r0 + k - r;
          const bool in = r < n && r0 + k < n && (phase ? d <= ku : -d <= kl);
          F[rr * ldf + (k - klo)] = in ? Bd[(size_t)r * W + (d + kl)] : mk<T>(0, 0);
        }
      }
      for (int e = tid; e < 256; e += 256)
        D[(e >> 4) * 17 + (e & 15)] = Dv[((size_t)(r0 / 16) + q) * 1024 + (phase ? 512 : 0) + e];
      __syncthreads();
      const int len = khi - klo, kh = ((len + 1) / 2 + 1) & ~1;
      const int ka = half ? min(kh, len) : 0, kb = half ? len : min(kh, len);
      cx<T> acc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = mk<T>(0, 0);
#pragma unroll 4
      for (int k = ka; k < kb; ++k) {
        const cx<T> y = Y[(klo + k) * LDY + lane];
#pragma unroll
        for (int u = 0; u < 4; ++u) cfma(acc[u], F[(rg + u) * ldf + k], y);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) P[(half * 16 + rg + u) * 32 + lane] = acc[u];
      __syncthreads();
      for (int e = tid; e < 512; e += 256) {
        const int rr = e >> 5, c = e & 31;
        P[e] = Y[(16 * q + rr) * LDY + c] - (P[e] + P[512 + e]);
      }
      __syncthreads();
      for (int rr = warp; rr < 16; rr += 8) {
        cx<T> x = mk<T>(0, 0);
#pragma unroll
        for (int p = 0; p < 16; ++p) cfma(x, D[rr * 17 + p], P[p * 32 + lane]);
        Y[(16 * q + rr) * LDY + lane] = x;
      }
      __syncthreads();
    }
  }
  const size_t base = ((size_t)slot * gridDim.x + blk) * b * b;
  for (int e = tid; e < b * 32; e += 256) {
    const int r = e >> 5, c = e & 31;
    if (c0 + c < b) put(Tr + base, b, r, c0 + c, Y[r * LDY + c]);
  }
  for (int c = warp; c < 32 && c0 + c < b; c += 8)
    for (int r = lane; r < b; r += 32) put(Tc + base, b, c0 + c, r, Y[r * LDY + c]);
}

// ---------------------------------------------------------------------------
// the solves
// ---------------------------------------------------------------------------
template <typename T>
struct BlockArgs {
  const cx<T> *rhs[2];
  cxd *X[2];
  const int *idx[2];      // off-diagonal entries of the matrix and of its conjugate transpose
  const cx<T> *va[2], *vb[2];
  int K;
  const cxd *z;           // node shifts (conjugated for side 1)
  int fmap[kMaxNe];
};

// grid (column groups, nodes, sides).  Two groups of 256 consumer threads and
// one producer warp, which streams the tiles of T, eight columns at a time,
// through shared memory with bulk copies (full / empty mbarriers, bounded
// waits).  The groups take alternate chunks, each with full mbarriers of its own,
// and their sums are added through shared memory.  (With an odd number of stages
// both groups meet every stage, in turns.  On full barriers shared by the groups
// each would see every second phase only, and a wait by parity for phase p + 2
// passes while p + 1 is still being filled: copies may land out of order, and a
// warp without rows gets there first.)  (One group, two warps a sub-partition, left the FMA pipe idle
// half of the time; copies issued by a consumer thread delayed its warp and
// with it everyone.)
// A step: the right-hand side of the product, t = source - M_{i,i-1} z
// (forward; the source is r_i, and t is kept for the way back) or t = kept -
// M_{i,i+1} x; the product T_i t; the solution zb.  Source and off-diagonal
// entries of the next step are copied in during the product, so no global
// latency is left on the chain.  A conjugated factor (conjugate node, or T^H)
// is applied as conj(T conj(t)).  mode 0: the solution goes to X; mode 1: it
// replaces the right-hand side (read to the end by then) for block_solve_sides
// to add to X, since a load of X on the chain cost as much as the product.
template <typename T, int C, int U>
__global__ void __launch_bounds__(kCons + 32, 1)
    k_block_solve(int n, int b, int nblk, int stages, const cx<T> *__restrict__ Tc, const cx<T> *__restrict__ Tr,
                  const __grid_constant__ BlockArgs<T> io, size_t rns, int m, size_t xns, int mode, cx<T> *ys, int *err) {
  using Prod = Product<T, C, U>;
  using Rhs = typename Prod::Rhs;
  constexpr int R = kGroups * C, KC = Chunk<T>::KC;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int side = blockIdx.z, node = blockIdx.y, c0 = blockIdx.x * R;
  const int slot = io.fmap[node] & 0xffff;
  const bool cj = (io.fmap[node] >> 16) & 1;
  const bool neg = (side == 1) != cj;
  const int K = io.K;
  const int tile = KC * b;  // entries of a stage
  cx<T> *stage = reinterpret_cast<cx<T> *>(smem_raw);
  Rhs *tb = reinterpret_cast<Rhs *>(stage + (size_t)stages * tile);  // b x R: right-hand side of the product
  cx<T> *zb = reinterpret_cast<cx<T> *>(tb + (size_t)b * R);         // b x R: solution of the neighbouring block
  cx<T> *src = zb + (size_t)b * R;                                   // b x R: source of the next step
  cx<T> *va = src + (size_t)b * R;                                   // b x K entries of A
  cx<T> *vb = va + (size_t)b * K;                                    // ... of B (if any)
  int *ix = reinterpret_cast<int *>(vb + (io.vb[0] ? (size_t)b * K : 0));  // b x K local columns
  uint64_t *full = reinterpret_cast<uint64_t *>(ix + (size_t)b * K);  // of group g and stage s at g kMaxStages + s
  uint64_t *empty = full + 2 * kMaxStages;
  const int period = (stages & 1) ? stages : stages / 2;  // chunks of a group between two uses of a stage
  const int tid = threadIdx.x;
  if (tid == 0) {
    for (int s = 0; s < stages; ++s) {
      mbar::init(&full[s], 1);
      mbar::init(&full[kMaxStages + s], 1);
      mbar::init(&empty[s], kGroup / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  const int nch = b / KC;                         // chunks of one product (even)
  const int nsteps = 2 * nblk - 1;
  const cx<T> *Tb = (side ? Tr : Tc) + (size_t)slot * nblk * b * b;
  auto block_of = [&](int s) { return s < nblk ? s : 2 * nblk - 2 - s; };

  if (tid >= kCons) {
    // ---- producer: the products' tiles in order, no division in the loop ----
    if (tid == kCons) {
      const uint32_t bytes = (uint32_t)(tile * sizeof(cx<T>));
      bool ok = true;
      int s = 0, par = 1, pending = 0;  // stage; parity of its release (the first round passes at once)
      for (int p = 0; p < nsteps && ok; ++p) {
        const cx<T> *g = Tb + (size_t)block_of(p) * b * b;
        for (int c = 0; c < nch; ++c, g += tile) {
          if (!mbar::wait(&empty[s], par, kSpin)) {
            ok = false;
            break;
          }
          uint64_t *f = &full[(c & 1) * kMaxStages + s];
          mbar::expect_tx(f, bytes);
          mbar::bulk_load(stage + (size_t)s * tile, g, bytes, f);
          ++pending;
          if (++s == stages) {
            s = 0;
            par ^= 1;
          }
        }
      }
      if (!ok) {
        atomicOr(err, DEVERR_TIMEOUT);
        // copies still in flight land (bounded) before the shared memory is given up
        for (int k = max(0, pending - stages); k < pending; ++k)
          mbar::wait(&full[(k & 1) * kMaxStages + k % stages], (k / 2 / period) & 1, kSpin);
      }
    }
    return;
  }
  const int half = tid / kGroup, gt = tid - half * kGroup;
  const int RG = ceil_div(b / Prod::kRowsPer, U);
  const int cg = gt / RG, rg = gt - cg * RG;
  const bool act = cg < kGroups;
  const cx<T> *Rh = (side ? io.rhs[1] : io.rhs[0]) + (size_t)node * rns;
  cxd *Xn = (side ? io.X[1] : io.X[0]) + (size_t)node * xns;
  cx<T> *Dn = const_cast<cx<T> *>(Rh);  // mode 1
  cx<T> *Ys = ys + (((size_t)side * gridDim.y + node) * gridDim.x + blockIdx.x) * (size_t)nblk * b * R;
  const int *gix = side ? io.idx[1] : io.idx[0];
  const cx<T> *gva = side ? io.va[1] : io.va[0], *gvb = side ? io.vb[1] : io.vb[0];
  const cxd zz = io.z[node];
  const cx<T> zn = mk<T>((T)zz.re, side ? (T)-zz.im : (T)zz.im);
  const size_t dirs = (size_t)nblk * b * K;
  bool dead = false;
  int st = half, uses = 0, par = 0;  // the group's next chunk: its stage, and the parity of that stage's use
  auto advance = [&]() {
    st += 2;
    if (st >= stages) st -= stages;
    if (++uses == period) {
      uses = 0;
      par ^= 1;
    }
  };
  Prod prod;

  // source rows and off-diagonal entries of step s
  auto prefetch = [&](int s) {
    const bool fwd = s < nblk;
    const int i = block_of(s);
    for (int e = tid; e < b * R; e += kCons) {
      if (fwd) {
        const int r = e / R, c = e - r * R, row = i * b + r;
        const bool in = row < n && c0 + c < m;
        cp_async(src + e, in ? Rh + (size_t)row * m + c0 + c : Rh, in);
      } else {
        cp_async(src + e, Ys + (size_t)i * b * R + e, true);
      }
    }
    if (s > 0) {
      const size_t o = (fwd ? 0 : dirs) + (size_t)i * b * K;
      for (int e = tid; e < b * K; e += kCons) {
        cp_async(ix + e, gix + o + e);
        cp_async(va + e, gva + o + e, true);
        if (gvb) cp_async(vb + e, gvb + o + e, true);
      }
    }
  };
  prefetch(0);
  cp_async_wait();
  cons_bar();
  for (int s = 0; s < nsteps; ++s) {
    const bool fwd = s < nblk;
    const int i = block_of(s);
    // ---- t = source - M_{i, neighbour} zb = source + A zb - z B zb ----
    for (int e = tid; e < b * kGroups; e += kCons) {
      const int r = e / kGroups, g = e - r * kGroups;
      cx<T> t[C];
      load_row(t, src + r * R + g * C);
      if (s > 0)
        for (int k = 0; k < K; ++k) {
          cx<T> v = va[r * K + k];
          if (gvb) v = v - zn * vb[r * K + k];
          cx<T> x[C];
          load_row(x, zb + ix[r * K + k] * R + g * C);
#pragma unroll
          for (int c = 0; c < C; ++c) cfma(t[c], v, x[c]);
        }
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (fwd && i + 1 < nblk) Ys[((size_t)i * b + r) * R + g * C + c] = t[c];
        tb[r * R + g * C + c] = Prod::rhs(neg ? conj(t[c]) : t[c]);
      }
    }
    cons_bar();
    if (s + 1 < nsteps) prefetch(s + 1);
    // ---- product ----
    prod.zero();
    for (int ch = half; ch < nch; ch += 2) {
      if (!dead && !mbar::wait(&full[half * kMaxStages + st], par, kSpin)) {
        dead = true;
        atomicOr(err, DEVERR_TIMEOUT);
      }
      if (act && !dead) prod.stage(stage + (size_t)st * tile, tb + (size_t)ch * KC * R + cg * C, b, R, rg, RG);
      __syncwarp();
      if ((tid & 31) == 0) mbar::arrive(&empty[st]);
      advance();
    }
    // zb is not read any more in this step: the second group's sums, then the
    // solution of the block
    if (act && half)
      prod.each(rg, RG, [&](int r, int c, cx<T> a) {
        if (r < b) zb[r * R + cg * C + c] = a;
      });
    cons_bar();
    if (act && !half)
      prod.each(rg, RG, [&](int r, int c, cx<T> a) {
        if (r >= b) return;
        a = a + zb[r * R + cg * C + c];
        zb[r * R + cg * C + c] = neg ? conj(a) : a;
      });
    cp_async_wait();
    cons_bar();
    if (s + 1 >= nblk)
      for (int e = tid; e < b * R; e += kCons) {
        const int r = e / R, c = e - r * R, row = i * b + r;
        if (row < n && c0 + c < m) {
          if (mode)
            Dn[(size_t)row * m + c0 + c] = zb[e];
          else
            Xn[(size_t)row * m + c0 + c] = ccast<double>(zb[e]);
        }
      }
  }
}

// X += D (complex T)
template <typename T>
__global__ void k_block_add(cxd *__restrict__ X, const cx<T> *__restrict__ D, size_t count) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
    X[e] = X[e] + ccast<double>(D[e]);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
constexpr size_t kSmem = 224 * 1024;  // dynamic shared memory of a CTA at most

static int sm_count() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <typename T> static size_t solve_bytes(int b, int R, int K, bool hasB, int stages) {
  const size_t es = sizeof(cx<T>), rs = sizeof(typename Product<T, 1, 1>::Rhs);
  return ((size_t)stages * Chunk<T>::KC * b + 2 * (size_t)b * R + (size_t)(hasB ? 2 : 1) * b * K) * es +
         (size_t)b * R * rs + (size_t)b * K * sizeof(int) + 3 * kMaxStages * sizeof(uint64_t);
}
template <typename T> static size_t inv_bytes(int b) {
  return ((size_t)b * 33 + 16 * (size_t)(b + 2) + 2 * 512 + 16 * 17) * sizeof(cx<T>);
}

// Columns of a CTA.  A CTA's time a step is that of its FMAs (proportional to
// the columns) plus a fixed part worth about 4 columns (the stream of T, the
// barriers); CTAs beyond one an SM take another round.
template <typename T> static int pick_columns(int m, int ne, int nsides) {
  if (sizeof(T) == 8) return 1;  // FP64-bound: 4 columns, several CTAs an SM
  const int sms = sm_count();
  int best = 4;
  double cost = 1e30;
  for (int c : {4, 2, 1}) {
    const int ctas = ceil_div(m, kGroups * c) * ne * nsides;
    const double t = (double)ceil_div(ctas, sms) * (kGroups * c + 4);
    if (t < cost - 1e-9) {
      cost = t;
      best = c;
    }
  }
  return best;
}

int block_size(int kl, int ku) { return std::max(16, ceil_div(std::max(kl, ku), 16) * 16); }

// Whether the block form is used (with kBlockMaxEntries, since the entries'
// products are formed for every few columns).  Blocks of up to 256: n = 12000,
// 8 nodes, 24 columns, factorisation and three solves took 10.6 ms against
// 15.6 with the triangular factors at a band of 100, 14.2 against 20.3 at 256;
// with 16 nodes and 62 columns, which fill the chip, 38.6 against 42.9 and 43.1
// against 43.5.  At 300 there the solves take as long (37.2 and 37.7 ms at
// n = 90000) and the inverses 35 ms, and more refinement steps are needed.
constexpr int kMaxBlock = 256;
bool block_solve_fits(int kl, int ku) { return block_size(kl, ku) <= kMaxBlock; }
// FP64: a filter takes two sweeps (the refinement), each bound by the FP64 pipe,
// so that its time goes with the number of rounds that its CTAs of four columns
// make on the chip; the triangular solves are one chain of windows whatever the
// columns.  8000 rows, ms a filter in 1, 2, 3, 4 rounds against the factors: b =
// 16 5.7, 11.6, 17.2, 22.9 and 20; b = 48 7.5, 15, 23, 30 and 28; b = 112 15, 30,
// 45, 60 and 45; b = 176 25, 50, 75, 100 and 66 to 72; b = 256 33, 66, 99, 132 and
// 88 to 94.
bool block_solve_pays_f64(int kl, int ku, int m, int ne, int nsides) {
  const int rounds = ceil_div(ceil_div(m, kGroups) * ne * nsides, sm_count());
  return rounds <= (block_size(kl, ku) <= 96 ? 3 : 2);
}

// Largest number of off-diagonal entries of a row towards one block into
// *d_kmax (zeroed by the caller).
void launch_block_count(const CsrView &A, const CsrView *B, int kl, int ku, int *d_kmax, cudaStream_t s) {
  k_block_count<<<grid_for(A.n), 256, 0, s>>>(A, B ? *B : A, B != nullptr, block_size(kl, ku), d_kmax);
  note_launch();
}
size_t block_entry_count(int n, int kl, int ku, int K) {
  const int b = block_size(kl, ku);
  return (size_t)2 * ceil_div(n, b) * b * K;
}
template <typename T>
void launch_block_entries(const CsrView &A, const CsrView *B, int kl, int ku, int K, int *idx, cx<T> *va, cx<T> *vb,
                          cudaStream_t s) {
  const int b = block_size(kl, ku), rows = ceil_div(A.n, b) * b;
  k_block_entries<T><<<grid_for(rows), 256, 0, s>>>(A, B ? *B : A, B != nullptr, b, K, rows, idx, va, vb);
  note_launch();
}
template void launch_block_entries<float>(const CsrView &, const CsrView *, int, int, int, int *, cxf *, cxf *,
                                          cudaStream_t);
template void launch_block_entries<double>(const CsrView &, const CsrView *, int, int, int, int *, cxd *, cxd *,
                                           cudaStream_t);

size_t block_elems(int n, int kl, int ku, int nf) {
  const int b = block_size(kl, ku);
  return (size_t)nf * ceil_div(n, b) * b * b;
}
size_t block_scratch_elems(int n, int kl, int ku, int m, int ne) {
  const int b = block_size(kl, ku);
  return (size_t)2 * ne * (ceil_div(m, 16) * 16) * ceil_div(n, b) * b;
}

template <typename T>
cudaError_t block_invert(int n, int kl, int ku, int klp, int kup, int nf, const cx<T> *band, const cx<T> *dinv,
                         cx<T> *Tc, cx<T> *Tr, cudaStream_t s) {
  const int b = block_size(kl, ku);
  auto kern = k_block_inv<T>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)inv_bytes<T>(b));
  if (e != cudaSuccess) return e;
  // the blocks on x: more than 65535 of them (the limit of y) from n = 1048561 with blocks of 16
  kern<<<dim3(ceil_div(n, b), ceil_div(b, 32), nf), 256, inv_bytes<T>(b), s>>>(
      n, klp, kup, b, band, (size_t)n * (klp + kup + 1), dinv, Tc, Tr);
  note_launch();
  return cudaGetLastError();
}
template cudaError_t block_invert<float>(int, int, int, int, int, int, const cxf *, const cxf *, cxf *, cxf *,
                                         cudaStream_t);
template cudaError_t block_invert<double>(int, int, int, int, int, int, const cxd *, const cxd *, cxd *, cxd *,
                                          cudaStream_t);

template <typename T>
cudaError_t block_solve_sides(int n, int kl, int ku, int ne, const int *fmap, const cx<T> *Tc, const cx<T> *Tr,
                              const BlockEntries &en, const cxd *d_z, const cx<T> *rhsR, const cx<T> *rhsL, size_t rns,
                              int m, cxd *XR, cxd *XL, size_t xns, int mode, cx<T> *ys, int *err, cudaStream_t s) {
  const int b = block_size(kl, ku), nblk = ceil_div(n, b), K = en.K;
  BlockArgs<T> io;
  io.rhs[0] = rhsR;
  io.rhs[1] = rhsL ? rhsL : rhsR;
  io.X[0] = XR;
  io.X[1] = XL ? XL : XR;
  for (int k = 0; k < 2; ++k) {
    io.idx[k] = en.idx[k];
    io.va[k] = reinterpret_cast<const cx<T> *>(en.va[k]);
    io.vb[k] = reinterpret_cast<const cx<T> *>(en.vb[k]);
  }
  io.K = K;
  io.z = d_z;
  for (int j = 0; j < kMaxNe; ++j) io.fmap[j] = j < ne ? fmap[j] : 0;
  const int nsides = (rhsL && XL) ? 2 : 1;
  const bool hasB = io.vb[0] != nullptr;
  int C = pick_columns<T>(m, ne, nsides);
  auto bytes = [&](int st) { return solve_bytes<T>(b, kGroups * C, K, hasB, st); };
  while (C > 1 && bytes(2) > kSmem) C /= 2;
  // FP64 CTAs share an SM where they can (the FP64 pipe is the bound), so few stages
  int stages = sizeof(T) == 8 ? 3 : kMaxStages;
  while (stages > 2 && bytes(stages) > kSmem) --stages;
  const int R = kGroups * C;
  const size_t smem = bytes(stages);
  const dim3 grid(ceil_div(m, R), ne, nsides);
  const int U = ceil_div(b / Product<T, 1, 1>::kRowsPer, kGroup / kGroups);
  cudaError_t e = cudaErrorInvalidValue;
#define BLK(c, u)                                                                                          \
  do {                                                                                                     \
    auto kern = k_block_solve<T, c, u>;                                                                    \
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);                \
    if (e == cudaSuccess) {                                                                                \
      kern<<<grid, kCons + 32, smem, s>>>(n, b, nblk, stages, Tc, Tr, io, rns, m, xns, mode, ys, err);     \
      note_launch();                                                                                       \
      e = cudaGetLastError();                                                                              \
    }                                                                                                      \
  } while (0)
  if constexpr (sizeof(T) == 8) {
    switch (U) {
      case 1: BLK(1, 1); break;
      case 2: BLK(1, 2); break;
      case 3: BLK(1, 3); break;
      case 4: BLK(1, 4); break;
    }
  } else {
#define BLKU(c)               \
  switch (U) {                \
    case 1: BLK(c, 1); break; \
    case 2: BLK(c, 2); break; \
  }
    if (C == 1) {
      BLKU(1)
    } else if (C == 2) {
      BLKU(2)
    } else {
      BLKU(4)
    }
#undef BLKU
  }
#undef BLK
  if (e != cudaSuccess || !mode) return e;
  const size_t count = (size_t)ne * n * m;
  for (int k = 0; k < nsides; ++k) {
    k_block_add<T><<<grid_for(count), 256, 0, s>>>(io.X[k], io.rhs[k], count);
    note_launch();
  }
  return cudaGetLastError();
}
template cudaError_t block_solve_sides<float>(int, int, int, int, const int *, const cxf *, const cxf *,
                                              const BlockEntries &, const cxd *, const cxf *, const cxf *, size_t, int,
                                              cxd *, cxd *, size_t, int, cxf *, int *, cudaStream_t);
template cudaError_t block_solve_sides<double>(int, int, int, int, const int *, const cxd *, const cxd *,
                                               const BlockEntries &, const cxd *, const cxd *, const cxd *, size_t, int,
                                               cxd *, cxd *, size_t, int, cxd *, int *, cudaStream_t);
