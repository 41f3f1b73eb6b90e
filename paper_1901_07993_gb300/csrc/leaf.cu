// leaf.cu -- batched leaf routine of Algorithms 1-2 ("factorize S^-1 = Z Z*"):
// for each nl x nl SPD matrix, the Cholesky factor S = L L^T and Z = L^-T.
//
// One thread-block cluster per matrix, FP64, 32 x 32 tiles.  An SM issues
// about two FP64 FMAs per clock, so a tile product (32^3 FMAs) takes 8 us on
// one SM and a 512-row leaf 11 ms: the work of a leaf is spread over up to 16
// SMs, which meet at cluster barriers.  L and W = L^-1 are built together,
// right-looking.  X(r, k) names tile (r, k) of the array: below the diagonal
// it holds A, then L; above it B^T, then W^T (= Z), B the right-hand side
// that starts as the identity.  Step k:
//   1. column k: below the diagonal Y L_kk^T = X(r, k) is solved by substitution
//      (Y = L_rk), above it X(r, k) <- X(r, k) W_kk^T (Z_rk), one tile per CTA;
//   2. X(r, j) -= X(r, k) X(j, k)^T for every j > k and r <= k (B, with
//      X(k, k) = W_kk^T and B_jk = 0 before) or r >= j (A); tile (k+1, k+1)
//      first, and CTA 0 factors it at once (L_kk and W_kk = L_kk^-1 for the
//      next step) while the others go on, so the serial chain of pivots overlaps
//      the updates.
// For accuracy a tile product is summed by itself and subtracted once (one chain
// of FMAs through all of a tile's products loses a factor of three on 3D
// leaves), and neither the panel nor the pivots go through a reciprocal: the
// panel times W_kk^T loses up to a factor of 15 in Z on chains of condition
// 1e6 and more.
// Every step has T^2 / 2 to T tile products (T = nl / 32); the columns of W
// after all of L would be chains of very different length.  Call times against
// one CTA per matrix: 8 leaves of 512 rows 15.9 -> 1.54 ms (0.47 TFLOP/s of the
// FP64 pipe's 1.25), one 15.9 -> 1.17 ms, 32 leaves 16.0 -> 3.9 ms, one of 128
// rows 572 -> 226 us, one of 1024 rows 113 -> 7.0 ms, 1000 of 32 rows 227 -> 202 us.
//
// A non-positive pivot j sets info = j + 1 (the pivot is replaced by 1 so the
// arithmetic stays finite; that matrix's Z is then meaningless).
#include "internal.cuh"

namespace ifac {

namespace {
constexpr int TB = 32;
constexpr int LD = TB + 1;  // padded shared-memory row
constexpr int NT = 256;
// CTA 0's update and factorization of the next diagonal tile, in tile products:
// eight leaves of 512 rows 1.66 ms with 3, 1.57 with 4, 1.54 with 5 or 6
constexpr int DIAG_COST = 5;

__device__ __forceinline__ int cluster_rank() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ int cluster_size() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// all threads of the cluster; global writes before it are visible after it
// (readers load through L2, __ldcg)
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// x / d from r ~ 1 / d: one Newton step on the residual, which leaves the
// quotient as accurate as a division (r up to an ulp off) in three dependent
// FP64 operations.  With a division and a root for every pivot a leaf of 32 rows
// took 77 us, eight of 512 rows 2.2 ms.
__device__ __forceinline__ double quotient(double x, double d, double r) {
  const double q = x * r;
  return fma(fma(-q, d, x), r, q);
}
// positive, of a magnitude whose root, reciprocal and residuals stay normal (on
// the exponent field: a comparison would wait for the FP64 pipe)
__device__ __forceinline__ bool usual(double x) {
  return (uint32_t)__double2hiint(x) - ((1023u - 800u) << 20) < (1600u << 20);
}

// W = L^-1 of the tile L L^T = t (LD rows, lower triangle used): four warps,
// lane = row, warp w holds columns w, w + 4, ... of the tile and of W, so the
// FP64 work of a pivot is spread over the SM; one named barrier per pivot.
// (The next pivot's root taken ahead of the other updates measured no faster.)
// L takes the tile's place.  Returns 1 + the first non-positive pivot, or 0 (the
// same in all four warps).
__device__ __forceinline__ int factor_tile(double* t, double* __restrict__ W) {
  __shared__ double col[2][TB + 1];
  __shared__ int sbad;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) sbad = 0;
  double a[TB / 4], b[TB / 4], rown = 1.0, rinv = 1.0;
#pragma unroll
  for (int q = 0; q < TB / 4; ++q) {
    a[q] = t[lane * LD + w + 4 * q];
    b[q] = (lane == w + 4 * q) ? 1.0 : 0.0;
  }
#pragma unroll
  for (int jq = 0; jq < TB / 4; ++jq) {
#pragma unroll 1
    for (int jw = 0; jw < 4; ++jw) {
      const int j = 4 * jq + jw;
      double* c = col[jw & 1];
      if (w == jw) {
        double d = __shfl_sync(0xffffffffu, a[jq], j);
        if (!usual(d) && !(d > 0.0)) {
          if (lane == 0 && !sbad) sbad = j + 1;
          d = 1.0;
        }
        // rows below the pivot: L_ij; row j: 1 / L_jj
        const double x = lane == j ? 1.0 : a[jq];
        double r, q;
        if (usual(d)) {  // the root by a Newton step from rsqrt
          const double rs = rsqrt(d), r0 = d * rs;
          r = fma(fma(-r0, r0, d), 0.5 * rs, r0);
          q = quotient(x, r, rs);
        } else {
          r = sqrt(d);
          q = x / r;
        }
        c[lane] = q;
        if (lane == 0) c[TB] = r;
        if (lane >= j) t[lane * LD + j] = lane == j ? r : q;
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      // row j of B stays unscaled until the end: its factor goes into L_ij
      const double li = lane > j ? -c[lane] : 0.0, lr = li * c[j];
      if (lane == j) {
        rown = c[TB];
        rinv = c[j];
      }
#pragma unroll
      for (int q = 0; q < TB / 4; ++q) {
        const int cc = w + 4 * q;
        if (cc > j) a[q] = fma(li, c[cc], a[q]);
        else b[q] = fma(lr, __shfl_sync(0xffffffffu, b[q], j), b[q]);
      }
    }
  }
  const bool quick = usual(rown);
#pragma unroll
  for (int q = 0; q < TB / 4; ++q) W[lane * TB + w + 4 * q] = quick ? quotient(b[q], rown, rinv) : b[q] / rown;
  asm volatile("bar.sync 1, 128;" ::: "memory");
  return sbad;
}

// Y L^T = X for the tile X in x (LD rows) by substitution, L lower triangular
// in l (LD rows), rd[j] = 1 / L_jj, Y in x's place: lane = row, warp w holds columns w, w + 8, ...,
// one barrier per column (256 threads; callers have synchronised).
__device__ __forceinline__ void solve_tile(double* x, const double* l, const double* rd) {
  __shared__ double col[2][TB];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double a[TB / 8];
#pragma unroll
  for (int q = 0; q < TB / 8; ++q) a[q] = x[lane * LD + w + 8 * q];
#pragma unroll
  for (int jq = 0; jq < TB / 8; ++jq) {
#pragma unroll 1
    for (int jw = 0; jw < 8; ++jw) {
      const int j = 8 * jq + jw;
      double* c = col[jw & 1];
      if (w == jw) {
        const double d = l[j * LD + j], y = usual(d) ? quotient(a[jq], d, rd[j]) : a[jq] / d;
        c[lane] = y;
        a[jq] = y;
      }
      __syncthreads();
      const double y = -c[lane];
#pragma unroll
      for (int q = jq; q < TB / 8; ++q)
        if (w + 8 * q > j) a[q] = fma(y, l[(w + 8 * q) * LD + j], a[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < TB / 8; ++q) x[lane * LD + w + 8 * q] = a[q];
}
}  // namespace

__global__ void __launch_bounds__(NT) k_leaf_invchol(double* __restrict__ Abase, int nl, int* __restrict__ info,
                                                     double* __restrict__ Wdiag_base) {
  __shared__ double xs[TB * LD], ys[TB * LD], zs[TB * LD], rd[TB];
  const int tid = threadIdx.x, rank = cluster_rank(), C = cluster_size();
  const int T = nl / TB;
  const size_t mat = blockIdx.x / C;
  double* A = Abase + mat * nl * nl;
  double* Wd = Wdiag_base + mat * T * TB * TB;  // W_kk, row-major, lower triangular
  int bad = 0;
  const auto tile = [&](int r, int c) { return A + (size_t)r * TB * nl + c * TB; };
  // this thread's four elements of a tile: rows tid / 32 + 8 i, column tid % 32
  const int er = tid >> 5, ec = tid & 31;
  const auto fetch = [&](const double* p, size_t ld, double (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __ldcg(p + (er + 8 * i) * ld + ec);
  };
  const auto place = [&](double* s, const double (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) s[(er + 8 * i) * LD + ec] = v[i];
  };
  const auto place_t = [&](double* s, const double (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) s[ec * LD + er + 8 * i] = v[i];
  };
  const auto factor = [&](int k) {  // the diagonal tile in xs (all threads; the first four warps work)
    if (tid < 128) {
      const int j = factor_tile(xs, Wd + (size_t)k * TB * TB);
      if (j && !bad) bad = k * TB + j;
    }
    __syncthreads();
    double* p = tile(k, k);  // L_kk, below and on the diagonal
#pragma unroll
    for (int i = 0; i < 4; ++i) p[(size_t)(er + 8 * i) * nl + ec] = xs[(er + 8 * i) * LD + ec];
  };

  if (rank == 0) {
    double v[4];
    fetch(tile(0, 0), nl, v);
    place(xs, v);
    __syncthreads();
    factor(0);
  }
  cluster_sync();
  for (int k = 0; k < T; ++k) {
    // ---- 1. column k: tiles u < k above the diagonal times W_kk^T, the others solved ----
    {
      bool have_w = false, have_l = false;  // W_kk in ys; L_kk in zs, 1 / its diagonal in rd
      for (int u = rank; u < T - 1; u += C) {
        const bool above = u < k;
        double* X = tile(above ? u : u + 1, k);
        double v[4], d4[4];
        const bool need = above ? !have_w : !have_l;
        if (need) {
          if (above) fetch(Wd + (size_t)k * TB * TB, TB, d4);
          else fetch(tile(k, k), nl, d4);
        }
        if (!above && need && tid < TB) rd[tid] = __ldcg(Wd + (size_t)k * TB * TB + tid * (TB + 1));
        fetch(X, nl, v);
        if (need) place(above ? ys : zs, d4);
        (above ? have_w : have_l) = true;
        place(xs, v);
        __syncthreads();
        if (above) {
          // warp w has columns 4w .. 4w + 3, which need the first 4w + 4 terms
          // of the lower-triangular W_kk
          const int c0 = (tid >> 5) * 4 + ((tid >> 4) & 1) * 2, r0 = (tid & 15) * 2, n = (tid >> 5) * 4 + 4;
          double s00 = 0, s01 = 0, s10 = 0, s11 = 0;
#pragma unroll 4
          for (int l = 0; l < n; ++l) {
            const double a0 = xs[r0 * LD + l], a1 = xs[(r0 + 1) * LD + l];
            const double b0 = ys[c0 * LD + l], b1 = ys[(c0 + 1) * LD + l];
            s00 = fma(a0, b0, s00);
            s01 = fma(a0, b1, s01);
            s10 = fma(a1, b0, s10);
            s11 = fma(a1, b1, s11);
          }
          __syncthreads();  // xs is reused: the result goes out in rows
          xs[r0 * LD + c0] = s00;
          xs[r0 * LD + c0 + 1] = s01;
          xs[(r0 + 1) * LD + c0] = s10;
          xs[(r0 + 1) * LD + c0 + 1] = s11;
        } else {
          solve_tile(xs, zs, rd);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) X[(size_t)(er + 8 * i) * nl + ec] = xs[(er + 8 * i) * LD + ec];
        __syncthreads();
      }
    }
    if (k + 1 == T) break;
    cluster_sync();
    // ---- 2. trailing updates ----
    // units: column j = k + 1 .. T - 1, rows 0 .. k and j .. T - 1, without (k + 1, k + 1)
    const int m = T - 1 - k;
    const int units = m * (k + 1) + m * (m + 1) / 2 - 1;
    const int share0 = C == 1 ? units : max(0, (units + DIAG_COST + C - 1) / C - DIAG_COST);
    const int first = rank == 0 ? -1 : share0 + rank - 1, step = rank == 0 ? 1 : C - 1;
    const int last = rank == 0 ? share0 : units;
    int r = k + 1, j = k + 1;  // unit -1: the next diagonal tile
    const auto decode = [&](int u) {
      int jj = k + 1, n = k + 1 + T - jj - 1;
      while (u >= n) {
        u -= n;
        ++jj;
        n = k + 1 + T - jj;
      }
      j = jj;
      r = u <= k ? u : jj + (u - (k + 1)) + (jj == k + 1 ? 1 : 0);
    };
    const int orow = (tid >> 4) * 2, ocol = (tid & 15) * 2;
    double va[4], vb[4], c0[4];  // the next unit's operands, loaded while this one is multiplied
    const auto load_unit = [&] {
      if (r == k) fetch(Wd + (size_t)k * TB * TB, TB, va);
      else fetch(tile(r, k), nl, va);
      fetch(tile(j, k), nl, vb);
      const double* p = tile(r, j) + (size_t)orow * nl + ocol;
#pragma unroll
      for (int i = 0; i < 4; ++i) c0[i] = r == k ? 0.0 : __ldcg(p + (size_t)(i >> 1) * nl + (i & 1));
    };
    if (rank != 0 && first < last) decode(first);
    if (first < last) load_unit();
    for (int u = first; u < last; u += step) {
      const int ur = r, uj = j;
      if (ur == k) place_t(xs, va);
      else place(xs, va);
      place(ys, vb);
      const double x00 = c0[0], x01 = c0[1], x10 = c0[2], x11 = c0[3];
      double s00 = 0.0, s01 = 0.0, s10 = 0.0, s11 = 0.0;
      __syncthreads();
      if (u >= 0 && u + step < last) {
        decode(u + step);
        load_unit();
      }
#pragma unroll 8
      for (int l = 0; l < TB; ++l) {
        const double a0 = xs[orow * LD + l], a1 = xs[(orow + 1) * LD + l];
        const double b0 = ys[ocol * LD + l], b1 = ys[(ocol + 1) * LD + l];
        s00 = fma(a0, b0, s00);
        s01 = fma(a0, b1, s01);
        s10 = fma(a1, b0, s10);
        s11 = fma(a1, b1, s11);
      }
      s00 = x00 - s00;
      s01 = x01 - s01;
      s10 = x10 - s10;
      s11 = x11 - s11;
      __syncthreads();
      if (u < 0) {  // CTA 0: factor the next diagonal tile
        xs[orow * LD + ocol] = s00;
        xs[orow * LD + ocol + 1] = s01;
        xs[(orow + 1) * LD + ocol] = s10;
        xs[(orow + 1) * LD + ocol + 1] = s11;
        __syncthreads();
        factor(k + 1);
        __syncthreads();
        if (last > 0) {
          decode(0);
          load_unit();
        }
        continue;
      }
      double* p = tile(ur, uj) + (size_t)orow * nl + ocol;
      p[0] = s00;
      p[1] = s01;
      p[nl] = s10;
      p[nl + 1] = s11;
    }
    cluster_sync();
  }
  cluster_sync();  // the strictly lower tiles are no longer read
  // diagonal tiles Z_kk = W_kk^T, strictly lower tiles cleared
  for (int u = rank; u < T * T; u += C) {
    const int r = u / T, c = u % T;
    if (r < c) continue;
    double* p = tile(r, c);
    if (r == c) {
      double v[4];
      fetch(Wd + (size_t)r * TB * TB, TB, v);
      place(xs, v);
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) p[(size_t)(er + 8 * i) * nl + ec] = r == c ? xs[ec * LD + er + 8 * i] : 0.0;
    if (r == c) __syncthreads();
  }
  if (rank == 0 && tid == 0) info[mat] = bad;
}

__global__ void k_pad_identity(const double* __restrict__ src, int nl, double* __restrict__ dst, int np, int count) {
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t per = (int64_t)np * np;
  if (e >= per * count) return;
  int64_t k = e / per, q = e % per;
  int r = (int)(q / np), c = (int)(q % np);
  dst[e] = (r < nl && c < nl) ? src[k * nl * nl + (int64_t)r * nl + c] : (r == c ? 1.0 : 0.0);
}

__global__ void k_unpad(const double* __restrict__ src, int np, double* __restrict__ dst, int nl, int count) {
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t per = (int64_t)nl * nl;
  if (e >= per * count) return;
  int64_t k = e / per, q = e % per;
  int r = (int)(q / nl), c = (int)(q % nl);
  dst[e] = src[k * np * np + (int64_t)r * np + c];
}

// CTAs per matrix: the largest cluster of which `count` fit on the GPU with
// one CTA per SM (two CTAs on an SM would share its FP64 pipe), no more than
// half a step's tile products.  The dynamic shared memory keeps a second CTA
// off an SM; the device's cluster counts are asked for once.
constexpr int LEAF_SMEM = 120 * 1024;

static cudaError_t leaf_config(int count, int tiles, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at) {
  static constexpr int kSizes[] = {16, 12, 10, 8, 6, 5, 4, 3, 2};
  static std::atomic<int> fit[64][9];  // 0: not asked yet, else 1 + clusters on the device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_leaf_invchol, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_leaf_invchol, cudaFuncAttributeMaxDynamicSharedMemorySize, LEAF_SMEM);
  if (e != cudaSuccess) return e;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg->blockDim = dim3(NT);
  cfg->dynamicSmemBytes = LEAF_SMEM;
  cfg->attrs = at;
  cfg->numAttrs = 1;
  for (int i = 0; i < 9; ++i) {
    const int c = kSizes[i];
    if (c > tiles * tiles / 2) continue;
    at->val.clusterDim.x = (unsigned)c;
    cfg->gridDim = dim3((unsigned)(count * c));
    int n = fit[dev & 63][i].load();
    if (n == 0) {
      int q = 0;
      if (cudaOccupancyMaxActiveClusters(&q, k_leaf_invchol, cfg) != cudaSuccess) {
        cudaGetLastError();  // this size is not available: the next one
        q = 0;
      }
      fit[dev & 63][i].store(n = q + 1);
    }
    if (n - 1 >= count) return cudaSuccess;
  }
  at->val.clusterDim.x = 1;
  cfg->gridDim = dim3((unsigned)count);
  cfg->dynamicSmemBytes = 0;  // more matrices than SMs: their chains overlap on one
  return cudaSuccess;
}

static cudaError_t launch_leaf(cudaStream_t stream, int count, int nl, double* A, int* info, double* wd) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  const cudaError_t e = leaf_config(count, nl / TB, &cfg, &at);
  if (e != cudaSuccess) return e;
  cfg.stream = stream;
  return cudaLaunchKernelEx(&cfg, k_leaf_invchol, A, nl, info, wd);
}

// A: count matrices of nl x nl (in place).  Pads to a multiple of 32 with an
// identity block when needed (the padded part factors to the identity).
void leaf_invchol(ifac_ctx* ctx, int count, int nl, double* A, int* info) {
  if (count == 0) return;
  const int np = ((nl + TB - 1) / TB) * TB;
  const int T = np / TB;
  Buf<double> wd(ctx, (size_t)count * T * TB * TB);
  if (np == nl) {
    IFAC_CK(launch_leaf(ctx->stream, count, nl, A, info, wd.p));
    ++ctx->launches;
    return;
  }
  Buf<double> pad(ctx, (size_t)count * np * np);
  int64_t tot = (int64_t)count * np * np;
  k_pad_identity<<<cdiv(tot, 256), 256, 0, ctx->stream>>>(A, nl, pad.p, np, count);
  IFAC_CK_LAUNCH();
  IFAC_CK(launch_leaf(ctx->stream, count, np, pad.p, info, wd.p));
  ++ctx->launches;
  int64_t tot2 = (int64_t)count * nl * nl;
  k_unpad<<<cdiv(tot2, 256), 256, 0, ctx->stream>>>(pad.p, np, A, nl, count);
  IFAC_CK_LAUNCH();
}

}  // namespace ifac

namespace ifac {

// Same computation as leaf_invchol, with the scratch supplied by the caller
// instead of allocated: wd holds count * ceil(nl/32) * 32 * 32 doubles and,
// when nl is not a multiple of 32, pad holds count * np * np doubles
// (np = nl rounded up to 32).  Returns the launch status.
cudaError_t leaf_invchol_launch_scratch(cudaStream_t stream, int count, int nl, double* A, int* info, double* wd,
                                        double* pad) {
  if (count == 0) return cudaSuccess;
  const int np = ((nl + TB - 1) / TB) * TB;
  if (np == nl) {
    return launch_leaf(stream, count, nl, A, info, wd);
  }
  int64_t tot = (int64_t)count * np * np;
  k_pad_identity<<<cdiv(tot, 256), 256, 0, stream>>>(A, nl, pad, np, count);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = launch_leaf(stream, count, np, pad, info, wd);
  if (e != cudaSuccess) return e;
  int64_t tot2 = (int64_t)count * nl * nl;
  k_unpad<<<cdiv(tot2, 256), 256, 0, stream>>>(pad, np, A, nl, count);
  return cudaGetLastError();
}

}  // namespace ifac
