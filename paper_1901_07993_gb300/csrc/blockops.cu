// blockops.cu -- memory-bound block operations: sums on a union pattern,
// block Frobenius norms, ||A||_F, the Gershgorin bound and Z_0 = c I.
//
// Sums follow the definition alpha*a + beta*b + gamma*[diag] with explicit
// round-to-nearest multiplies and adds (no fused multiply-add), in that
// order, so each element is rounded exactly as the plain definition is.
// Reductions run in a fixed order (per row, then over rows), so results are
// deterministic from run to run.  The block norms of sums are summed through
// FP32 (SqAcc, SqAcc4: about 2^-44 relative) so that these kernels spend the FP64
// pipe -- GB300 runs about two FP64 operations per clock per SM -- on the
// sums alone.
#include <cmath>

#include "internal.cuh"
#include "tc_common.cuh"

using ifac::tc::load4;
using ifac::tc::SqAcc;

namespace ifac {

__device__ __forceinline__ double block_reduce_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < nw; ++w) t += red[w];
  __syncthreads();
  return t;  // valid in thread 0
}

// alpha x, rounded to nearest.  GB300's FP64 pipe is narrow, so the common
// scales avoid it: alpha = +-1 is a sign change and alpha = 2^k an exponent
// change on the bit pattern (same result), other alphas one multiply.
struct Scale {
  int mode;  // 0 multiply, 1 identity, 2 negate, 3 power of two
  int k;     // mode 3: alpha = 2^k
  double alpha;
};

static Scale make_scale(double alpha) {
  Scale s{0, 0, alpha};
  if (alpha == 1.0) s.mode = 1;
  else if (alpha == -1.0) s.mode = 2;
  else if (alpha > 0.0 && std::isfinite(alpha)) {
    int e = 0;
    if (std::frexp(alpha, &e) == 0.5) {
      s.mode = 3;
      s.k = e - 1;
    }
  }
  return s;
}

__device__ __forceinline__ double scaled(const Scale& s, double x) {
  if (s.mode == 1) return x;
  const int hi = __double2hiint(x), lo = __double2loint(x);
  if (s.mode == 2) return __hiloint2double(hi ^ (int)0x80000000, lo);
  if (s.mode == 3) {
    const int ex = (hi >> 20) & 0x7ff, en = ex + s.k;
    if (ex > 0 && ex < 0x7ff && en > 0 && en < 0x7ff) return __hiloint2double(hi + (s.k << 20), lo);
  }
  return __dmul_rn(s.alpha, x);
}

__device__ __forceinline__ double add_elem(const Scale& sa, const double* a, const Scale& sb, const double* b,
                                           bool diag, double gamma, int e) {
  double v = 0.0;
  if (a) v = scaled(sa, a[e]);
  if (b) {
    const double t = scaled(sb, b[e]);
    v = a ? __dadd_rn(v, t) : t;
  }
  if (diag) v = (a || b) ? __dadd_rn(v, gamma) : gamma;
  return v;
}

// four values times the scale, the mode tested once
__device__ __forceinline__ void scale4(const Scale& s, double (&x)[4]) {
  if (s.mode == 1) return;
  if (s.mode == 2) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = __hiloint2double(__double2hiint(x[i]) ^ (int)0x80000000, __double2loint(x[i]));
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = scaled(s, x[i]);
}

__device__ __forceinline__ void widen4(const double (&w)[4], double (&x)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = w[i];
}
__device__ __forceinline__ void widen4(const float (&w)[4], double (&x)[4]) { ifac::tc::f32_to_f64_x4(w, x); }

// the K-major low-precision copy that the tensor-core products read (TF32:
// FP32 round-to-nearest-even then TF32 round-half-away; BF16 round-to-
// nearest-even, as their operand conversion rounds), written beside the
// FP64 result: lp_elt 4 TF32, 2 BF16, 0 none
__device__ __forceinline__ void lp_store4(void* lp, int lp_elt, size_t i, const double (&x)[4]) {
  if (lp_elt == 4) {
    uint32_t w[4];
    ifac::tc::f64_to_tf32_x4(x, w);
    *reinterpret_cast<uint4*>(static_cast<uint32_t*>(lp) + i) = make_uint4(w[0], w[1], w[2], w[3]);
  } else if (lp_elt == 2) {
    uint32_t w[4];
    ifac::tc::f64_to_bf16_x4(x, w);
    *reinterpret_cast<uint2*>(static_cast<uint16_t*>(lp) + i) = make_uint2(w[0] | (w[1] << 16), w[2] | (w[3] << 16));
  }
}

// position of column c in ci[lo, hi) (sorted), -1 when absent: the warp probes
// 32 entries at a time, so a short row takes one load
__device__ __forceinline__ int find_warp(const int32_t* __restrict__ ci, int lo, int hi, int c) {
  const int lane = threadIdx.x & 31;
  while (hi - lo > 32) {
    const int step = (hi - lo + 31) / 32, p = lo + lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, p < hi && ci[p] <= c);
    if (!m) return -1;
    lo += (31 - __clz((int)m)) * step;
    hi = min(hi, lo + step);
  }
  const unsigned m = __ballot_sync(0xffffffffu, lo + lane < hi && ci[lo + lane] == c);
  return m ? lo + __ffs((int)m) - 1 : -1;
}

// the block's norm from its warps' sums of squares, added in warp order (one
// barrier per block: the caller alternates between two sets of partials)
template <int W>
__device__ __forceinline__ void block_norm(const ifac::tc::SqAcc4& sq, double (&part)[W], double* out) {
  const double t = sq.total().warp_total();
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = t;
  if constexpr (W > 1) __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
#pragma unroll
    for (int w = 0; w < W; ++w) sum += part[w];
    *out = sqrt(sum);
  }
}

// One CTA of W warps per output block (grid-stride over blocks).  Element by
// element v = 0 + alpha a + beta b + gamma [diagonal], left to right, each
// step rounded; the leading 0 + x is x.  B's values are FP64 or FP32 (TB).
// Bound by HBM: four values a thread and step as one 32-byte load per operand
// and one 32-byte store, their squares in four independent chains, and no
// branch per value.  (One warp per block, two values and a test of every
// value's magnitude at a time ran at 2.5 - 3.4 TB/s of 6.8, and small sums
// left most of the SMs' warps empty.)  Z + M of the 262,144-row chain with M
// in FP32 and Z's TF32 copy (1.2 GB): 349 -> 228 us; the FP64 sum of the 65,536-row
// chain with beta = -0.375 (302 MB, two FP64 operations a value): 123 -> 76 us; of
// the 4096-row chain at bs 32: 16 -> 5.6 us.
template <int W, typename TB>
__global__ void __launch_bounds__(32 * W)
    k_add(const int32_t* __restrict__ crow, const int32_t* __restrict__ cci, int64_t cnnz, int bs, Scale sa,
          const int32_t* __restrict__ arp, const int32_t* __restrict__ aci, const double* __restrict__ aval, Scale sb,
          const int32_t* __restrict__ brp, const int32_t* __restrict__ bci, const TB* __restrict__ bval,
          const int32_t* __restrict__ bmap, double gamma, double* __restrict__ cval, double* __restrict__ cnorm,
          void* __restrict__ lp, int lp_elt, bool awide, bool bwide, bool cwide) {
  __shared__ double part[2][W];
  const int bsz = bs * bs;
  int par = 0;
  for (int64_t p = blockIdx.x; p < cnnz; p += gridDim.x, par ^= 1) {
    const int I = crow[p], J = cci[p];
    const int qa = find_warp(aci, arp[I], arp[I + 1], J);
    const int qb = bval ? find_warp(bci, brp[I], brp[I + 1], J) : -1;
    const double* a = aval + (size_t)(qa < 0 ? 0 : qa) * bsz;
    const TB* b = bval + (size_t)(qb < 0 ? 0 : (bmap ? bmap[qb] : qb)) * bsz;
    double* c = cval + (size_t)p * bsz;
    const bool dblk = I == J && gamma != 0.0;
    ifac::tc::SqAcc4 sq;
#pragma unroll 2
    for (int e = (int)threadIdx.x * 4; e < bsz; e += 128 * W) {
      double v[4] = {0.0, 0.0, 0.0, 0.0}, t[4];
      if (qa >= 0) load4(a + e, v, awide);
      if (qb >= 0) load4(b + e, t, bwide);
      if (qa >= 0) scale4(sa, v);
      if (qb >= 0) {
        scale4(sb, t);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = qa >= 0 ? __dadd_rn(v[i], t[i]) : t[i];
      }
      if (dblk) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if ((e + i) / bs == (e + i) % bs) v[i] = (qa >= 0 || qb >= 0) ? __dadd_rn(v[i], gamma) : gamma;
      }
      ifac::tc::store4(c + e, v, cwide);
      if (lp_elt) lp_store4(lp, lp_elt, (size_t)p * bsz + e, v);
      sq.add4(v);
    }
    block_norm<W>(sq, part[par], cnorm + p);
  }
}

// the same for block sizes whose square is no multiple of four: one warp per
// block, element by element
__global__ void k_add_odd(const int32_t* __restrict__ crow, const int32_t* __restrict__ cci, int64_t cnnz, int bs,
                          Scale sa, const int32_t* __restrict__ arp, const int32_t* __restrict__ aci,
                          const double* __restrict__ aval, Scale sb, const int32_t* __restrict__ brp,
                          const int32_t* __restrict__ bci, const double* __restrict__ bval,
                          const int32_t* __restrict__ bmap, double gamma, double* __restrict__ cval,
                          double* __restrict__ cnorm) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int bsz = bs * bs;
  for (int64_t p = w0; p < cnnz; p += nw) {
    const int I = crow[p], J = cci[p];
    const int qa = find_warp(aci, arp[I], arp[I + 1], J);
    const int qb = bval ? find_warp(bci, brp[I], brp[I + 1], J) : -1;
    const double* a = qa >= 0 ? aval + (size_t)qa * bsz : nullptr;
    const double* b = qb >= 0 ? bval + (size_t)(bmap ? bmap[qb] : qb) * bsz : nullptr;
    const bool dblk = I == J && gamma != 0.0;
    SqAcc sq;
    for (int e = lane; e < bsz; e += 32) {
      const double v = add_elem(sa, a, sb, b, dblk && e / bs == e % bs, gamma, e);
      cval[(size_t)p * bsz + e] = v;
      sq.add_f64(v);
    }
    const double ss = sq.warp_total();
    if (lane == 0) cnorm[p] = sqrt(ss);
  }
}

template <int W, typename TB>
static void launch_add(ifac_ctx* ctx, Scale sa, const ifac_bsr& A, Scale sb, const ifac_bsr* B, double gamma,
                       ifac_bsr& C, const int32_t* crow, const int32_t* bmap, void* lp, int lp_elt) {
  const int grid = (int)std::min<int64_t>(C.nnzb, 152 * 64 / W);
  k_add<W, TB><<<grid, 32 * W, 0, ctx->stream>>>(
      crow, C.col_idx, C.nnzb, C.bs, sa, A.row_ptr, A.col_idx, A.val, sb, B ? B->row_ptr : nullptr,
      B ? B->col_idx : nullptr, B ? reinterpret_cast<const TB*>(B->val) : nullptr, bmap, gamma, C.val, C.norms, lp,
      lp_elt, aligned32(A.val), B && aligned32(B->val), aligned32(C.val));
}

void add_numeric(ifac_ctx* ctx, double alpha, const ifac_bsr& A, double beta, const ifac_bsr* B, double gamma,
                 ifac_bsr& C, const int32_t* crow, const int32_t* bmap, void* lp, int lp_elt, bool b32) {
  const int bsz = C.bs * C.bs;
  if (lp_elt && bsz % 4 != 0) fail(IFAC_ERR_UNSUPPORTED, "low-precision copy: even block size");
  if (b32 && B && bsz % 4 != 0) fail(IFAC_ERR_UNSUPPORTED, "FP32 operand values: even block size");
  if (C.nnzb == 0) return;
  const Scale sa = make_scale(alpha), sb = make_scale(beta);
  if (bsz % 4 != 0) {
    const int64_t warps = std::min<int64_t>(C.nnzb, 152 * 64);
    k_add_odd<<<cdiv(warps * 32, 256), 256, 0, ctx->stream>>>(
        crow, C.col_idx, C.nnzb, C.bs, sa, A.row_ptr, A.col_idx, A.val, sb, B ? B->row_ptr : nullptr,
        B ? B->col_idx : nullptr, B ? B->val : nullptr, bmap, gamma, C.val, C.norms);
  } else if (b32 && B) {  // bs 32, 64 or 128
    if (bsz >= 4096) launch_add<8, float>(ctx, sa, A, sb, B, gamma, C, crow, bmap, lp, lp_elt);
    else launch_add<4, float>(ctx, sa, A, sb, B, gamma, C, crow, bmap, lp, lp_elt);
  } else if (bsz >= 4096) {  // eight warps with 16 values a thread or more, four with eight, one below
    launch_add<8, double>(ctx, sa, A, sb, B, gamma, C, crow, bmap, lp, lp_elt);
  } else if (bsz >= 1024) {
    launch_add<4, double>(ctx, sa, A, sb, B, gamma, C, crow, bmap, lp, lp_elt);
  } else {
    launch_add<1, double>(ctx, sa, A, sb, B, gamma, C, crow, bmap, lp, lp_elt);
  }
  IFAC_CK_LAUNCH();
}

// C = alpha (U + strict_upper(U)^T) + beta B + gamma I, one CTA per output
// block.  Block (I, J), J >= I, is add_elem of alpha U_IJ and beta B_IJ;
// block (I, J), J < I, takes alpha U_JI^T in place of alpha U_IJ, moved
// through shared memory as one 64 x 64 tile, so that U is read in whole rows
// (stripes of four output rows per warp read half sectors of FP32 values).
// bs = 64.  U's values are FP64 or FP32 (TU).  delta of the 262,144-row chain
// with its TF32 copy: 354 -> 198 us from FP32 values, 262 -> 150 us from FP64.
constexpr int SYM_WARPS = 8;

template <typename TU>
__global__ void __launch_bounds__(32 * SYM_WARPS)
    k_sym(const int32_t* __restrict__ crow, const int32_t* __restrict__ cci, int64_t cnnz, Scale sa,
          const int32_t* __restrict__ urp, const int32_t* __restrict__ uci, const TU* __restrict__ uval,
          const int32_t* __restrict__ umap, Scale sb,
          const int32_t* __restrict__ brp, const int32_t* __restrict__ bci, const double* __restrict__ bval,
          double gamma, double* __restrict__ cval, double* __restrict__ cnorm, int mirror, void* __restrict__ lp,
          int lp_elt, bool uwide, bool bwide, bool cwide) {
  constexpr int BS = 64, BSZ = BS * BS, STEP = 128 * SYM_WARPS;
  __shared__ TU tile[BS][BS + 1];
  __shared__ double part[2][SYM_WARPS];
  int par = 0;
  for (int64_t p = blockIdx.x; p < cnnz; p += gridDim.x, par ^= 1) {
    const int I = crow[p], J = cci[p];
    const bool lower = J < I;
    const int r = lower ? J : I, c = lower ? I : J;
    const int qu = find_warp(uci, urp[r], urp[r + 1], c);
    const int qb = bval ? find_warp(bci, brp[I], brp[I + 1], J) : -1;
    const TU* u = uval + (size_t)(qu < 0 ? 0 : (umap ? umap[qu] : qu)) * BSZ;
    const double* b = bval + (size_t)(qb < 0 ? 0 : qb) * BSZ;
    const bool dblk = I == J && gamma != 0.0;
    // mirror: a diagonal block takes its strictly lower triangle from its
    // upper one as well, so the result is exactly symmetric
    const bool moved = qu >= 0 && (lower || (mirror && I == J));  // CTA-uniform
    if (moved) {
#pragma unroll
      for (int e = (int)threadIdx.x; e < BSZ; e += 32 * SYM_WARPS) tile[e / BS][e % BS] = u[e];
      __syncthreads();
    }
    ifac::tc::SqAcc4 sq;
#pragma unroll 2
    for (int e = (int)threadIdx.x * 4; e < BSZ; e += STEP) {
      const int rr = e / BS, c0 = e % BS;
      double v[4] = {0.0, 0.0, 0.0, 0.0}, t[4];
      if (moved) {
        TU w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = (lower || c0 + i < rr) ? tile[c0 + i][rr] : tile[rr][c0 + i];
        widen4(w, v);
      } else if (qu >= 0) {
        load4(u + e, v, uwide);
      }
      if (qb >= 0) load4(b + e, t, bwide);
      if (qu >= 0) scale4(sa, v);
      if (qb >= 0) {
        scale4(sb, t);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = qu >= 0 ? __dadd_rn(v[i], t[i]) : t[i];
      }
      if (dblk) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (rr == c0 + i) v[i] = (qu >= 0 || qb >= 0) ? __dadd_rn(v[i], gamma) : gamma;
      }
      ifac::tc::store4(cval + (size_t)p * BSZ + e, v, cwide);
      if (lp_elt) lp_store4(lp, lp_elt, (size_t)p * BSZ + e, v);
      sq.add4(v);
    }
    // (the barrier inside also keeps the tile until every warp has read it)
    block_norm<SYM_WARPS>(sq, part[par], cnorm + p);
  }
}

template <typename TU>
static void launch_sym(ifac_ctx* ctx, double alpha, const ifac_bsr& U, double beta, const ifac_bsr* B, double gamma,
                       ifac_bsr& C, const int32_t* crow, const int32_t* umap, bool mirror, void* lp, int lp_elt) {
  const int grid = (int)std::min<int64_t>(C.nnzb, 152 * 64 / SYM_WARPS);
  k_sym<TU><<<grid, 32 * SYM_WARPS, 0, ctx->stream>>>(
      crow, C.col_idx, C.nnzb, make_scale(alpha), U.row_ptr, U.col_idx, reinterpret_cast<const TU*>(U.val), umap,
      make_scale(beta), B ? B->row_ptr : nullptr, B ? B->col_idx : nullptr, B ? B->val : nullptr, gamma, C.val,
      C.norms, mirror ? 1 : 0, lp, lp_elt, aligned32(U.val), B && aligned32(B->val), aligned32(C.val));
}

void sym_numeric(ifac_ctx* ctx, double alpha, const ifac_bsr& U, double beta, const ifac_bsr* B, double gamma,
                 ifac_bsr& C, const int32_t* crow, const int32_t* umap, bool mirror, void* lp, int lp_elt, bool u32) {
  if (C.nnzb == 0) return;
  if (U.bs != 64) fail(IFAC_ERR_UNSUPPORTED, "symmetric completion needs bs = 64");
  if (u32) launch_sym<float>(ctx, alpha, U, beta, B, gamma, C, crow, umap, mirror, lp, lp_elt);
  else launch_sym<double>(ctx, alpha, U, beta, B, gamma, C, crow, umap, mirror, lp, lp_elt);
  IFAC_CK_LAUNCH();
}

__global__ void k_block_norms(const double* __restrict__ val, int64_t nnzb, int bsz, double* __restrict__ norms) {
  __shared__ double red[32];
  for (int64_t p = blockIdx.x; p < nnzb; p += gridDim.x) {
    const double* v = val + (size_t)p * bsz;
    double ss = 0.0;
    for (int e = threadIdx.x; e < bsz; e += blockDim.x) ss = fma(v[e], v[e], ss);
    double t = block_reduce_sum(ss, red);
    if (threadIdx.x == 0) norms[p] = sqrt(t);
  }
}

void block_norms(ifac_ctx* ctx, const ifac_bsr& A, double* norms) {
  if (A.nnzb == 0) return;
  int grid = (int)std::min<int64_t>(A.nnzb, 152 * 16);
  k_block_norms<<<grid, 256, 0, ctx->stream>>>(A.val, A.nnzb, A.bs * A.bs, norms);
  IFAC_CK_LAUNCH();
}

// rowsq[I] = sum over the blocks of block row I of norm^2 (warp per row)
__global__ void k_row_sq(const int32_t* __restrict__ rp, int nb, const double* __restrict__ norms,
                         double* __restrict__ rowsq) {
  int row = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (row >= nb) return;
  double s = 0.0;
  for (int p = rp[row] + lane; p < rp[row + 1]; p += 32) s = fma(norms[p], norms[p], s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) rowsq[row] = s;
}

void row_sq_norms(ifac_ctx* ctx, const ifac_bsr& A, double* rowsq) {
  Buf<double> tmp;
  const double* norms = A.norms;
  if (!norms) {
    tmp = Buf<double>(ctx, A.nnzb);
    block_norms(ctx, A, tmp.p);
    norms = tmp.p;
  }
  k_row_sq<<<cdiv((int64_t)A.nb * 32, 256), 256, 0, ctx->stream>>>(A.row_ptr, A.nb, norms, rowsq);
  IFAC_CK_LAUNCH();
}

// out = sum of x[0..n) in a fixed order (single CTA)
__global__ void k_sum(const double* __restrict__ x, int n, double* __restrict__ out) {
  __shared__ double red[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
  double t = block_reduce_sum(s, red);
  if (threadIdx.x == 0) *out = t;
}

double fro_host(ifac_ctx* ctx, const ifac_bsr& A) {
  Buf<double> rowsq(ctx, A.nb), out(ctx, 1);
  row_sq_norms(ctx, A, rowsq.p);
  k_sum<<<1, 1024, 0, ctx->stream>>>(rowsq.p, A.nb, out.p);
  IFAC_CK_LAUNCH();
  double h = 0.0;
  to_host(ctx, &h, out.p, sizeof(double));
  return sqrt(h);
}

// row sums of |a_ij| for every scalar row (warp per scalar row), then max
__global__ void k_abs_rowsum(const int32_t* __restrict__ rp, int nb, int bs, const double* __restrict__ val,
                             double* __restrict__ rs) {
  int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (w >= (int64_t)nb * bs) return;
  int I = (int)(w / bs), r = (int)(w % bs);
  double s = 0.0;
  for (int p = rp[I]; p < rp[I + 1]; ++p) {
    const double* row = val + (size_t)p * bs * bs + (size_t)r * bs;
    for (int c = lane; c < bs; c += 32) s += fabs(row[c]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) rs[w] = s;
}

__global__ void k_max(const double* __restrict__ x, int64_t n, double* __restrict__ out) {
  __shared__ double red[32];
  double m = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, x[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t = fmax(t, red[i]);
    *out = t;
  }
}

void gershgorin_rows(ifac_ctx* ctx, const ifac_bsr& A, double* rs) {
  const int64_t rows = (int64_t)A.nb * A.bs;
  k_abs_rowsum<<<cdiv(rows * 32, 256), 256, 0, ctx->stream>>>(A.row_ptr, A.nb, A.bs, A.val, rs);
  IFAC_CK_LAUNCH();
}

double gershgorin_host(ifac_ctx* ctx, const ifac_bsr& A) {
  int64_t rows = (int64_t)A.nb * A.bs;
  Buf<double> rs(ctx, rows), out(ctx, 1);
  k_abs_rowsum<<<cdiv(rows * 32, 256), 256, 0, ctx->stream>>>(A.row_ptr, A.nb, A.bs, A.val, rs.p);
  IFAC_CK_LAUNCH();
  k_max<<<1, 1024, 0, ctx->stream>>>(rs.p, rows, out.p);
  IFAC_CK_LAUNCH();
  double h = 0.0;
  to_host(ctx, &h, out.p, sizeof(double));
  return h;
}

__global__ void k_scaled_identity(int nb, int bs, double c, int32_t* __restrict__ rp, int32_t* __restrict__ ci,
                                  double* __restrict__ val) {
  int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int64_t bsz = (int64_t)bs * bs;
  if (e < (int64_t)nb * bsz) {
    int64_t k = e % bsz;
    val[e] = ((k / bs) == (k % bs)) ? c : 0.0;
  }
  if (e < nb) ci[e] = (int32_t)e;
  if (e <= nb) rp[e] = (int32_t)e;
}

Mat scaled_identity(ifac_ctx* ctx, int64_t n, int bs, int nb, double c) {
  Mat M = mat_alloc(ctx, n, bs, nb, nb);
  int64_t tot = std::max<int64_t>((int64_t)nb * bs * bs, nb + 1);
  k_scaled_identity<<<cdiv(tot, 256), 256, 0, ctx->stream>>>(nb, bs, c, M.m.row_ptr, M.m.col_idx, M.m.val);
  IFAC_CK_LAUNCH();
  block_norms(ctx, M.m, M.m.norms);
  return M;
}

}  // namespace ifac
