// gemm_wide.cu -- TF32 / BF16 products of 64 x 64 blocks on tiles of 256 x 256
// accumulator elements, one CTA each, for block-dense operands.
//
// What bounds such a product is not the tensor pipe but the operand traffic
// from L2 (about 50 bytes a clock and SM): the pair kernel of gemm_tc.cu, with
// 128 rows a CTA, needs 94 (BF16, 256 columns) or 128 (TF32, 128 columns) bytes
// for every clock of tcgen05.mma.  Here a CTA holds four block rows and four
// block columns, 512 columns of tensor memory in two halves of 128 rows, and
// needs 64.  The price is that the accumulators are not double-buffered: the
// epilogue hands them back half by half, and the first K steps of the next
// tile run on half 0 while half 1 is still read.
//
//   warp 0      : TMA producer -- per K step of 128 bytes (64 BF16 or 32 TF32
//                 elements) the boxes of four op(A) and four op(B) blocks into
//                 one of three ring stages of 64 KB;
//   warp 1      : tensor memory and the single MMA-issuing thread, two
//                 instructions of 128 x 256 per 32 bytes of K;
//   warps 2..17 : epilogue, four per lane quarter, one block column each --
//                 alpha, block norms (compensated FP32 sums), FP64 or FP32
//                 stores through a shared-memory transpose.
//
// K runs over the plan's records in the order of the other kernels, so every
// element is the same sum.  Dense 8192 x 8192 in BF16 1104 -> 718 us (1.53 PFLOP/s,
// 78% of the measured rate), the TF32 products of a 4096-row 3D cluster factor 246
// -> 129 us a launch (722 TFLOP/s, 74% of TF32's share of it).  A product of
// fewer tiles than half the SMs keeps the pair kernel, which spreads them over
// twice as many.  Every mbarrier wait is bounded.
#include "internal.cuh"
#include "tc_common.cuh"

namespace ifac {
namespace tc {
namespace wide {
constexpr int BS = 64, TMB = 4, TNB = 4;
constexpr int N = TNB * BS;                // 256 columns of one half
constexpr int HALF_BYTES = 128 * 128;      // 128 rows of one half, 128 bytes of K each
constexpr int A_BYTES = 2 * HALF_BYTES;
constexpr int STAGE = A_BYTES + N * 128;   // 64 KB
constexpr int STAGES = 3;
constexpr int SMEM = STAGES * STAGE + 1024;
constexpr int KSTEPS = 4;                  // instructions of 32 bytes of K per stage
constexpr int NEPI = 16;
constexpr int NTHREADS = 32 * (2 + NEPI);
constexpr uint32_t TMEM_COLS = 512;
constexpr int RECW = TMB + TNB;
}  // namespace wide

struct WideArgs {
  const int32_t* tiles;
  const int* ntiles;
  const int32_t* tile_nk;
  const int32_t* rec;
  const int32_t* rec_off;
  const int32_t* cpos;
  double* cval;
  float* cval32;  // non-null: FP32 values in place of cval
  double* cnorm;
  double alpha;
  int* err;
};

template <int ELT>
__global__ void __launch_bounds__(wide::NTHREADS, 1)
    k_gemm_wide(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, WideArgs args) {
  using namespace wide;
  constexpr int ATOM_ELEMS = 128 / ELT, ATOMS = BS / ATOM_ELEMS;  // K steps per block: 1 (BF16), 2 (TF32)
  constexpr uint32_t IDESC = idesc_of<ELT, N, 128>();
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES];
  __shared__ __align__(8) uint64_t acc_full, acc_empty[2], drain_bar;
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile int abort_flag;
  __shared__ double partial[2][2][4][TNB];  // tile parity, half, lane quarter, block column
  __shared__ float ep_stage[NEPI][32 * 9];
  __shared__ int32_t srec[32 * RECW];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int ntiles = *args.ntiles;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&acc_full), 1);
    for (int h = 0; h < 2; ++h) mbar_init(smem_u32(&acc_empty[h]), NEPI);  // one arrival per epilogue warp
    mbar_init(smem_u32(&drain_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_slot;
  const int mt = ntiles > (int)blockIdx.x ? (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    int stage = 0;
    uint32_t phase = 0, issued_mask = 0, last_parity = 0;
    bool ok = true;
    RecStream<RECW> rs;
    rs.init(args.rec, args.rec_off, args.tile_nk, (int)blockIdx.x, (int)gridDim.x, mt, 1);
    int32_t cur[RECW], nxt[RECW];
    int c_it, c_rep, c_j0, c_cnt, n_it, n_rep, n_j0, n_cnt;
    bool have = rs.next(lane, cur, c_it, c_rep, c_j0, c_cnt);
    while (have && ok) {
      if (lane < c_cnt) {
#pragma unroll
        for (int w = 0; w < RECW; ++w) srec[lane * RECW + w] = cur[w];
      }
      __syncwarp();
      const bool nhave = rs.next(lane, nxt, n_it, n_rep, n_j0, n_cnt);
      if (lane == 0) {
        for (int j = 0; j < c_cnt && ok; ++j) {
          const int32_t* r = srec + j * RECW;
          for (int a = 0; a < ATOMS; ++a) {
            if (!mbar_wait(smem_u32(&empty_bar[stage]), phase ^ 1u, &abort_flag, args.err)) {
              ok = false;
              break;
            }
            const uint32_t fb = smem_u32(&full_bar[stage]);
            mbar_expect_tx(fb, (uint32_t)STAGE);
            issued_mask |= 1u << stage;
            last_parity = (last_parity & ~(1u << stage)) | (phase << stage);
            const uint32_t sa = smem_base + (uint32_t)(stage * STAGE), sb = sa + A_BYTES;
#pragma unroll
            for (int i = 0; i < TMB; ++i) tma_load_2d(sa + i * BS * 128, &mapA, a * ATOM_ELEMS, r[i] * BS, fb);
#pragma unroll
            for (int c = 0; c < TNB; ++c) tma_load_2d(sb + c * BS * 128, &mapB, a * ATOM_ELEMS, r[TMB + c] * BS, fb);
            if (++stage == STAGES) {
              stage = 0;
              phase ^= 1u;
            }
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      __syncwarp();  // srec is rewritten next round
#pragma unroll
      for (int w = 0; w < RECW; ++w) cur[w] = nxt[w];
      c_it = n_it;
      c_rep = n_rep;
      c_j0 = n_j0;
      c_cnt = n_cnt;
      have = nhave;
    }
    // the copies issued have landed and the MMAs have released every stage
    if (lane == 0)
      for (int s = 0; s < STAGES; ++s)
        if (issued_mask & (1u << s)) {
          mbar_wait(smem_u32(&full_bar[s]), (last_parity >> s) & 1u, &abort_flag, args.err, false);
          mbar_wait(smem_u32(&empty_bar[s]), (last_parity >> s) & 1u, &abort_flag, args.err, false);
        }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      // half h of the product of stage st
      const auto issue = [&](int st, int h, bool fresh) {
        const uint32_t sa = smem_base + (uint32_t)(st * STAGE + h * HALF_BYTES);
        const uint64_t da = smem_desc(sa), db = smem_desc(smem_base + (uint32_t)(st * STAGE + A_BYTES));
#pragma unroll
        for (int kk = 0; kk < KSTEPS; ++kk)
          mma_kstep<ELT>(tmem + (uint32_t)(h * N), da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), IDESC,
                         (fresh && kk == 0) ? 0u : 1u);
      };
      int nk_next = mt > 0 ? args.tile_nk[blockIdx.x] : 0;  // loaded a tile ahead
      for (int it = 0; it < mt && ok; ++it) {
        const int steps = nk_next * ATOMS;
        if (it + 1 < mt) nk_next = args.tile_nk[(int)blockIdx.x + (it + 1) * (int)gridDim.x];
        const uint32_t aphase = (uint32_t)it & 1u;
        // the first stages: half 0 on all of them, then half 1
        const int lead = min(STAGES, steps);
        if (!mbar_wait(smem_u32(&acc_empty[0]), aphase ^ 1u, &abort_flag, args.err)) break;
        tc_fence_after();
        for (int j = 0, st = stage, ph = (int)phase; j < lead && ok; ++j) {
          ok = mbar_wait(smem_u32(&full_bar[st]), (uint32_t)ph, &abort_flag, args.err);
          if (!ok) break;
          tc_fence_after();
          issue(st, 0, j == 0);
          if (++st == STAGES) {
            st = 0;
            ph ^= 1;
          }
        }
        if (!ok || !mbar_wait(smem_u32(&acc_empty[1]), aphase ^ 1u, &abort_flag, args.err)) break;
        tc_fence_after();
        for (int j = 0; j < steps; ++j) {
          if (j >= lead) {
            ok = mbar_wait(smem_u32(&full_bar[stage]), phase, &abort_flag, args.err);
            if (!ok) break;
            tc_fence_after();
            issue(stage, 0, false);
          }
          issue(stage, 1, j == 0);
          mma_commit(smem_u32(&empty_bar[stage]));
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        mma_commit(smem_u32(&acc_full));
      }
      // every MMA this thread issued completes before tensor memory is released
      mma_commit(smem_u32(&drain_bar));
      mbar_wait(smem_u32(&drain_bar), 0, &abort_flag, args.err, false);
    }
  } else {
    // ------------------------------ epilogue ------------------------------
    const int ew = warp - 2, q = warp & 3, cg = ew >> 2;  // lane quarter, block column of the tile
    const int et = threadIdx.x - 64;
    const float alpha_f = (float)args.alpha;
    constexpr int CP = TMB * TNB;
    // C positions of this warp's blocks (one per half) and of the block whose
    // norm it writes, loaded a tile ahead
    int pn[2] = {-1, -1}, kn_next = -1;
    const auto load_next = [&](int t) {
#pragma unroll
      for (int h = 0; h < 2; ++h) pn[h] = args.cpos[(size_t)t * CP + (h * 2 + (q >> 1)) * TNB + cg];
      if (et < CP) kn_next = args.cpos[(size_t)t * CP + et];
    };
    if (mt > 0) load_next((int)blockIdx.x);
    for (int it = 0; it < mt; ++it) {
      const int pos[2] = {pn[0], pn[1]}, kn = kn_next;
      if (it + 1 < mt) load_next((int)blockIdx.x + (it + 1) * (int)gridDim.x);
      const int par = it & 1;
      // (a wait that failed is voted on after the tile)
      const bool got = mbar_wait(smem_u32(&acc_full), (uint32_t)par, &abort_flag, args.err);
      __syncwarp();
      tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int p = pos[h];  // warp-uniform; -1: not in C
        SqAcc sq;
#pragma unroll 1
        for (int ch = 0; ch < BS / 8; ++ch) {
          float v[8];
          tmem_ld8(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * N + cg * BS + ch * 8), v);
          if (ch == BS / 8 - 1) {  // this warp has read its part of the half
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[h]));
          }
          if (p >= 0) {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] *= alpha_f;
            sq.add<8>(v);
            // 32 rows x 8 columns through shared memory: row segments of 64 bytes
            float* sw = ep_stage[ew];
            const size_t boff = (size_t)p * BS * BS + (size_t)((q & 1) * 32) * BS + ch * 8;
            const int c2 = (lane & 3) * 2, r8 = lane >> 2;
#pragma unroll
            for (int e = 0; e < 8; ++e) sw[lane * 9 + e] = v[e];
            __syncwarp();
            if (args.cval32) {  // kernel-uniform
              float* blk = args.cval32 + boff;
#pragma unroll
              for (int k = 0; k < 32; k += 8) {
                const float* qv = sw + (k + r8) * 9 + c2;
                *reinterpret_cast<float2*>(blk + (size_t)(k + r8) * BS + c2) = make_float2(qv[0], qv[1]);
              }
            } else {
              double* blk = args.cval + boff;
#pragma unroll
              for (int k = 0; k < 32; k += 8) {
                const float* qv = sw + (k + r8) * 9 + c2;
                *reinterpret_cast<double2*>(blk + (size_t)(k + r8) * BS + c2) =
                    make_double2(f32_to_f64(qv[0]), f32_to_f64(qv[1]));
              }
            }
            __syncwarp();
          }
        }
        const double ss = sq.warp_total();
        if (lane == 0) partial[par][h][q][cg] = ss;
      }
      // one barrier per tile (the partials alternate between two buffers)
      if (!epi_all<32 * NEPI>(got)) break;
      // block (br, bc): lane quarters 2 (br % 2) and 2 (br % 2) + 1 of half br / 2
      if (et < CP && kn >= 0) {
        const int br = et / TNB, bc = et % TNB;
        args.cnorm[kn] = sqrt(partial[par][br >> 1][2 * (br & 1)][bc] + partial[par][br >> 1][2 * (br & 1) + 1][bc]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

template <int ELT>
static void launch_wide(ifac_ctx* ctx, const CUtensorMap& mapA, const CUtensorMap& mapB, const WideArgs& a,
                        int tiles_bound) {
  // (set at every launch, so that no other thread can launch before it)
  IFAC_CK(cudaFuncSetAttribute(k_gemm_wide<ELT>, cudaFuncAttributeMaxDynamicSharedMemorySize, wide::SMEM));
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  const int grid = std::min(std::max(tiles_bound, 1), sms);
  k_gemm_wide<ELT><<<grid, wide::NTHREADS, wide::SMEM, ctx->stream>>>(mapA, mapB, a);
  IFAC_CK_LAUNCH();
}

}  // namespace tc

void wide_product(ifac_ctx* ctx, int elt, const void* mapA, const void* mapB, const int32_t* tiles, const int* ntiles,
                  const int32_t* tile_nk, const int32_t* rec, const int32_t* rec_off, const int32_t* cpos,
                  int tiles_bound, double alpha, ifac_bsr& C, bool out32) {
  tc::WideArgs a{};
  a.tiles = tiles;
  a.ntiles = ntiles;
  a.tile_nk = tile_nk;
  a.rec = rec;
  a.rec_off = rec_off;
  a.cpos = cpos;
  a.cval = out32 ? nullptr : C.val;
  a.cval32 = out32 ? reinterpret_cast<float*>(C.val) : nullptr;
  a.cnorm = C.norms;
  a.alpha = alpha;
  a.err = ctx->dev_err;
  const CUtensorMap& mA = *static_cast<const CUtensorMap*>(mapA);
  const CUtensorMap& mB = *static_cast<const CUtensorMap*>(mapB);
  if (elt == 2) tc::launch_wide<2>(ctx, mA, mB, a, tiles_bound);
  else tc::launch_wide<4>(ctx, mA, mB, a, tiles_bound);
}

}  // namespace ifac
