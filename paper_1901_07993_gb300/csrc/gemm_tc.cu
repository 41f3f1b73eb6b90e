// gemm_tc.cu -- tensor-core numeric phase of C = alpha op(A) op(B) for
// 64 x 64 blocks, with BF16 or TF32 inputs and FP32 accumulation in tensor
// memory (the low-precision products of the mixed-precision schedule).
//
// Operands.  op(A) and op(B) are first copied in their own CSR order to a
// low-precision array, each block stored K-major (op(A)_IK as [i][k],
// op(B)_KJ as [j][k]), so that a transposed use of an FP64 matrix costs only
// a transposed copy; one all-zero block is appended to each copy.
//
// Tiles.  The output is cut into tiles of TM x TN blocks (M = 128 rows, N =
// 256 (BF16) or 128 (TF32) columns); only tiles that hold a block of C's
// pattern are visited, by a persistent grid.  For a tile, K runs over the
// union of the stored K's of its TM op(A) block rows; a block missing inside
// the tile (op(A)_IK or op(B)_KJ not stored) is read from the zero block, so
// every K step is one dense M x N x 64 contraction.
//
// Pairs.  Two CTAs take one super-tile of 2 TM x TN blocks: each computes
// TM block rows against the same op(B) panel and walks the same K set (the
// union over the super-tile's rows), so the panel is read from HBM once and
// from L2 by the second CTA.  Each CTA loads its own copy of every tile it
// contracts (no cluster, no cross-CTA signalling).
//
// Products with enough 256 x 256 tiles for half the SMs run in gemm_wide.cu
// instead, banded ones in gemm_band.cu; run() decides.
//
// Roles (320 threads, one CTA per SM):
//   warp 0      : TMA producer -- one 64-row box per block and 128-byte
//                 atom, 128-byte swizzle, into a STAGES-deep ring;
//   warp 1      : tensor-memory allocation and the single MMA-issuing
//                 thread (tcgen05.mma, accumulate in TMEM, tcgen05.commit
//                 releases ring slots and hands the accumulator over);
//   warps 2..9  : epilogue, two warps per tensor-memory lane quarter, each
//                 on half of the tile's column blocks -- tcgen05.ld of the
//                 accumulator, alpha, Frobenius norm per output block, FP64
//                 store into C.
// Every mbarrier wait is bounded; on expiry the CTA records an error flag,
// drains its own copies and MMAs, releases tensor memory and returns.
#include <cuda.h>
#include <climits>
#include <type_traits>
#include <cuda_bf16.h>

#include "internal.cuh"
#include "scan_tail.cuh"
#include "tc_common.cuh"

namespace ifac {
namespace tc {

constexpr int BS = 64;
constexpr int TM = 2;
constexpr int PAIR = 2;                    // CTAs per super-tile (consecutive blockIdx.x)
constexpr int NEPI = 8;                    // epilogue warps: two per tensor-memory lane quarter
constexpr int NTHREADS = 64 + 32 * NEPI;
// split mode: K steps per exact FP32 window, table sizes
constexpr int KW = 16;
constexpr int MAX_UNITS = 16;
constexpr int MAX_PAIRS = 40;

template <int ELT>
struct Cfg {
  static constexpr int ATOM_ELEMS = 128 / ELT;          // elements in one 128-byte row
  static constexpr int ATOMS = BS / ATOM_ELEMS;         // 128-byte atoms along K per block
  static constexpr int MMA_K = 32 / ELT;                // 32 bytes of K per tcgen05.mma
  static constexpr int KSTEPS = BS / MMA_K;             // MMAs per K block
  static constexpr int TN = (ELT == 2) ? 4 : 2;         // block columns per tile
  static constexpr int N = TN * BS;
  static constexpr int M = TM * BS;
  static constexpr int A_ATOM_BYTES = M * 128;          // one K atom of the A tile
  static constexpr int B_ATOM_BYTES = N * 128;
  static constexpr int A_BYTES = ATOMS * A_ATOM_BYTES;
  static constexpr int B_BYTES = ATOMS * B_ATOM_BYTES;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = (ELT == 2) ? 4 : 3;
  static constexpr int TMEM_COLS = 2 * N;               // two FP32 accumulators (double buffer)
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024;
  static constexpr uint32_t TX_BYTES = (uint32_t)(TM + TN) * BS * BS * ELT;
};

template <int ELT>
__host__ __device__ constexpr uint32_t instr_desc() {
  return idesc_of<ELT, Cfg<ELT>::N, Cfg<ELT>::M>();
}

template <int ELT>
__device__ __forceinline__ void mma_issue(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  mma_kstep<ELT>(tmem_d, adesc, bdesc, instr_desc<ELT>(), accumulate);
}

__device__ __forceinline__ void epi_bar() { epi_bar<32 * NEPI>(); }

// ---------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------
struct TileArgs {
  const int32_t* tiles;      // [2*t] tile row, [2*t+1] tile column
  const int* ntiles;         // device: number of tiles
  const int* tile_nk;        // device: K steps of each tile
  int nwin;                  // split mode: the largest number of K windows of a tile
  int nb;
  const int32_t* rec;        // plan: per K step, copy indices of op(A)_IK (super-tile rows) and op(B)_KJ
  const int32_t* rec_off;    // first record of each tile
  const int32_t* crp;    // C pattern
  const int32_t* cci;
  double* cval;
  float* cval32;  // TF32/BF16 products: non-null, C's values as FP32 (the
                  // accumulators exactly, half the bytes of cval) in place of cval
  double* cnorm;
  // split mode: fixed-point sums, per C block 2048 longlong2 in hand-over
  // order ((row half, column half, pair e) x 32 lanes), so that a warp's
  // read-modify-write of one register pair covers 512 contiguous bytes
  longlong2* cpart;
  double alpha;
  int* err;
  // split mode (FP64-accurate products): the copies of op(A) and op(B) hold
  // NS BF16 slices each; pair p multiplies the slices starting at rows
  // pair_ya[p] / pair_yb[p] of the tensor maps; the pairs of unit u,
  // [unit_end[u-1], unit_end[u]), share one FP32 accumulator and its weight
  // weight 2^sh_u in the 64-bit fixed-point sums that the epilogue keeps in
  // C's value array (no norms; converted after the kernel)
  int split;
  int nunits;
  int unit_end[MAX_UNITS];
  int pair_ya[MAX_PAIRS], pair_yb[MAX_PAIRS];
  int unit_sh[MAX_UNITS];
  int* ovf;  // set to 2 on a fixed-point overflow (reported as an error by the host)
  // failure-path self-test only (0 in every product): the producer and the MMA
  // issuer do no work, so the epilogue's first accumulator wait expires after
  // wait_limit polls and the kernel reports a timeout
  int stall;
  long long wait_limit;
};

template <int ELT>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_gemm_tc(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, TileArgs args) {
  using C = Cfg<ELT>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[C::STAGES], empty_bar[C::STAGES];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], drain_bar;
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile int abort_flag;
  __shared__ double partial[4][C::TN];
  __shared__ int s_unit_end[MAX_UNITS], s_pair_ya[MAX_PAIRS], s_pair_yb[MAX_PAIRS];
  __shared__ int s_unit_sh[MAX_UNITS];
  __shared__ float ep_stage[NEPI][32 * 17];  // plain epilogue: per-warp transpose for coalesced stores

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long wl = args.wait_limit;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int ntiles = *args.ntiles;
  // CTAs 2c and 2c + 1 (pair c of ncl) take one super-tile of PAIR*TM x TN
  // blocks; CTA `crank` of the pair computes block rows (super row * PAIR +
  // crank) * TM.  Both step through the same K set (the union over the
  // super-tile's rows) and load the whole op(B) panel into their own shared
  // memory.
  const int crank = (int)(blockIdx.x % PAIR);
  const int cid = (int)(blockIdx.x / PAIR), ncl = (int)(gridDim.x / PAIR);

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int u = 0; u < MAX_UNITS; ++u) {
      s_unit_end[u] = args.unit_end[u];
      s_unit_sh[u] = args.unit_sh[u];
    }
    for (int p = 0; p < MAX_PAIRS; ++p) {
      s_pair_ya[p] = args.pair_ya[p];
      s_pair_yb[p] = args.pair_yb[p];
    }
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);  // released by this CTA's MMAs
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&acc_full[b]), 1);
      mbar_init(smem_u32(&acc_empty[b]), 1);
    }
    mbar_init(smem_u32(&drain_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"((uint32_t)C::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_slot;

  // work items: this pair's tiles (cid, cid + ncl, ...), in split mode once
  // per K window, window-major: every pair runs window w of its tiles before
  // window w + 1, so the slices of one K range are shared through L2, while a
  // tile's fixed-point sums are only ever updated by the one CTA that owns its rows
  const int mt = ntiles > cid ? (ntiles - cid + ncl - 1) / ncl : 0;
  const int nitems = mt * (args.split ? args.nwin : 1);
  auto item = [&](int j, int& t, int& kb, int& cnt) -> bool {
    t = cid + (j % mt) * ncl;
    const int nk = args.tile_nk[t];
    if (!args.split) {
      kb = 0;
      cnt = nk;
      return cnt > 0;
    }
    kb = (j / mt) * KW;
    if (kb >= nk) return false;
    cnt = min(KW, nk - kb);
    return true;
  };

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    // The warp reads the tile's K-step records from the plan 32 at a time,
    // lane-parallel; lane 0 then issues the loads of each record into the next
    // ring slot.  In split mode the records come in windows of KW, and every
    // window is loaded once per slice pair, unit by unit.
    __shared__ int rec[32][TM + Cfg<ELT>::TN];
    __shared__ int wrec[KW][TM + Cfg<ELT>::TN];
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued_mask = 0, last_parity = 0;  // lane 0: stages filled / parity of their last fill
    bool ok = true;
    // lane 0: one ring slot with the blocks of record r, slices at rows ya / yb
    auto issue = [&](const int* r, int ya, int yb) -> bool {
      if (!mbar_wait(smem_u32(&empty_bar[stage]), phase ^ 1u, &abort_flag, args.err, true, wl)) return false;
      const uint32_t fb = smem_u32(&full_bar[stage]);
      mbar_expect_tx(fb, C::TX_BYTES);
      issued_mask |= 1u << stage;
      last_parity = (last_parity & ~(1u << stage)) | (phase << stage);
      const uint32_t sa = smem_base + stage * C::STAGE_BYTES;
      const uint32_t sb = sa + C::A_BYTES;
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int a = 0; a < C::ATOMS; ++a)
          tma_load_2d(sa + a * C::A_ATOM_BYTES + i * BS * 128, &mapA, a * C::ATOM_ELEMS, ya + r[i] * BS, fb);
#pragma unroll
      for (int c = 0; c < C::TN; ++c)
#pragma unroll
        for (int a = 0; a < C::ATOMS; ++a)
          tma_load_2d(sb + a * C::B_ATOM_BYTES + c * BS * 128, &mapB, a * C::ATOM_ELEMS, yb + r[TM + c] * BS, fb);
      if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
      return true;
    };
    // lane 0, split mode: the cnt records of the open window for every slice pair
    auto issue_window = [&](int cnt) -> bool {
      int p = 0;
      for (int u = 0; u < args.nunits; ++u)
        for (; p < s_unit_end[u]; ++p)
          for (int j = 0; j < cnt; ++j)
            if (!issue(wrec[j], s_pair_ya[p], s_pair_yb[p])) return false;
      return true;
    };
    constexpr int RECW = PAIR * TM + C::TN;  // plan record: op(A) rows of the super-tile, then op(B) columns
    for (int it = 0; it < nitems && ok && !args.stall; ++it) {
      int t, kb, cnt;
      if (!item(it, t, kb, cnt)) continue;
      const int32_t* base = args.rec + (size_t)(args.rec_off[t] + kb) * RECW;
      if (!args.split) {
        for (int k0 = 0; k0 < cnt && ok; k0 += 32) {
          const int n = min(32, cnt - k0);
          if (lane < n) {
            const int32_t* r = base + (size_t)(k0 + lane) * RECW;
#pragma unroll
            for (int i = 0; i < TM; ++i) rec[lane][i] = r[crank * TM + i];
#pragma unroll
            for (int c = 0; c < C::TN; ++c) rec[lane][TM + c] = r[PAIR * TM + c];
          }
          __syncwarp();
          if (lane == 0)
            for (int j = 0; j < n && ok; ++j) ok = issue(rec[j], 0, 0);
          ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
          __syncwarp();
        }
      } else {
        if (lane < cnt) {
          const int32_t* r = base + (size_t)lane * RECW;
#pragma unroll
          for (int i = 0; i < TM; ++i) wrec[lane][i] = r[crank * TM + i];
#pragma unroll
          for (int c = 0; c < C::TN; ++c) wrec[lane][TM + c] = r[PAIR * TM + c];
        }
        __syncwarp();
        if (lane == 0) ok = issue_window(cnt);
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        __syncwarp();
      }
    }
    // before the CTA exits: the copies lane 0 issued have landed and the MMAs
    // have released every slot
    if (lane == 0)
      for (int s = 0; s < C::STAGES; ++s)
        if (issued_mask & (1u << s)) {
          mbar_wait(smem_u32(&full_bar[s]), (last_parity >> s) & 1u, &abort_flag, args.err, false, wl);
          mbar_wait(smem_u32(&empty_bar[s]), (last_parity >> s) & 1u, &abort_flag, args.err, false, wl);
        }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int tl = 0;  // accumulator hand-overs so far: buffer tl & 1, its phase (tl >> 1) & 1
      bool ok = true;
      // nsteps ring slots contracted into one accumulator, then handed to the epilogue
      auto run_acc = [&](int nsteps) -> bool {
        const int ab = tl & 1;
        const uint32_t aphase = (uint32_t)(tl >> 1) & 1u;
        const uint32_t tacc = tmem + (uint32_t)(ab * C::N);
        if (!mbar_wait(smem_u32(&acc_empty[ab]), aphase ^ 1u, &abort_flag, args.err, true, wl)) return false;
        tc_fence_after();
        for (int k = 0; k < nsteps; ++k) {
          if (!mbar_wait(smem_u32(&full_bar[stage]), phase, &abort_flag, args.err, true, wl)) return false;
          tc_fence_after();
          const uint32_t sa = smem_base + stage * C::STAGE_BYTES;
          const uint32_t sb = sa + C::A_BYTES;
#pragma unroll
          for (int kk = 0; kk < C::KSTEPS; ++kk) {
            const int atom = kk / (C::ATOM_ELEMS / C::MMA_K), off = (kk % (C::ATOM_ELEMS / C::MMA_K)) * 32;
            mma_issue<ELT>(tacc, smem_desc(sa + atom * C::A_ATOM_BYTES + off),
                           smem_desc(sb + atom * C::B_ATOM_BYTES + off), (k > 0 || kk > 0) ? 1u : 0u);
          }
          mma_commit(smem_u32(&empty_bar[stage]));
          if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
        }
        mma_commit(smem_u32(&acc_full[ab]));
        ++tl;
        return true;
      };
      for (int it = 0; it < nitems && ok && !args.stall; ++it) {
        int t, kb, cnt;
        if (!item(it, t, kb, cnt)) continue;  // (a tile holds a block of C's pattern, so nk >= 1)
        if (!args.split) {
          ok = run_acc(cnt);
        } else {
          int p = 0;
          for (int u = 0; u < args.nunits && ok; ++u) {
            ok = run_acc((s_unit_end[u] - p) * cnt);
            p = s_unit_end[u];
          }
        }
      }
      // every MMA this thread issued completes before tensor memory is released
      mma_commit(smem_u32(&drain_bar));
      mbar_wait(smem_u32(&drain_bar), 0, &abort_flag, args.err, false, wl);
    }
  } else {
    // ------------------------------ epilogue ------------------------------
    const int q = warp & 3;            // tensor-memory lane quarter of this warp
    const int c0 = ((warp - 2) >> 2) * (C::TN / 2), c1 = c0 + C::TN / 2;  // this warp's column blocks
    const int row = q * 32 + lane;     // accumulator row 0..127
    const int r_blk = row / BS;
    const int et = threadIdx.x - 64;   // 0 .. 32 NEPI - 1
    const float alpha_f = (float)args.alpha;
    int tl = 0;
    bool good = true;
    for (int it = 0; it < nitems && good; ++it) {
      int t, kb, cnt;
      if (!item(it, t, kb, cnt)) continue;
      const int I0 = (args.tiles[2 * t] * PAIR + crank) * TM, J0 = args.tiles[2 * t + 1] * C::TN;
      const int I = I0 + r_blk;  // warp-uniform: a warp's 32 rows lie in one block row
      int pc[C::TN];             // position of C_{I, J0+c} in C, or -1
#pragma unroll
      for (int c = 0; c < C::TN; ++c) {
        const int J = J0 + c;
        pc[c] = -1;
        if (I < args.nb && J < args.nb) {
          const int lo = args.crp[I], hi = args.crp[I + 1];
          const int k = lower_bound_i32(args.cci, lo, hi, J);
          if (k < hi && args.cci[k] == J) pc[c] = k;
        }
      }
      if (!args.split) {
        const int ab = tl & 1;
        const uint32_t aphase = (uint32_t)(tl >> 1) & 1u;
        ++tl;
        const bool got = mbar_wait(smem_u32(&acc_full[ab]), aphase, &abort_flag, args.err, true, wl);
        if (!epi_all<32 * NEPI>(got)) break;  // all epilogue warps go on, or all stop
        tc_fence_after();
#pragma unroll 1
        for (int c = c0; c < c1; ++c) {
          const int p = pc[c];
          SqAcc sq;  // this thread's 64 squares, accurate to about 2^-42 (FP32 pipe)
#pragma unroll
          for (int h = 0; h < BS / 32; ++h) {
            float v[32];
            tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * C::N + c * BS + h * 32), v);
            if (p >= 0) {  // warp-uniform
#pragma unroll
              for (int e = 0; e < 32; ++e) v[e] *= alpha_f;
              sq.add32(v);
              // 32 rows x 16 columns at a time through shared memory, so that
              // each store instruction writes two 128-byte row segments
              float* sw = ep_stage[warp - 2];
              const size_t boff = (size_t)p * BS * BS + (size_t)((q & 1) * 32) * BS + h * 32;
              const int cc = lane & 15, rr = lane >> 4;
#pragma unroll
              for (int half = 0; half < 2; ++half) {
#pragma unroll
                for (int e = 0; e < 16; ++e) sw[lane * 17 + e] = v[half * 16 + e];
                __syncwarp();
                if (args.cval32) {  // kernel-uniform
                  float* blk = args.cval32 + boff;
#pragma unroll 4
                  for (int k = 0; k < 32; k += 2) blk[(size_t)(k + rr) * BS + half * 16 + cc] = sw[(k + rr) * 17 + cc];
                } else {
                  double* blk = args.cval + boff;
#pragma unroll 4
                  for (int k = 0; k < 32; k += 2)
                    blk[(size_t)(k + rr) * BS + half * 16 + cc] = f32_to_f64(sw[(k + rr) * 17 + cc]);
                }
                __syncwarp();
              }
            }
          }
          const double ss = sq.warp_total();
          if (lane == 0) partial[q][c] = ss;
        }
        tc_fence_before();
        epi_bar();
        // norms: block row rb is covered by lane quarters 2rb and 2rb+1, summed in that order
        if (et < TM * C::TN) {
          const int rb = et / C::TN, c = et % C::TN;
          const int Ib = I0 + rb, J = J0 + c;
          if (Ib < args.nb && J < args.nb) {
            const int lo = args.crp[Ib], hi = args.crp[Ib + 1];
            const int k = lower_bound_i32(args.cci, lo, hi, J);
            if (k < hi && args.cci[k] == J) args.cnorm[k] = sqrt(partial[2 * rb][c] + partial[2 * rb + 1][c]);
          }
        }
        epi_bar();
        if (et == 0) mbar_arrive(smem_u32(&acc_empty[ab]));
      } else {
        // C_int += acc 2^sh_u, one hand-over per unit of this window; C is held
        // as 64-bit fixed point (scale 2^-f relative to sigma_i tau_j) until the
        // conversion after the kernel
        for (int u = 0; u < args.nunits; ++u) {
          const int ab = tl & 1;
          const uint32_t aphase = (uint32_t)(tl >> 1) & 1u;
          ++tl;
          const bool got = mbar_wait(smem_u32(&acc_full[ab]), aphase, &abort_flag, args.err, true, wl);
          if (!epi_all<32 * NEPI>(got)) { good = false; break; }
          tc_fence_after();
          const int sh = s_unit_sh[u];
#pragma unroll 1
          for (int c = c0; c < c1; ++c) {
            const int p = pc[c];
#pragma unroll
            for (int h = 0; h < BS / 32; ++h) {
              longlong2 dv[16];
              longlong2* dst = args.cpart + (size_t)(p < 0 ? 0 : p) * (BS * BS / 2) +
                               (size_t)(((q & 1) * 2 + h) * 16) * 32 + lane;
              if (p >= 0) {
#pragma unroll
                for (int e = 0; e < 16; ++e) dv[e] = dst[e * 32];
              }
              float v[32];
              tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * C::N + c * BS + h * 32), v);
              if (p >= 0) {
                bool bad = false;
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                  dv[e].x = fixed_add(dv[e].x, __float2int_rn(v[2 * e]), sh, bad);
                  dv[e].y = fixed_add(dv[e].y, __float2int_rn(v[2 * e + 1]), sh, bad);
                  dst[e * 32] = dv[e];
                }
                if (bad) *args.ovf = 2;
              }
            }
          }
          tc_fence_before();
          epi_bar();
          if (et == 0) mbar_arrive(smem_u32(&acc_empty[ab]));
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)C::TMEM_COLS));
  }
}

// ---------------------------------------------------------------------------
// operand conversion and tile list
// ---------------------------------------------------------------------------
// dst[q] = low-precision copy of block src[q] of X (B x B blocks; K-major:
// transposed when TR), one zero block appended.  X's values are FP64 (V =
// double) or the FP32 results of a TF32/BF16 product (V = float), rounded
// alike.  Bound by HBM: four values a thread and step, one vector load and one
// vector store; a transposed copy goes through shared memory in tiles of 64 x
// 64 whose columns are permuted by their row, so that neither side meets bank
// conflicts.  One value at a time and 32 x 32 tiles before: BF16 copies of the
// dense 8192 x 8192 matrix 165 -> 101 us as stored, 165 -> 121 us transposed (640
// MB each, 5.3 - 6.3 TB/s); TF32 copies of the 262,144-row chain 115 -> 94 us
// from FP64, 123 -> 64 us from FP32.
template <int ELT, typename V>
__device__ __forceinline__ void convert4(const V* __restrict__ p, bool wide, uint32_t (&w)[4]) {
  if constexpr (std::is_same<V, float>::value) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p));
    const float f[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = ELT == 2 ? f32_to_bf16_bits_rne(f[i]) : f32_to_tf32(f32_flush(f[i]));
  } else {
    double x[4];
    load4(p, x, wide);
    if constexpr (ELT == 4) f64_to_tf32_x4(x, w);
    else f64_to_bf16_x4(x, w);
  }
}

template <int ELT>
__device__ __forceinline__ void put4(void* dst, size_t i, const uint32_t (&w)[4]) {
  if constexpr (ELT == 4)
    *reinterpret_cast<uint4*>(static_cast<uint32_t*>(dst) + i) = make_uint4(w[0], w[1], w[2], w[3]);
  else
    *reinterpret_cast<uint2*>(static_cast<uint16_t*>(dst) + i) = make_uint2(w[0] | (w[1] << 16), w[2] | (w[3] << 16));
}

template <int ELT, int B, bool TR, typename V>
__global__ void __launch_bounds__(256) k_convert(const V* __restrict__ val, bool wide, const int32_t* __restrict__ src,
                                                 int64_t nblk, void* __restrict__ dst) {
  constexpr int BSZ = B * B, TS = B < 64 ? B : 64;
  using T = typename std::conditional<ELT == 2, uint16_t, uint32_t>::type;
  __shared__ T tile[TR ? TS * TS : 1];
  // element (r, c) of a tile: rows of four permute the groups' places
  const auto at = [](int r, int c) { return r * TS + (c ^ ((r >> 2) & 15)); };
  for (int64_t qb = blockIdx.x; qb <= nblk; qb += gridDim.x) {
    const size_t d = (size_t)qb * BSZ;
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (qb == nblk) {  // the zero block
      for (int e = (int)threadIdx.x * 4; e < BSZ; e += 1024) put4<ELT>(dst, d + e, w);
      continue;
    }
    const V* s = val + (size_t)(src ? src[qb] : qb) * BSZ;
    if constexpr (!TR) {
#pragma unroll 4
      for (int e = (int)threadIdx.x * 4; e < BSZ; e += 1024) {
        convert4<ELT>(s + e, wide, w);
        put4<ELT>(dst, d + e, w);
      }
    } else {
      for (int ti = 0; ti < B / TS; ++ti)
        for (int tj = 0; tj < B / TS; ++tj) {
          // stored rows ti TS.., columns tj TS.. -> copy rows tj TS.., columns ti TS..
#pragma unroll
          for (int e = (int)threadIdx.x * 4; e < TS * TS; e += 1024) {
            const int r = e / TS, c = e % TS;
            convert4<ELT>(s + (size_t)(ti * TS + r) * B + tj * TS + c, wide, w);
#pragma unroll
            for (int i = 0; i < 4; ++i) tile[at(r, c + i)] = (T)w[i];
          }
          __syncthreads();
#pragma unroll
          for (int e = (int)threadIdx.x * 4; e < TS * TS; e += 1024) {
            const int r = e / TS, c = e % TS;
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = tile[at(c + i, r)];
            put4<ELT>(dst, d + (size_t)(tj * TS + r) * B + ti * TS + c, w);
          }
          __syncthreads();
        }
    }
  }
}

// out[q] = vmap[src[q]] (src null: identity): the value position of view entry
// q of a matrix whose kept blocks stayed in place after truncation
__global__ void k_compose(const int32_t* __restrict__ src, const int32_t* __restrict__ vmap, int64_t n,
                          int32_t* __restrict__ out) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q < n) out[q] = vmap[src ? src[q] : q];
}

static const int32_t* value_src(ifac_ctx* ctx, const int32_t* src, const int32_t* vmap, int64_t n,
                                Buf<int32_t>& keep) {
  if (!vmap) return src;
  keep = Buf<int32_t>(ctx, (size_t)std::max<int64_t>(n, 1));
  if (n > 0) {
    k_compose<<<cdiv(n, 256), 256, 0, ctx->stream>>>(src, vmap, n, keep.p);
    IFAC_CK_LAUNCH();
  }
  return keep.p;
}

// P = b1 D + b2 W, the correction polynomial of Eq. (2.1) at m = 2 in the
// mixed schedule, written straight into the low-precision op(B) copy that
// M = Z P reads (P itself is never stored in FP64): block p of P's pattern,
// (I, J), is stored transposed ([j][k], as op(B) blocks are), W_IJ = U_IJ for
// J >= I and U_JI^T below, U the upper block triangle of delta^2.  The block
// is assembled in FP32 in shared memory (inputs rounded to FP32 on their bit
// patterns, one FMA per element), then rounded to TF32 / BF16 as k_convert
// rounds.  One CTA per block (grid-stride).  U's values are FP64 or the FP32
// results of its TF32/BF16 product (UV = float), rounded alike.
template <int ELT, typename UV>
__global__ void __launch_bounds__(256)
    k_poly2_lp(const int32_t* __restrict__ prow, const int32_t* __restrict__ pci, int64_t pnnz,
               const int32_t* __restrict__ urp, const int32_t* __restrict__ uci, const UV* __restrict__ uval,
               const int32_t* __restrict__ umap, const int32_t* __restrict__ drp, const int32_t* __restrict__ dci,
               const double* __restrict__ dval, float b1, float b2, void* __restrict__ dst) {
  constexpr int B = 64, BSZ = B * B;
  using T = typename std::conditional<ELT == 2, uint16_t, uint32_t>::type;
  __shared__ float t[B][B + 1];
  __shared__ int sq[2];
  const auto f32 = [](double x) { return __uint_as_float(f64_to_f32_bits_rne(x)); };
  const auto u32 = [](UV x) {
    if constexpr (std::is_same<UV, float>::value) return f32_flush(x);
    else return __uint_as_float(f64_to_f32_bits_rne(x));
  };
  T* out = reinterpret_cast<T*>(dst);
  for (int64_t p = blockIdx.x; p < pnnz; p += gridDim.x) {
    const int I = prow[p], J = pci[p];
    if (threadIdx.x == 0) {
      int k = lower_bound_i32(dci, drp[I], drp[I + 1], J);
      sq[0] = (k < drp[I + 1] && dci[k] == J) ? k : -1;
      const int r = I < J ? I : J, c = I < J ? J : I;
      k = lower_bound_i32(uci, urp[r], urp[r + 1], c);
      sq[1] = (k < urp[r + 1] && uci[k] == c) ? (umap ? umap[k] : k) : -1;
    }
    __syncthreads();
    const int qd = sq[0], qu = sq[1];
    for (int e = threadIdx.x; e < BSZ; e += blockDim.x)
      t[e >> 6][e & 63] = qd >= 0 ? b1 * f32(dval[(size_t)qd * BSZ + e]) : 0.0f;
    __syncthreads();
    if (qu >= 0) {
      const UV* u = uval + (size_t)qu * BSZ;
      if (J >= I) {
        for (int e = threadIdx.x; e < BSZ; e += blockDim.x)
          t[e >> 6][e & 63] = fmaf(b2, u32(u[e]), t[e >> 6][e & 63]);
      } else {  // U_JI read in its stored order, added transposed
        for (int e = threadIdx.x; e < BSZ; e += blockDim.x)
          t[e & 63][e >> 6] = fmaf(b2, u32(u[e]), t[e & 63][e >> 6]);
      }
      __syncthreads();
    }
    // row c of the copy is column c of P_IJ
    T* d = out + (size_t)p * BSZ;
    for (int e = threadIdx.x; e < BSZ; e += blockDim.x) {
      const float v = t[e & 63][e >> 6];
      if constexpr (ELT == 2) d[e] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
      else d[e] = f32_to_tf32(v);
    }
    __syncthreads();  // t is rewritten for the next block
  }
}

// Tiles of a sparse C in one pass over its blocks: block p owns its tile
// (I / tm, J / tn) when the tile holds no earlier block, i.e. neither the block
// before it in row I nor a block of the tile's earlier rows lies in the tile's
// column range.  The owners, in C's order, list every tile once.
__global__ void __launch_bounds__(256)
    k_tile_owner(const int32_t* __restrict__ row, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                 int64_t nnz, int tm, int tn, int32_t* __restrict__ own, int32_t* __restrict__ off,
                 unsigned* __restrict__ ticket) {  // off null: scanned afterwards
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p < nnz) {
    const int I = row[p], c0 = (ci[p] / tn) * tn;
    int o = (p > rp[I] && ci[p - 1] >= c0) ? 0 : 1;
    for (int I2 = (I / tm) * tm; o && I2 < I; ++I2) {
      const int hi = rp[I2 + 1];
      const int q = lower_bound_i32(ci, rp[I2], hi, c0);
      if (q < hi && ci[q] < c0 + tn) o = 0;
    }
    own[p] = o;
  }
  if (off) scan_tail<256>(own, off, (int)nnz, ticket, nullptr);
}

__global__ void k_tile_owner_write(const int32_t* __restrict__ row, const int32_t* __restrict__ ci, int64_t nnz,
                                   int tm, int tn, const int32_t* __restrict__ off, int32_t* __restrict__ out) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= nnz || off[p + 1] == off[p]) return;
  out[2 * (size_t)off[p]] = row[p] / tm;
  out[2 * (size_t)off[p] + 1] = ci[p] / tn;
}

// Tile compaction in grouped order: linear index li runs over groups of GROUP
// tile rows, column by column inside a group, so that CTAs running at the same
// time share op(B) panels in L2.  Three passes: count per chunk, scan, write.
constexpr int GROUP = 8;
constexpr int CHUNK = 1024;

__device__ __forceinline__ int64_t grouped_to_rowmajor(int64_t li, int ntr, int ntc) {
  const int64_t g = li / ((int64_t)GROUP * ntc);
  const int64_t rows = min((int64_t)GROUP, (int64_t)ntr - g * GROUP);
  const int64_t off = li - g * GROUP * ntc;
  return (g * GROUP + off % rows) * ntc + off / rows;
}

// flag[li] = 1 when tile li (grouped order) holds a block of C's pattern;
// counts per chunk and their scan
__global__ void __launch_bounds__(CHUNK)
    k_tile_mark(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int nb, int tm, int tn, int ntr,
                int ntc, uint8_t* __restrict__ flag, int32_t* __restrict__ cnt, int32_t* __restrict__ off,
                unsigned* __restrict__ ticket) {
  const int64_t tot = (int64_t)ntr * ntc;
  const int64_t li = (int64_t)blockIdx.x * CHUNK + threadIdx.x;
  int f = 0;
  if (li < tot) {
    const int64_t i = grouped_to_rowmajor(li, ntr, ntc);
    const int I0 = (int)(i / ntc) * tm, c0 = (int)(i % ntc) * tn;
    for (int I = I0; !f && I < min(I0 + tm, nb); ++I) {
      const int hi = rp[I + 1], q = lower_bound_i32(ci, rp[I], hi, c0);
      f = (q < hi && ci[q] < c0 + tn) ? 1 : 0;
    }
    flag[li] = (uint8_t)f;
  }
  const int c = __syncthreads_count(f);
  if (threadIdx.x == 0) cnt[blockIdx.x] = c;
  scan_tail<CHUNK>(cnt, off, (int)gridDim.x, ticket, nullptr);
}

__global__ void k_tile_write(const uint8_t* __restrict__ flag, int ntr, int ntc, const int32_t* __restrict__ off,
                             int32_t* __restrict__ out) {
  __shared__ int wbase[32];
  const int64_t tot = (int64_t)ntr * ntc;
  const int64_t li = (int64_t)blockIdx.x * CHUNK + threadIdx.x;
  const int64_t i = li < tot ? grouped_to_rowmajor(li, ntr, ntc) : 0;
  const bool f = li < tot && flag[li];
  const unsigned m = __ballot_sync(0xffffffffu, f);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) wbase[w] = __popc(m);
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int k = 0; k < CHUNK / 32; ++k) {
      const int c = wbase[k];
      wbase[k] = acc;
      acc += c;
    }
  }
  __syncthreads();
  if (f) {
    const int pos = off[blockIdx.x] + wbase[w] + __popc(m & ((1u << lane) - 1u));
    out[2 * pos] = (int32_t)(i / ntc);
    out[2 * pos + 1] = (int32_t)(i % ntc);
  }
}

// The same list for up to 65,536 tiles and blocks, in one CTA: flags in shared
// memory from C's blocks, then one thread per tile.  (Two launches of searches
// take 9 us on a few hundred block rows.)
constexpr int SMALL_TILES = 65536;

template <int TMB, int TNB>
__global__ void __launch_bounds__(1024)
    k_tiles_small(const int32_t* __restrict__ row, const int32_t* __restrict__ ci, int nnz, int ntr, int ntc,
                  int32_t* __restrict__ out, int32_t* __restrict__ count) {
  extern __shared__ uint32_t tbits[];  // [words] bit per tile, grouped order; [words] tiles before each word
  __shared__ int wsum[32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tot = ntr * ntc, words = (tot + 31) / 32, per = (words + 1023) / 1024;
  int* before = reinterpret_cast<int*>(tbits + words);
  for (int i = tid; i < words; i += 1024) tbits[i] = 0u;
  __syncthreads();
#pragma unroll 4
  for (int p = tid; p < nnz; p += 1024) {
    const int tr = row[p] / TMB, tc = ci[p] / TNB, g = tr / GROUP, rows = min(GROUP, ntr - g * GROUP);
    const int li = g * GROUP * ntc + (tr - g * GROUP) + rows * tc;
    const uint32_t bit = 1u << (li & 31);
    if (!(tbits[li >> 5] & bit)) atomicOr(&tbits[li >> 5], bit);
  }
  __syncthreads();
  const int w0 = min(tid * per, words), w1 = min(w0 + per, words);
  int c = 0;
  for (int w = w0; w < w1; ++w) c += __popc(tbits[w]);
  int x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  int pos = x - c;
  for (int w = 0; w < wid; ++w) pos += wsum[w];
  if (tid == 1023) *count = pos + c;
  for (int w = w0; w < w1; ++w) {
    before[w] = pos;
    pos += __popc(tbits[w]);
  }
  __syncthreads();
  for (int li = tid; li < tot; li += 1024) {
    const uint32_t u = tbits[li >> 5], bit = 1u << (li & 31);
    if (!(u & bit)) continue;
    const int q = before[li >> 5] + __popc(u & (bit - 1u));
    const int g = li / (GROUP * ntc), rows = min(GROUP, ntr - g * GROUP), off = li - g * GROUP * ntc;
    out[2 * q] = g * GROUP + off % rows;
    out[2 * q + 1] = off / rows;
  }
}

// What a tile plan reads, one warp per block row: the bitmap of op(A)'s row
// (its K set) and, where they are kept, row I of the dense block-index maps,
// map[I nb + J] = q for block q, else the zero block's index.
//
// Also the number of stored block pairs (op(A)_IK, op(B)_KJ) of the product,
// i.e. |row K of op(B)| for every block (I, K): all of them, or with upper
// only those with J >= I.  pairs (nullable) gets one per pair, wpairs
// (nullable) w per pair.
__global__ void __launch_bounds__(256)
    k_plan_rows(const int32_t* __restrict__ arp, const int32_t* __restrict__ aci, const int32_t* __restrict__ brp,
                const int32_t* __restrict__ bci, int nb, int W, uint32_t* __restrict__ bm, int32_t* __restrict__ mapA,
                int32_t* __restrict__ mapB, int a_zero, int b_zero, int upper,
                unsigned long long* __restrict__ pairs, unsigned long long* __restrict__ wpairs, int w) {
  const int row = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (row >= nb) return;
  uint32_t* bits = bm + (size_t)row * W;
  for (int i = lane; i < W; i += 32) bits[i] = 0u;
  if (mapA)
    for (int c = lane; c < nb; c += 32) {
      mapA[(size_t)row * nb + c] = a_zero;
      mapB[(size_t)row * nb + c] = b_zero;
    }
  __syncwarp();
  unsigned long long c = 0;
  for (int p = arp[row] + lane; p < arp[row + 1]; p += 32) {
    const int K = aci[p];
    atomicOr(bits + (K >> 5), 1u << (K & 31));
    if (mapA) mapA[(size_t)row * nb + K] = p;
    if (pairs) c += (unsigned long long)(brp[K + 1] - (upper ? lower_bound_i32(bci, brp[K], brp[K + 1], row) : brp[K]));
  }
  if (mapB)
    for (int p = brp[row] + lane; p < brp[row + 1]; p += 32) mapB[(size_t)row * nb + bci[p]] = p;
  if (!pairs) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0 && c) {
    atomicAdd(pairs, c);
    if (wpairs) atomicAdd(wpairs, c * (unsigned long long)w);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encoder() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    IFAC_CK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !p) fail(IFAC_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Exclusive scan for longer lists than scan_tail is good for (its one CTA of
// 256 threads takes 31 us for 20,000 counts, one of 1024 threads 16 us).  CTA b
// adds up everything before its 4096 counts by itself, so no CTA waits for
// another: 80 KB from L2 at most for those 20,000, but reads grow with the
// square (0.5 GB at 10^6 counts), so from SCAN_LONG counts on (1 MB a CTA)
// k_chunk_sums leaves each chunk's sum first and a CTA adds up those before its
// own: a TF32 product of 10^6 blocks, two scans, 8.87 -> 8.81 ms.  The total and
// the longest tile (kmax, nullable) for the host.
constexpr int TAIL_SCAN = 8192;
constexpr int SCAN_CHUNK = 4096;
constexpr int SCAN_LONG = 1 << 18;

// sum of a thread's values over a CTA of 1024 threads, in every thread
__device__ __forceinline__ int cta_sum(int s, int* wsum) {
  s = (int)__reduce_add_sync(0xffffffffu, (unsigned)s);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = s;
  __syncthreads();
  return (int)__reduce_add_sync(0xffffffffu, (unsigned)wsum[threadIdx.x & 31]);
}

__global__ void __launch_bounds__(1024) k_chunk_sums(const int32_t* __restrict__ cnt, int n, int32_t* __restrict__ sums) {
  __shared__ int wsum[32];
  int s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_CHUNK / 1024; ++k) {
    const int64_t i = (int64_t)blockIdx.x * SCAN_CHUNK + k * 1024 + threadIdx.x;
    s += i < n ? cnt[i] : 0;
  }
  s = cta_sum(s, wsum);
  if (threadIdx.x == 0) sums[blockIdx.x] = s;
}

// sums: the chunks' sums, or null
__global__ void __launch_bounds__(1024) k_scan(const int32_t* __restrict__ cnt, const int32_t* __restrict__ sums,
                                               int32_t* __restrict__ out, int n, int32_t* total, int* kmax,
                                               int32_t* host_kmax) {
  __shared__ int wsum[2][32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, c0 = (int)blockIdx.x * SCAN_CHUNK;
  int s = 0;
  if (sums) {
    for (int i = tid; i < (int)blockIdx.x; i += 1024) s += sums[i];
  } else {
#pragma unroll 8
    for (int i = tid; i < c0; i += 1024) s += cnt[i];
  }
  const int base = cta_sum(s, wsum[0]);
  int v[4], t = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = n - c0 > tid * 4 + k ? cnt[c0 + tid * 4 + k] : 0;
    t += v[k];
  }
  int x = t;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[1][wid] = x;
  __syncthreads();
  const int own = wsum[1][lane];
  int run = base + (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < wid ? own : 0)) + x - t;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int i = c0 + tid * 4 + k;
    if (i < n) out[i] = run;
    run += v[k];
    if (i == n - 1) {
      out[n] = run;
      if (total) *total = run;
      if (kmax) *host_kmax = atomicExch(kmax, 0);
    }
  }
}

static void scan_counts(ifac_ctx* ctx, const int32_t* cnt, int32_t* out, int64_t n, int32_t* total, int* kmax,
                        int32_t* host_kmax) {
  const int chunks = cdiv(n, SCAN_CHUNK);
  Buf<int32_t> sums;
  if (n >= SCAN_LONG) {
    sums = Buf<int32_t>(ctx, chunks);
    k_chunk_sums<<<chunks, 1024, 0, ctx->stream>>>(cnt, (int)n, sums.p);
    IFAC_CK_LAUNCH();
  }
  k_scan<<<chunks, 1024, 0, ctx->stream>>>(cnt, sums.p, out, (int)n, total, kmax, host_kmax);
  IFAC_CK_LAUNCH();
}

// Plan records of every super-tile: for each K of the union of its rows'
// bitmaps at which some op(B)_KJ of its columns is stored, the copy index of
// op(A)_IK for each of its ROWS block rows and of op(B)_KJ for each of its
// COLS block columns (the zero block when absent); K steps whose op(B) blocks
// are all absent contribute nothing and are left out.  One warp per tile,
// candidate K's 32 at a time, lane-parallel.  PLAN_COUNT: the number of records
// into nk[t], their offsets, and the total and the largest for the host;
// PLAN_RECORDS: the records, from off[t] on; PLAN_BOTH: both in one pass, tile
// t's records from t nb on.  With the records, the position in C's pattern of
// each of the tile's ROWS x COLS blocks (-1 where C holds none), so that a
// product's epilogue finds its output blocks with one load instead of a
// search.
enum PlanMode { PLAN_COUNT, PLAN_RECORDS, PLAN_BOTH };
constexpr int PLAN_NT = 256;

template <int ROWS, int COLS, int MODE>
__global__ void __launch_bounds__(PLAN_NT) k_tile_plan(const int32_t* __restrict__ tiles, const int* __restrict__ ntiles,
                            const int32_t* __restrict__ off, const uint32_t* __restrict__ bm, int nb, int W,
                            const int32_t* __restrict__ mapA, const int32_t* __restrict__ mapB,
                            const int32_t* __restrict__ arp, const int32_t* __restrict__ aci,
                            const int32_t* __restrict__ brp, const int32_t* __restrict__ bci, int a_zero, int b_zero,
                            const int32_t* __restrict__ amap, int32_t* __restrict__ rec, int32_t* __restrict__ nk_out,
                            int* __restrict__ kmax, const int32_t* __restrict__ crp = nullptr,
                            const int32_t* __restrict__ cci = nullptr, int32_t* __restrict__ cpos = nullptr,
                            const int32_t* __restrict__ bmap = nullptr, int nt = 0, int32_t* off_out = nullptr,
                            unsigned* ticket = nullptr, int32_t* host_kmax = nullptr) {
  static_assert(ROWS * COLS <= 32, "one lane per block of the tile");
  const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  constexpr bool COUNT = MODE == PLAN_COUNT;  // no records
  // the grid covers an upper bound nt of the tile count
  const int e0 = MODE == PLAN_COUNT ? 0 : MODE == PLAN_BOTH ? (int)t * nb : (t < *ntiles ? off[t] : 0);
  int e = e0;
  if (t < *ntiles) {
  const int I0 = tiles[2 * t] * ROWS, J0 = tiles[2 * t + 1] * COLS;
  if (!COUNT && cpos && lane < ROWS * COLS) {
    const int I = I0 + lane / COLS, J = J0 + lane % COLS;
    int pos = -1;
    if (I < nb && J < nb) {
      const int hi = crp[I + 1];
      const int q = lower_bound_i32(cci, crp[I], hi, J);
      if (q < hi && cci[q] == J) pos = q;
    }
    cpos[(size_t)t * (ROWS * COLS) + lane] = pos;
  }
  // op(B)'s copy indices of K, true when any block is stored
  const auto b_blocks = [&](int K, int (&rb)[COLS]) -> bool {
    bool any = false;
    if (mapA) {
#pragma unroll
      for (int c = 0; c < COLS; ++c) rb[c] = (J0 + c < nb) ? mapB[(size_t)K * nb + J0 + c] : b_zero;
    } else {
      const int hi = brp[K + 1];
      int q = lower_bound_i32(bci, brp[K], hi, J0);
#pragma unroll
      for (int c = 0; c < COLS; ++c) {
        int idx = b_zero;
        if (q < hi && bci[q] == J0 + c) idx = q++;
        rb[c] = idx;
      }
    }
#pragma unroll
    for (int c = 0; c < COLS; ++c) any |= rb[c] != b_zero;
    return any;
  };
  // 32 words of the K set at a time.  The lanes take the 32 K's of one word
  // together (one K per word and lane left all but two lanes idle at 64 block
  // rows).  The records are in the order of the products' K loops, which their
  // FP32 sums depend on: the first K of every word, then the second, ...
  for (int wbase = 0; wbase < W; wbase += 32) {
    const int w = wbase + lane;
    uint32_t word = 0;
    if (w < W) {
#pragma unroll
      for (int r = 0; r < ROWS; ++r)
        if (I0 + r < nb) word |= bm[(size_t)(I0 + r) * W + w];
    }
    const unsigned nz = __ballot_sync(0xffffffffu, word != 0u);
    if (!nz) continue;
    uint32_t ranks = 0;  // this lane's word: bit j set when its j-th K has a record
    for (unsigned z = nz; z; z &= z - 1u) {
      const int src = __ffs((int)z) - 1;
      const uint32_t wd = __shfl_sync(0xffffffffu, word, src);
      int rb[COLS];
      const bool rec_here = ((wd >> lane) & 1u) && b_blocks((wbase + src) * 32 + lane, rb);
      const uint32_t m = __reduce_or_sync(0xffffffffu, rec_here ? 1u << __popc(wd & ((1u << lane) - 1u)) : 0u);
      if (lane == src) ranks = m;
    }
    const int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(ranks));
    if constexpr (!COUNT) {
      // lane j: the words that have a j-th record, and the records before its j-th ones
      uint32_t col = 0;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const uint32_t b = __ballot_sync(0xffffffffu, (ranks >> j) & 1u);
        if (lane == j) col = b;
      }
      int before = __popc(col);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before += y;
      }
      before -= __popc(col);
      for (unsigned z = nz; z; z &= z - 1u) {
        const int src = __ffs((int)z) - 1;
        const uint32_t wd = __shfl_sync(0xffffffffu, word, src);
        const int K = (wbase + src) * 32 + lane, j = __popc(wd & ((1u << lane) - 1u)) & 31;
        const int pos = __shfl_sync(0xffffffffu, before, j) +
                        __popc(__shfl_sync(0xffffffffu, col, j) & ((1u << src) - 1u));
        int ra[ROWS], rb[COLS];
        if (((wd >> lane) & 1u) && b_blocks(K, rb)) {
          if (mapA) {
#pragma unroll
            for (int r = 0; r < ROWS; ++r) ra[r] = (I0 + r < nb) ? mapA[(size_t)(I0 + r) * nb + K] : a_zero;
          } else {
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
              int idx = a_zero;
              if (I0 + r < nb) {
                const int hi = arp[I0 + r + 1];
                const int q = lower_bound_i32(aci, arp[I0 + r], hi, K);
                if (q < hi && aci[q] == K) idx = q;
              }
              ra[r] = idx;
            }
          }
          int32_t* out = rec + (size_t)(e + pos) * (ROWS + COLS);
#pragma unroll
          for (int r = 0; r < ROWS; ++r) out[r] = (amap && ra[r] != a_zero) ? amap[ra[r]] : ra[r];
#pragma unroll
          for (int c = 0; c < COLS; ++c) out[ROWS + c] = (bmap && rb[c] != b_zero) ? bmap[rb[c]] : rb[c];
        }
      }
    }
    e += total;
  }
  }
  if constexpr (MODE == PLAN_BOTH) {
    if (lane == 0 && t < nt) {
      nk_out[t] = e - e0;
      off_out[t] = e0;
      atomicMax(kmax, e - e0);
    }
    // the longest tile for the host
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(ticket, 1u) == gridDim.x - 1) {
      *ticket = 0u;
      const int longest = atomicExch(kmax, 0);
      if (host_kmax) *host_kmax = longest;
    }
  }
  if constexpr (COUNT) {
    if (lane == 0 && t < nt) {
      nk_out[t] = e;
      atomicMax(kmax, e);
    }
  }
}

// The tile plan of a product: super-tiles of ROWS x COLS blocks holding a
// block of C's pattern (grouped order), their K-step counts and records.
struct Plan {
  Buf<int32_t> tiles, coff, tnk, off, rec, cpos;  // cpos: C positions of each tile's blocks
  int nchunk = 0;
  int64_t ntot = 0;
  int ntiles = 0;  // upper bound of the tile count (the count itself stays on the device)
  int kmax = 0;
};

// the block pairs a plan counts on the way (once per product)
struct PairCount {
  bool upper = false;
  unsigned long long* pairs = nullptr;
  unsigned long long* wpairs = nullptr;
  int w = 0;
};

template <int ROWS, int COLS>
static Plan make_plan(ifac_ctx* ctx, const View& arows, const ifac_bsr& A, const View& brows, const ifac_bsr& B,
                      const ifac_bsr& C, const int32_t* crow, const PairCount& pc, bool want_kmax,
                      int kmax_limit = 0, const int32_t* amap = nullptr, const HostRead* extra = nullptr,
                      const int32_t* bmap = nullptr) {
  // amap (nullable): copy index of each op(A) view position, when op(A)'s
  // low-precision copy is not in view order (a shared copy of a transposed
  // operand, held in the stored order).  bmap (nullable): the same for
  // op(B) (a symmetric op(B) read from its op(A) copy).  extra (nullable): one
  // more small read-back the caller needs, taken behind the plan's kernels.
  // kmax_limit > 0: a plan whose longest tile has more K steps is not wanted;
  // it returns after the count pass with kmax set and no records
  const int nb = A.nb, W = words_per_row(nb);
  Plan P;
  // K sets (bitmap rows of op(A)); dense block-index maps of op(A), op(B)
  // while they stay small, binary searches in the CSR patterns beyond that
  Buf<uint32_t> bmA(ctx, (size_t)nb * W);
  const int64_t nb2 = (int64_t)nb * nb;
  const bool dense_maps = nb2 <= (int64_t)4 << 20;
  Buf<int32_t> imA, imB;
  if (dense_maps) {
    imA = Buf<int32_t>(ctx, nb2);
    imB = Buf<int32_t>(ctx, nb2);
  }
  k_plan_rows<<<cdiv((int64_t)nb * 32, 256), 256, 0, ctx->stream>>>(
      arows.rp, arows.ci, brows.rp, brows.ci, nb, W, bmA.p, imA.p, imB.p, (int)A.nnzb, (int)B.nnzb, pc.upper ? 1 : 0,
      pc.pairs, pc.wpairs, pc.w);
  IFAC_CK_LAUNCH();
  const int ntr = cdiv(nb, ROWS), ntc = cdiv(nb, COLS);
  P.ntot = (int64_t)ntr * ntc;
  if ((int64_t)C.nnzb * 16 < P.ntot) {
    // a sparse C (a banded product): its tiles from its blocks, in C's order
    P.nchunk = (int)C.nnzb;
    P.tiles = Buf<int32_t>(ctx, (size_t)2 * C.nnzb);
    P.coff = Buf<int32_t>(ctx, (size_t)C.nnzb + 1);
    Buf<int32_t> own(ctx, (size_t)C.nnzb);
    const bool tail = C.nnzb <= TAIL_SCAN;
    k_tile_owner<<<cdiv(C.nnzb, 256), 256, 0, ctx->stream>>>(crow, C.row_ptr, C.col_idx, C.nnzb, ROWS, COLS, own.p,
                                                             tail ? P.coff.p : nullptr, ctx->ticket);
    IFAC_CK_LAUNCH();
    if (!tail) {
      scan_counts(ctx, own.p, P.coff.p, C.nnzb, nullptr, nullptr, nullptr);
    }
    k_tile_owner_write<<<cdiv(C.nnzb, 256), 256, 0, ctx->stream>>>(crow, C.col_idx, C.nnzb, ROWS, COLS, P.coff.p,
                                                                   P.tiles.p);
    IFAC_CK_LAUNCH();
  } else if (P.ntot <= SMALL_TILES && C.nnzb <= SMALL_TILES) {
    P.nchunk = 0;
    P.tiles = Buf<int32_t>(ctx, (size_t)2 * P.ntot);
    P.coff = Buf<int32_t>(ctx, 1);
    k_tiles_small<ROWS, COLS><<<1, 1024, (size_t)cdiv(P.ntot, 32) * 8, ctx->stream>>>(
        crow, C.col_idx, (int)C.nnzb, ntr, ntc, P.tiles.p, P.coff.p);
    IFAC_CK_LAUNCH();
  } else {
    P.nchunk = cdiv(P.ntot, CHUNK);
    Buf<uint8_t> flags(ctx, (size_t)P.ntot);
    Buf<int32_t> ccnt(ctx, P.nchunk);
    P.tiles = Buf<int32_t>(ctx, (size_t)2 * P.ntot);
    P.coff = Buf<int32_t>(ctx, P.nchunk + 1);
    k_tile_mark<<<P.nchunk, CHUNK, 0, ctx->stream>>>(C.row_ptr, C.col_idx, nb, ROWS, COLS, ntr, ntc, flags.p, ccnt.p,
                                                     P.coff.p, ctx->ticket);
    IFAC_CK_LAUNCH();
    k_tile_write<<<P.nchunk, CHUNK, 0, ctx->stream>>>(flags.p, ntr, ntc, P.coff.p, P.tiles.p);
    IFAC_CK_LAUNCH();
  }
  const int* ntiles = P.coff.p + P.nchunk;
  // the per-tile kernels and arrays are sized by a bound of the tile count
  // (every tile holds a block of C, which is not empty), not by all ntr x ntc
  // positions
  const int nt = (int)std::min<int64_t>(P.ntot, C.nnzb);
  P.ntiles = nt;
  P.tnk = Buf<int32_t>(ctx, (size_t)nt);
  P.off = Buf<int32_t>(ctx, (size_t)nt + 1);
  P.cpos = Buf<int32_t>(ctx, (size_t)nt * (ROWS * COLS));
  const int pgrid = cdiv((int64_t)nt * 32, PLAN_NT);
  int* const kmax_dev = reinterpret_cast<int*>(ctx->ticket + 1);
  // While every tile could have nb K steps within 128 MB (in a caller's memory:
  // within an eighth of C's values), the records are written in one pass at a
  // fixed stride, and only the longest tile is read back; a longer list is
  // counted first.
  const int64_t most = (int64_t)nt * nb * (ROWS + COLS), fits = (int64_t)32 << 20;
  if (most <= (ctx->custom_alloc ? std::min(fits, C.nnzb * C.bs * C.bs / 8) : fits)) {
    P.rec = Buf<int32_t>(ctx, (size_t)nt * nb * (ROWS + COLS));
    k_tile_plan<ROWS, COLS, PLAN_BOTH><<<pgrid, PLAN_NT, 0, ctx->stream>>>(
        P.tiles.p, ntiles, nullptr, bmA.p, nb, W, imA.p, imB.p, arows.rp, arows.ci, brows.rp, brows.ci, (int)A.nnzb,
        (int)B.nnzb, amap, P.rec.p, P.tnk.p, kmax_dev, C.row_ptr, C.col_idx, P.cpos.p, bmap, nt, P.off.p,
        ctx->ticket, want_kmax ? host_word(ctx, HW_KMAX) : nullptr);  // (a word nobody reads is not written)
    IFAC_CK_LAUNCH();
    if (extra) to_host_many(ctx, {*extra});
    if (want_kmax) P.kmax = read_word(ctx, HW_KMAX);
    return P;
  }
  k_tile_plan<ROWS, COLS, PLAN_COUNT><<<pgrid, PLAN_NT, 0, ctx->stream>>>(
      P.tiles.p, ntiles, nullptr, bmA.p, nb, W, imA.p, imB.p, arows.rp, arows.ci, brows.rp, brows.ci, (int)A.nnzb,
      (int)B.nnzb, nullptr, nullptr, P.tnk.p, kmax_dev, nullptr, nullptr, nullptr, nullptr, nt, nullptr, nullptr,
      nullptr);
  IFAC_CK_LAUNCH();
  scan_counts(ctx, P.tnk.p, P.off.p, nt, host_word(ctx, HW_PLAN), kmax_dev, host_word(ctx, HW_KMAX));
  // the caller's extra read-back waits for the stream; the record count and
  // the longest tile are there then, or polled
  if (extra) to_host_many(ctx, {*extra});
  const int64_t total = read_word(ctx, HW_PLAN);
  P.kmax = read_word(ctx, HW_KMAX);
  if (total > (int64_t)0x7fffffff / (ROWS + COLS))
    fail(IFAC_ERR_TOO_LARGE, "tensor-core product: tile plan exceeds 2^31 entries");
  if (kmax_limit > 0 && P.kmax > kmax_limit) return P;
  P.rec = Buf<int32_t>(ctx, (size_t)std::max<int64_t>(total, 1) * (ROWS + COLS));
  k_tile_plan<ROWS, COLS, PLAN_RECORDS><<<pgrid, PLAN_NT, 0, ctx->stream>>>(
      P.tiles.p, ntiles, P.off.p, bmA.p, nb, W, imA.p, imB.p, arows.rp, arows.ci, brows.rp, brows.ci, (int)A.nnzb,
      (int)B.nnzb, amap, P.rec.p, nullptr, nullptr, C.row_ptr, C.col_idx, P.cpos.p, bmap);
  IFAC_CK_LAUNCH();
  // the plan kernel has read the maps and the bitmap before they are freed
  // (stream-ordered frees)
  return P;
}

// 2D view of a low-precision block array: rows = (nblk) * 64, 64 elements per
// row; boxes of one 128-byte atom x 64 rows, 128-byte swizzle
template <int ELT>
static CUtensorMap make_map(void* base, int64_t nblk) {
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)BS, (cuuint64_t)nblk * BS};
  cuuint64_t strides[1] = {(cuuint64_t)BS * ELT};
  cuuint32_t box[2] = {(cuuint32_t)Cfg<ELT>::ATOM_ELEMS, (cuuint32_t)BS};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = encoder()(&m, ELT == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base,
                         dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(IFAC_ERR_CUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
  return m;
}

// the same for bs x bs blocks (rows = nblk * bs, bs elements per row) with
// boxes of one swizzle atom (atom_elems elements, 64- or 128-byte swizzle) by
// bs rows, as the narrow-tile kernel reads them
static CUtensorMap make_map_bs(int elt, int bs, void* base, int64_t nblk, const BandShape& sh) {
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)bs, (cuuint64_t)nblk * bs};
  cuuint64_t strides[1] = {(cuuint64_t)bs * elt};
  cuuint32_t box[2] = {(cuuint32_t)sh.atom_elems, (cuuint32_t)bs};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = encoder()(&m, elt == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base,
                         dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         sh.atom_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(IFAC_ERR_CUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
  return m;
}

// BF16 slices of bs x bs blocks with boxes of inner x rows elements, 64- or
// 128-byte swizzle (inner * 2 bytes)
static CUtensorMap make_map_box(int bs, void* base, int64_t nblk, int inner, int rows) {
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)bs, (cuuint64_t)nblk * bs};
  cuuint64_t strides[1] = {(cuuint64_t)bs * 2};
  cuuint32_t box[2] = {(cuuint32_t)inner, (cuuint32_t)rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = encoder()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE,
                         inner * 2 == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(IFAC_ERR_CUDA, "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
  return m;
}

template <int ELT, bool TR, typename V>
static void launch_convert(ifac_ctx* ctx, int bs, const V* val, const int32_t* src, int64_t nblk, void* dst) {
  const int grid = (int)std::min<int64_t>(nblk + 1, 152 * 16);
  const bool wide = aligned32(val);
  if (bs == 32) k_convert<ELT, 32, TR, V><<<grid, 256, 0, ctx->stream>>>(val, wide, src, nblk, dst);
  else if (bs == 64) k_convert<ELT, 64, TR, V><<<grid, 256, 0, ctx->stream>>>(val, wide, src, nblk, dst);
  else k_convert<ELT, 128, TR, V><<<grid, 256, 0, ctx->stream>>>(val, wide, src, nblk, dst);
  IFAC_CK_LAUNCH();
}

template <int ELT, typename V = double>
static void convert_blocks(ifac_ctx* ctx, int bs, const V* val, const int32_t* src, int64_t nblk, bool tr,
                           void* dst) {
  if (tr) launch_convert<ELT, true>(ctx, bs, val, src, nblk, dst);
  else launch_convert<ELT, false>(ctx, bs, val, src, nblk, dst);
}

// the narrow-tile plan of a block size (tile of 128 / bs x max(64, bs) / bs blocks)
static Plan band_plan(ifac_ctx* ctx, int bs, const View& arows, const ifac_bsr& A, const View& brows,
                      const ifac_bsr& B, const ifac_bsr& C, const int32_t* crow, const PairCount& pc, bool want_kmax,
                      int kmax_limit, const int32_t* amap, const HostRead* extra = nullptr, const int32_t* bmap = nullptr) {
  if (bs == 32) return make_plan<4, 2>(ctx, arows, A, brows, B, C, crow, pc, want_kmax, kmax_limit, amap, extra, bmap);
  if (bs == 64) return make_plan<2, 1>(ctx, arows, A, brows, B, C, crow, pc, want_kmax, kmax_limit, amap, extra, bmap);
  return make_plan<1, 1>(ctx, arows, A, brows, B, C, crow, pc, want_kmax, kmax_limit, amap, extra, bmap);
}

// out32: C's values are written as FP32 (C.val holds floats); b32: B's values
// are FP32 (an earlier product's out32 result)
template <int ELT>
static void run(ifac_ctx* ctx, const View& arows, bool tA, const ifac_bsr& A, const View& brows, bool tB,
                const ifac_bsr& B, double alpha, ifac_bsr& C, const int32_t* crow, bool upper,
                unsigned long long* pairs, OperandCache* ac, OperandCache* bc, const OperandCache* bpre,
                const int32_t* avmap, const int32_t* bvmap, bool out32, bool b32) {
  using Cf = Cfg<ELT>;
  const int nb = A.nb, bs = A.bs;
  const size_t bbytes = (size_t)bs * bs * ELT;
  // a cache filled by an earlier product's op(B) holds transposed blocks in
  // the stored order: it serves op(A) = that matrix transposed, through the
  // view's source indices, and nothing else
  if (ac && ac->from_b && !(tA && ac->conv_elt == ELT)) ac = nullptr;
  const int32_t* amap = (ac && ac->from_b) ? arows.src : nullptr;
  // low-precision, K-major copies of op(A) and op(B) plus one zero block each
  // (op(A)'s taken from the cache when it holds one of this format, op(B)'s
  // from bpre when its producer wrote it in this format)
  const bool bhit = bpre && bpre->b_ready && bpre->conv_elt == ELT && !tB;
  // an exactly symmetric op(B) = B whose op(A) copy is at hand: block (K, J)
  // of the op(B) copy, B_KJ^T = B_JK, is that copy's block at tpos
  const bool bsym = !bhit && bpre && bpre->tpos.p && bpre->conv_elt == ELT && !tB;
  const int32_t* bmap = bsym ? bpre->tpos.p : nullptr;
  Buf<uint8_t> la, lb;
  const bool hit = ac && ac->conv_elt == ELT;
  if (!hit) {
    la = Buf<uint8_t>(ctx, (size_t)(A.nnzb + 1) * bbytes);
    Buf<int32_t> asrc;
    convert_blocks<ELT>(ctx, bs, A.val, value_src(ctx, arows.src, avmap, A.nnzb, asrc), A.nnzb, tA, la.p);
    if (ac) {
      ac->conv = std::move(la);
      ac->conv_elt = ELT;
    }
  }
  uint8_t* const la_p = ac ? ac->conv.p : la.p;
  if (!bhit && !bsym) {
    lb = Buf<uint8_t>(ctx, (size_t)(B.nnzb + 1) * bbytes);
    Buf<int32_t> bsrc;
    const int32_t* vs = value_src(ctx, brows.src, bvmap, B.nnzb, bsrc);
    if (b32) convert_blocks<ELT, float>(ctx, bs, reinterpret_cast<const float*>(B.val), vs, B.nnzb, !tB, lb.p);
    else convert_blocks<ELT>(ctx, bs, B.val, vs, B.nnzb, !tB, lb.p);
  }
  uint8_t* const lb_p = (bhit || bsym) ? bpre->conv.p : lb.p;
  if (bc && !tB && !bhit && !bsym) {  // op(B) = B in its stored order: keep the copy for a later op(A) = B^T
    bc->reset();
    bc->conv = std::move(lb);
    bc->conv_elt = ELT;
    bc->from_b = true;
  }
  PairCount pc;
  pc.upper = upper;
  pc.pairs = pairs;
  // narrow tiles (gemm_band.cu) for every product at bs 32 and 128, and for
  // the banded ones at bs 64 (no 128 x 64 tile with more than KW K steps);
  // the super-tiles below for the other bs-64 products
  // (the context's schedule can ask for super-tiles only, or narrow tiles up
  // to another K length)
  const int nk_lim = ctx->narrow_kmax < 0 ? KW : ctx->narrow_kmax;
  // (no plan is made to find out where a full operand tells: every tile's K
  // set is then as long as a row of the other, which holds more than nk_lim
  // blocks on average)
  const int64_t full = (int64_t)nb * nb;
  const bool wide = (B.nnzb == full && A.nnzb > (int64_t)nk_lim * nb) ||
                    (A.nnzb == full && B.nnzb > (int64_t)nk_lim * nb);
  if (bs != 64 || (nk_lim > 0 && !wide)) {
    const BandShape sh = band_lp_shape(ELT, bs);
    Plan Pb = band_plan(ctx, bs, arows, A, brows, B, C, crow, pc, bs == 64, bs == 64 ? nk_lim : 0, amap, nullptr, bmap);
    pc.pairs = nullptr;  // counted
    if (bs != 64 || (Pb.kmax >= 1 && Pb.kmax <= nk_lim)) {
      const CUtensorMap mapA = make_map_bs(ELT, bs, la_p, A.nnzb + 1, sh);
      const CUtensorMap mapB = make_map_bs(ELT, bs, lb_p, B.nnzb + 1, sh);
      prof_begin(ctx, 1);
      band_lp_product(ctx, ELT, bs, &mapA, &mapB, Pb.tiles.p, Pb.coff.p + Pb.nchunk, Pb.tnk.p, Pb.rec.p, Pb.off.p,
                      Pb.cpos.p, Pb.ntiles, alpha, C, out32);
      prof_end(ctx);
      ++ctx->tc_launches;
      return;
    }
  }
  const CUtensorMap mapA = make_map<ELT>(la_p, A.nnzb + 1);
  const CUtensorMap mapB = make_map<ELT>(lb_p, B.nnzb + 1);
  // C's blocks fill more tiles of 4 x 4 than half the SMs: 256 x 256 elements a
  // CTA (gemm_wide.cu); a smaller product spreads over CTA pairs.  Scattered
  // blocks fill fewer tiles than that, and still: with one block in each tile
  // (every fourth row and column, 17 to 100 K blocks) TF32 is 1.06 - 1.15 times as
  // fast as on pairs, BF16 1.3 - 1.8 times; mostly one-pair blocks beside a few
  // long rows 0.92 times in TF32 (600 block rows), 1.25 in BF16.
  if (C.nnzb > 16 * 76) {
    Plan Pw = make_plan<4, 4>(ctx, arows, A, brows, B, C, crow, pc, false, 0, amap, nullptr, bmap);
    prof_begin(ctx, 1);
    wide_product(ctx, ELT, &mapA, &mapB, Pw.tiles.p, Pw.coff.p + Pw.nchunk, Pw.tnk.p, Pw.rec.p, Pw.off.p, Pw.cpos.p,
                 Pw.ntiles, alpha, C, out32);
    prof_end(ctx);
    ++ctx->tc_launches;
    return;
  }
  Plan P = make_plan<PAIR * TM, Cf::TN>(ctx, arows, A, brows, B, C, crow, pc, false, 0, amap, nullptr, bmap);
  static std::atomic<unsigned long long> attr{0};
  if (first_on_device(attr, ctx->device))
    IFAC_CK(cudaFuncSetAttribute(k_gemm_tc<ELT>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cf::SMEM_BYTES));
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  TileArgs args;
  args.tiles = P.tiles.p;
  args.ntiles = P.coff.p + P.nchunk;  // the scan's total
  args.tile_nk = P.tnk.p;
  args.nwin = 1;
  args.nb = nb;
  args.rec = P.rec.p;
  args.rec_off = P.off.p;
  args.crp = C.row_ptr;
  args.cci = C.col_idx;
  args.cval = out32 ? nullptr : C.val;
  args.cval32 = out32 ? reinterpret_cast<float*>(C.val) : nullptr;
  args.cnorm = C.norms;
  args.alpha = alpha;
  args.err = ctx->dev_err;
  args.split = 0;
  args.cpart = nullptr;
  args.ovf = nullptr;
  args.nunits = 0;
  for (int u = 0; u < MAX_UNITS; ++u) args.unit_end[u] = args.unit_sh[u] = 0;
  for (int p = 0; p < MAX_PAIRS; ++p) args.pair_ya[p] = args.pair_yb[p] = 0;
  args.stall = 0;
  args.wait_limit = WAIT_LIMIT;
  // one CTA per SM, in pairs; at most one pair per tile (idle pairs return at once)
  const int64_t pairs_grid = std::min<int64_t>(std::max(P.ntiles, 1), sms / PAIR);
  prof_begin(ctx, 1);
  k_gemm_tc<ELT><<<(unsigned)(pairs_grid * PAIR), NTHREADS, Cf::SMEM_BYTES, ctx->stream>>>(mapA, mapB, args);
  IFAC_CK_LAUNCH();
  prof_end(ctx);
  ++ctx->tc_launches;
}

// ---------------------------------------------------------------------------
// FP64-accurate products on the tensor cores by error-free splitting
// (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012): every row i of op(A) is scaled
// by a power of two sigma_i >= its largest magnitude and split into NS slices
// of 7-bit integers (exact in BF16), a = sigma_i sum_s q_s 2^(-7 s) + rest;
// likewise the columns of op(B) with tau_j.  A product of two slices
// (first slices |q| <= 128, later ones |q| <= 64) is a sum of integers, exact
// in FP32 while its magnitude bound stays <= 2^24.  Slice pairs with equal
// weight 2^(-7(s+t)), s + t <= NS + 1, are summed in accumulation units whose
// bound over a window of K blocks stays <= 2^24.  On narrow tiles every weight
// class is one unit, and a window as long as that allows (six blocks of 64 with
// NS = 8); the super-tile kernel's windows hold KW = 16 K blocks (1024 terms),
// or the longest tile's when fewer, and a class is packed greedily into as many
// units as it needs (NS = 7: 13 at full windows, 7 up to 7 K steps).  Per tile
// and window the epilogue adds each unit, scaled, into 64-bit sums.
// ---------------------------------------------------------------------------
constexpr int SPLIT_BITS = 7;

// GB300's FP64 pipe is narrow, so the splitting below works on the bit
// patterns of the FP64 inputs.

// two consecutive values (an even offset into a matrix's values); wide: the
// values start on a 16-byte boundary (a caller's own array may start on any
// multiple of eight)
__device__ __forceinline__ double2 load_pair(const double* p, bool wide) {
  if (wide) return *reinterpret_cast<const double2*>(p);
  return make_double2(p[0], p[1]);
}

// blocks whose values one thread may add up in FP32 (row_bounds)
constexpr int ROW_BLOCKS = 32;

// x 2^k in FP32, k of any size (sums are non-negative; too large: infinity)
__device__ __forceinline__ float scale_f32(float x, int k) {
  return x == 0.0f ? 0.0f : ldexpf(x, max(-2000, min(2000, k)));
}

// What a thread has seen of a row: the largest |x| by its high word, the low
// words' bits (for rows of subnormals), and the sums of |x| and x^2 in FP32
// relative to 2^(ref - 896), off the narrow FP64 pipe (one FP64 FMA per
// element for the squares held this kernel at 2.0 TB/s).  ref follows the
// values: one above 2^32 of the reference becomes the new one (rare after the
// first nonzero value).  Values below 2^-126 of the reference (2^-63 for the
// squares) add nothing, which row_bounds makes up for.
struct RowScale {
  uint32_t hi = 0, lo = 0, top = 0;
  int ref = 0;  // subtracted from the FP64 exponent field
  float l1 = 0.0f, sq = 0.0f;
  __device__ __forceinline__ void add(double x) {
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu, l = (uint32_t)__double2loint(x);
    if (h > top) {
      const int r = max((int)(h >> 20) - 127, 0);
      l1 = scale_f32(l1, ref - r);
      sq = scale_f32(sq, 2 * (ref - r));
      ref = r;
      top = (uint32_t)(r + 127 + 32) << 20;
    }
    hi = h > hi ? h : hi;
    lo |= l;
    const int t = (int)h - ref * (1 << 20);
    // the FP32 pattern: exponent field moved by ref, 23 of the 52 fraction bits
    float f = __uint_as_float(__funnelshift_l(l, (uint32_t)t, 3));
    if (t < (1 << 20)) f = 0.0f;
    l1 += f;
    sq = fmaf(f, f, sq);
  }
};

// exponent e of a row whose largest magnitude has these words: |x| < 2^e
__device__ __forceinline__ int row_exponent(uint32_t hi, uint32_t lo) {
  const int ea = (int)(hi >> 20);
  if (ea > 0) return ea - 1022;                        // [2^(ea-1023), 2^(ea-1022))
  if (hi != 0) return (64 - __clz((int)hi)) - 1074;    // subnormal: [2^(L-1075), 2^(L-1074))
  return lo != 0 ? 32 - __clz((int)lo) - 1074 : 0;
}

// the row's scaled 1- and 2-norm bounds from its sums relative to 2^e, as FP32 bits
__device__ __forceinline__ void row_bounds(bool any, int e, float l1, float sq, int nscalars, uint32_t& n1, uint32_t& n2) {
  n1 = n2 = 0u;
  if (!any) return;
  if (e < -800) {  // the reference stops at the smallest exponents: no bound
    n1 = n2 = __float_as_uint(3.0e38f);
    return;
  }
  // The sums decide how many bits the fixed-point sums of a product keep, so
  // the bounds are tight: magnitudes are truncated to 24 bits (1.2e-7), a thread
  // adds at most ROW_BLOCKS blocks (1024 values: 6.1e-5 of the squares' sum,
  // 3.1e-5 of its root), and the few partial sums that follow add 1e-6; 5e-5
  // covers them.  (The 1-norm's like share is within the margin its user adds.)
  // Values left out of a sum are below 2^-126 (2^-63 for the squares) of a
  // value of the row.
  n1 = __float_as_uint(fminf(l1 + (float)nscalars * 1.2e-38f, 3.0e38f));
  n2 = __float_as_uint(fminf(sqrtf(sq + (float)nscalars * 1.2e-38f) * 1.00005f + 1e-30f, 3.0e38f));
}

// the warp's largest norm bounds, one atomic each (32 rows' atomics on one
// word would queue up)
__device__ __forceinline__ void row_scale_max(uint32_t n1, uint32_t n2, unsigned int* l1max, unsigned int* l2max) {
  n1 = __reduce_max_sync(0xffffffffu, n1);
  n2 = __reduce_max_sync(0xffffffffu, n2);
  if ((threadIdx.x & 31) == 0 && n1) {
    atomicMax(l1max, n1);
    atomicMax(l2max, n2);
  }
}

// Row scales of a view: the exponent e of sigma = 2^e for every scalar row of op(X),
// max_k |x_rk| = m 2^e with m in [0.5, 1) (e = 0 for an all-zero row), the largest
// scaled 1-norm sum_k |x_rk| / sigma of a row into *l1max and the largest scaled
// 2-norm into *l2max, both as FP32 bits.  While the block rows are short, CTA I reads block row I
// (k_row_scale); else CTA c the view's blocks [c L, (c + 1) L), row by row
// (k_row_parts).  16-byte loads; TR: op(X) row r is column r of the stored blocks, a
// thread takes two columns and every (512 / B)-th row; else eight lanes share a
// row in segments of 128 bytes.  The sums of each block row it meets go to
// `part`, and k_row_scale_join adds a row's parts in order, so no long row is one
// CTA's alone.  Measured: 3D cluster factor of 4096 rows (64 block rows of 64
// blocks) 896 -> 39 us (one CTA of 64 threads per block row before), 262,144-row
// chain (4096 block rows of three, 400 MB) 212 -> 101 us, rows stored as rows
// 486 -> 92 us; a product A^T B, bs 64, of 2000 block rows of three and one full
// block column of A 17.9 -> 1.5 ms in all (one CTA of 256 threads per block row
// before).
struct RowPart {
  uint32_t hi, lo;
  int e;  // l1 and sq relative to 2^e and 2^2e
  float l1, sq;
};

template <int B, bool TR>
constexpr int row_scale_smem() { return (TR ? 512 / B : 8) * B * (int)sizeof(RowScale); }

// the sums of op() row threadIdx.x (< B; the others' result is meaningless)
// over the view's blocks qa .. qe - 1, by the whole CTA
template <int B, bool TR>
__device__ __forceinline__ RowPart row_scale_part(const int32_t* __restrict__ src, int qa, int qe,
                                                  const double* __restrict__ val, bool wide, uint8_t* smem) {
  constexpr int RG = TR ? 512 / B : 8;  // threads that share a row of op(X)
  RowScale(*sh)[B] = reinterpret_cast<RowScale(*)[B]>(smem);
  const int tid = threadIdx.x;
  if constexpr (TR) {
    const int c = (tid % (B / 2)) * 2, r0 = tid / (B / 2);
    RowScale a0, a1;
    for (int q = qa; q < qe; ++q) {
      const double* blk = val + (size_t)(src ? src[q] : q) * B * B + c;
#pragma unroll 8
      for (int k = r0; k < B; k += RG) {
        const double2 x = load_pair(blk + k * B, wide);
        a0.add(x.x);
        a1.add(x.y);
      }
    }
    sh[r0][c] = a0;
    sh[r0][c + 1] = a1;
  } else {
    const int wid = tid >> 5, lane = tid & 31;
    constexpr int RS = B / 32;  // groups of four rows per warp
    RowScale a[RS];
    for (int q = qa; q < qe; ++q) {
      const double* blk = val + (size_t)(src ? src[q] : q) * B * B + (lane & 7) * 2;
#pragma unroll
      for (int g = 0; g < RS; ++g) {
        const double* row = blk + ((wid * RS + g) * 4 + (lane >> 3)) * B;
#pragma unroll
        for (int i = 0; i < B; i += 16) {
          const double2 x = load_pair(row + i, wide);
          a[g].add(x.x);
          a[g].add(x.y);
        }
      }
    }
#pragma unroll
    for (int g = 0; g < RS; ++g) sh[lane & 7][(wid * RS + g) * 4 + (lane >> 3)] = a[g];
  }
  __syncthreads();
  RowPart t{0u, 0u, 0, 0.0f, 0.0f};
  if (tid < B) {
#pragma unroll
    for (int g = 0; g < RG; ++g) {
      t.hi = max(t.hi, sh[g][tid].hi);
      t.lo |= sh[g][tid].lo;
    }
    t.e = row_exponent(t.hi, t.lo);
#pragma unroll
    for (int g = 0; g < RG; ++g) {  // a sum's unit is 2^(ref + 127 - 1023)
      const int k = sh[g][tid].ref - 896 - t.e;
      t.l1 += scale_f32(sh[g][tid].l1, k);
      t.sq += scale_f32(sh[g][tid].sq, 2 * k);
    }
  }
  __syncthreads();  // (the caller may use smem again)
  return t;
}

template <int B, bool TR>
__global__ void __launch_bounds__(256) k_row_scale(const int32_t* __restrict__ rp, const int32_t* __restrict__ src,
                                                   const double* __restrict__ val, bool wide, int* __restrict__ eout,
                                                   unsigned int* __restrict__ l1max, unsigned int* __restrict__ l2max) {
  __shared__ __align__(16) uint8_t sh[row_scale_smem<B, TR>()];
  const int I = (int)blockIdx.x, tid = threadIdx.x, q0 = rp[I], q1 = rp[I + 1];
  const RowPart t = row_scale_part<B, TR>(src, q0, q1, val, wide, sh);
  if (tid >= B) return;
  uint32_t n1, n2;
  eout[(size_t)I * B + tid] = t.e;
  row_bounds((t.hi | t.lo) != 0u, t.e, t.l1, t.sq, (q1 - q0) * B, n1, n2);
  row_scale_max(n1, n2, l1max, l2max);
}

// part[(c + I) B + r]: CTA c's sums of row r of block row I (c + I grows from
// each segment to the next, so no two share a place)
template <int B, bool TR>
__global__ void __launch_bounds__(256) k_row_parts(const int32_t* __restrict__ rp, const int32_t* __restrict__ src,
                                                   int nb, int nblk, int L, const double* __restrict__ val, bool wide,
                                                   RowPart* __restrict__ part) {
  __shared__ __align__(16) uint8_t sh[row_scale_smem<B, TR>()];
  const int c = (int)blockIdx.x, qe = min((c + 1) * L, nblk), lane = threadIdx.x & 31;
  int I = 0, end = nb;  // the row that holds block c L: the last with rp[I] <= c L
  while (end - I > 1) {  // (every warp by itself, 32 probes at a time)
    const int step = (end - I + 31) / 32, p = I + lane * step;
    const unsigned m = __ballot_sync(0xffffffffu, p < end && rp[p] <= c * L);
    I += (31 - __clz((int)m)) * step;  // (probe 0 holds)
    end = min(end, I + step);
  }
  for (int q = c * L; q < qe; ++I) {
    const int q1 = min(rp[I + 1], qe);
    if (q1 <= q) continue;  // an empty row
    const RowPart t = row_scale_part<B, TR>(src, q, q1, val, wide, sh);
    if (threadIdx.x < B) part[(size_t)(c + I) * B + threadIdx.x] = t;
    q = q1;
  }
}

// the parts of every row joined, in order (nrows is a multiple of 32)
__global__ void k_row_scale_join(const int32_t* __restrict__ rp, int bs, int64_t nrows, int L,
                                 const RowPart* __restrict__ part, int* __restrict__ eout,
                                 unsigned int* __restrict__ l1max, unsigned int* __restrict__ l2max) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= nrows) return;
  const int I = (int)(r / bs), q0 = rp[I], q1 = rp[I + 1];
  const int c0 = q0 / L, n = q1 > q0 ? (q1 - 1) / L - c0 + 1 : 0;
  const RowPart* p = part + (size_t)(c0 + I) * bs + r % bs;
  uint32_t hi = 0, lo = 0;
#pragma unroll 8
  for (int s = 0; s < n; ++s) {
    hi = max(hi, p[(size_t)s * bs].hi);
    lo |= p[(size_t)s * bs].lo;
  }
  const int e = row_exponent(hi, lo);
  float l1 = 0.0f, sq = 0.0f, rest = 0.0f;  // (a row may have thousands of parts: what each add of squares loses is kept)
#pragma unroll 4
  for (int s = 0; s < n; ++s) {
    const RowPart t = p[(size_t)s * bs];
    l1 += scale_f32(t.l1, t.e - e);
    const float y = scale_f32(t.sq, 2 * (t.e - e)) - rest, z = sq + y;
    rest = (z - sq) - y;
    sq = z;
  }
  uint32_t n1, n2;
  eout[r] = e;
  row_bounds((hi | lo) != 0u, e, l1, sq, (q1 - q0) * bs, n1, n2);
  row_scale_max(n1, n2, l1max, l2max);
}

// Whether one CTA for each block row will do: the longest row (-1: not known)
// holds no more blocks than a quarter of an SM's share of them all, or 16, and
// no more than a thread may add up.
static bool rows_short(int nb, int64_t nnzb, int longest) {
  return (longest < 0 ? nb : longest) <= std::min<int64_t>(ROW_BLOCKS, std::max<int64_t>(16, nnzb / (4 * 152)));
}

// sigma exponents (and the scaled norm bounds) of the rows of a row view of nnzb blocks
static void row_scales(ifac_ctx* ctx, int bs, const int32_t* rp, const int32_t* src, int nb, int64_t nnzb, int longest,
                       bool tr, const double* val, int* eout, unsigned int* l1max, unsigned int* l2max) {
  const bool wide = aligned16(val);
  const auto pick = [&](auto k32t, auto k32, auto k64t, auto k64, auto k128t, auto k128, auto go) {
    if (bs == 32) tr ? go(k32t) : go(k32);
    else if (bs == 64) tr ? go(k64t) : go(k64);
    else tr ? go(k128t) : go(k128);
  };
  // (block rows of four blocks and more are shared out as well while they are
  // fewer than four a SM: batch of eight members of 8 to 16 full block rows, BF16,
  // 9.5 ms with one CTA a row, 9.0 shared out)
  if (rows_short(nb, nnzb, longest) && (nb >= 4 * 152 || nnzb < 4 * (int64_t)nb)) {
    pick(k_row_scale<32, true>, k_row_scale<32, false>, k_row_scale<64, true>, k_row_scale<64, false>,
         k_row_scale<128, true>, k_row_scale<128, false>, [&](auto kernel) {
           kernel<<<nb, 256, 0, ctx->stream>>>(rp, src, val, wide, eout, l1max, l2max);
           IFAC_CK_LAUNCH();
         });
    return;
  }
  // about four CTAs per SM, each with 2 to ROW_BLOCKS blocks
  const int64_t rows = (int64_t)nb * bs;
  const int L = (int)std::max<int64_t>(2, std::min<int64_t>(ROW_BLOCKS, nnzb / (4 * 152)));
  const int grid = cdiv(std::max<int64_t>(nnzb, 1), L);
  Buf<RowPart> part(ctx, (size_t)(grid + nb) * bs);
  pick(k_row_parts<32, true>, k_row_parts<32, false>, k_row_parts<64, true>, k_row_parts<64, false>,
       k_row_parts<128, true>, k_row_parts<128, false>, [&](auto kernel) {
         kernel<<<grid, 256, 0, ctx->stream>>>(rp, src, nb, (int)nnzb, L, val, wide, part.p);
         IFAC_CK_LAUNCH();
       });
  k_row_scale_join<<<cdiv(rows, 128), 128, 0, ctx->stream>>>(rp, bs, rows, L, part.p, eout, l1max, l2max);
  IFAC_CK_LAUNCH();
}

// NS BF16 slice copies (K-major, op() CSR order) of a view; row r of a block
// has a scale exponent e (|x| < 2^e).  With Y = x 2^(62 - e) held as a 64-bit
// integer (|Y| < 2^62; bits below 2^-62 of sigma dropped by rounding) and
// R_k = Y rounded (half up) to a multiple of 2^(62 - 7k), the digits up to k
// sum to R_k.  Three digits at a time, c = R_(k+3) - 2^21 R_k is a 22-bit
// integer (32-bit arithmetic on the low words suffices), whose digits q
// (|q| <= 64, the first 128) FP32 arithmetic separates exactly: an integer
// unit result is half the rate of an FP32 one, and digit by digit the integers
// were what bounded this kernel (60 operations a value).
//
// Four values of one row, slices k0 .. k0 + N - 1 from the digits in c.
template <int N>
__device__ __forceinline__ void put_digits(const int (&c)[4], int k0, __nv_bfloat16* dst, size_t slice_stride) {
  constexpr float M = 12582912.0f;  // 1.5 2^23: adding it rounds to an integer
  float q[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    // (half a unit more, so that ties round up, as the R_k do)
    float f = (__int_as_float(0x4B400000 + c[i]) - M) + 0.5f;
    if (N == 3) {
      q[0][i] = fmaf(f, 0x1p-14f, M) - M;
      f = fmaf(-0x1p14f, q[0][i], f);
    }
    if (N >= 2) {
      q[N - 2][i] = fmaf(f, 0x1p-7f, M) - M;
      f = fmaf(-0x1p7f, q[N - 2][i], f);
    }
    q[N - 1][i] = f - 0.5f;
  }
#pragma unroll
  for (int k = 0; k < N; ++k) {  // integers up to 128: the upper half of their FP32 pattern is exact
    uint2 w;
    w.x = __byte_perm(__float_as_uint(q[k][0]), __float_as_uint(q[k][1]), 0x7632);
    w.y = __byte_perm(__float_as_uint(q[k][2]), __float_as_uint(q[k][3]), 0x7632);
    *reinterpret_cast<uint2*>(dst + (size_t)(k0 + k) * slice_stride) = w;
  }
}

__device__ __forceinline__ void split4(const double (&x)[4], int e, int ns, __nv_bfloat16* dst, size_t slice_stride) {
  long long y[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t h = (uint32_t)__double2hiint(x[i]), l = (uint32_t)__double2loint(x[i]);
    const int ea = (int)((h >> 20) & 0x7ffu);
    const uint32_t m = (h & 0xfffffu) | (ea ? 0x100000u : 0u);
    // |x| = mant 2^(max(ea, 1) - 1075), |Y| = mant 2^9 2^-t, t >= 0 since |x| < 2^e
    const int t = 1022 + e - max(ea, 1);
    const unsigned long long v = ((unsigned long long)__funnelshift_l(l, m, 9) << 32) | (l << 9);
    const unsigned long long half = t > 0 ? 1ull << ((t - 1) & 63) : 0ull;
    const unsigned long long Y = t > 62 ? 0ull : (v + half) >> (t & 63);
    y[i] = (h >> 31) ? -(long long)Y : (long long)Y;
  }
  int r3[4], c[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] = r3[i] = (int)((y[i] + (1ll << 40)) >> 41);  // (ns >= 3)
  put_digits<3>(c, 0, dst, slice_stride);
  if (ns == 3) return;
  // digits 4 .. k2, k2 = min(ns, 6)
  const int n2 = min(ns, 6) - 3, d2 = 41 - 7 * n2;
  int r6[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    r6[i] = (int)((y[i] + (1ll << (d2 - 1))) >> d2);
    c[i] = (int)((uint32_t)r6[i] - ((uint32_t)r3[i] << (7 * n2)));
  }
  if (n2 == 3) put_digits<3>(c, 3, dst, slice_stride);
  else if (n2 == 2) put_digits<2>(c, 3, dst, slice_stride);
  else put_digits<1>(c, 3, dst, slice_stride);
  if (ns <= 6) return;
  const int n3 = ns - 6, d3 = 20 - 7 * n3;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    c[i] = (int)((uint32_t)((y[i] + (1ll << (d3 - 1))) >> d3) - ((uint32_t)r6[i] << (7 * n3)));
  if (n3 == 2) put_digits<2>(c, 6, dst, slice_stride);
  else put_digits<1>(c, 6, dst, slice_stride);
}

// the slices of one stored block s (the whole CTA, 256 threads); se: the scale
// exponents of its op() rows.  TR: op() row r is column r of the stored block,
// moved through shared memory in tiles of 64 x 64, whose columns are permuted
// by their row so that neither side meets bank conflicts.
template <int B, bool TR>
__device__ __forceinline__ void split_block(const double* __restrict__ s, bool wide, const int* se, int ns,
                                            __nv_bfloat16* __restrict__ d, size_t slice_stride, double* tile) {
  double x[4];
  if constexpr (!TR) {
#pragma unroll 2
    for (int e = (int)threadIdx.x * 4; e < B * B; e += 1024) {
      load4(s + e, x, wide);
      split4(x, se[e / B], ns, d + e, slice_stride);
    }
  } else {
    constexpr int TS = B < 64 ? B : 64;
    const auto at = [](int r, int c) { return r * TS + (c ^ ((r >> 2) & 15)); };
    for (int ti = 0; ti < B / TS; ++ti)
      for (int tj = 0; tj < B / TS; ++tj) {
#pragma unroll
        for (int e = (int)threadIdx.x * 4; e < TS * TS; e += 1024) {
          const int r = e / TS, c = e % TS;
          load4(s + (size_t)(ti * TS + r) * B + tj * TS + c, x, wide);
#pragma unroll
          for (int i = 0; i < 4; ++i) tile[at(r, c + i)] = x[i];
        }
        __syncthreads();
#pragma unroll 2
        for (int e = (int)threadIdx.x * 4; e < TS * TS; e += 1024) {
          const int r = e / TS, c = e % TS;  // op() row tj TS + r, columns ti TS + c ..
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i] = tile[at(c + i, r)];
          split4(x, se[tj * TS + r], ns, d + (size_t)(tj * TS + r) * B + ti * TS + c, slice_stride);
        }
        __syncthreads();
      }
  }
}

// the zero block of every slice
__device__ __forceinline__ void split_zero(int bsz, int ns, __nv_bfloat16* __restrict__ d, size_t slice_stride) {
  for (int k = 0; k < ns; ++k)
    for (int e = threadIdx.x; e < bsz / 2; e += blockDim.x)
      *reinterpret_cast<uint32_t*>(d + (size_t)k * slice_stride + 2 * e) = 0u;
}

// Slices with the scales at hand; the block qb of the view has the exponents
// sexp[sblk[qb] * B ..].
template <int B, bool TR>
__global__ void __launch_bounds__(256) k_split(const double* __restrict__ val, bool wide,
                                               const int32_t* __restrict__ src, int64_t nblk,
                                               const int32_t* __restrict__ sblk, const int* __restrict__ sexp, int ns,
                                               __nv_bfloat16* __restrict__ dst) {
  constexpr int BSZ = B * B, TS = B < 64 ? B : 64;
  __shared__ double tile[TR ? TS * TS : 1];
  const size_t slice_stride = (size_t)(nblk + 1) * BSZ;
  for (int64_t qb = blockIdx.x; qb <= nblk; qb += gridDim.x) {
    __nv_bfloat16* d = dst + (size_t)qb * BSZ;
    if (qb == nblk) split_zero(BSZ, ns, d, slice_stride);
    else
      split_block<B, TR>(val + (size_t)(src ? src[qb] : qb) * BSZ, wide, sexp + (size_t)sblk[qb] * B, ns, d,
                         slice_stride, tile);
  }
}

// Scales and slices in one kernel for short block rows (a banded operand): CTA
// I finds the scales of the op() rows of view row I, then reads the row's
// blocks again, from L2, for their slices, so that HBM sees the values once:
// 280 us for the 262,144-row chain with 5 to 7 slices (1.0 - 1.1 GB), 485 us in
// two kernels before.
// out (nullable): the copy index of each view entry, else its position.
template <int B, bool TR>
__global__ void __launch_bounds__(256) k_split_rows(const int32_t* __restrict__ rp, const int32_t* __restrict__ src,
                                                    const int32_t* __restrict__ out, int nb, int64_t nblk,
                                                    const double* __restrict__ val, bool wide, int ns,
                                                    int* __restrict__ eout, unsigned int* __restrict__ l1max,
                                                    unsigned int* __restrict__ l2max,
                                                    __nv_bfloat16* __restrict__ dst) {
  constexpr int BSZ = B * B, TS = B < 64 ? B : 64;
  constexpr int SH = row_scale_smem<B, TR>();
  constexpr int TILE = TR ? TS * TS * (int)sizeof(double) : 8;
  __shared__ __align__(16) uint8_t sh[SH > TILE ? SH : TILE];
  __shared__ int se[B];
  const size_t slice_stride = (size_t)(nblk + 1) * BSZ;
  const int I = blockIdx.x;
  if (I == nb) {
    split_zero(BSZ, ns, dst + (size_t)nblk * BSZ, slice_stride);
    return;
  }
  const int q0 = rp[I], q1 = rp[I + 1];
  const RowPart t = row_scale_part<B, TR>(src, q0, q1, val, wide, sh);
  if (threadIdx.x < B) {
    uint32_t n1, n2;
    se[threadIdx.x] = t.e;
    eout[(size_t)I * B + threadIdx.x] = t.e;
    row_bounds((t.hi | t.lo) != 0u, t.e, t.l1, t.sq, (q1 - q0) * B, n1, n2);
    row_scale_max(n1, n2, l1max, l2max);
  }
  __syncthreads();
  for (int q = q0; q < q1; ++q) {
    const int sb = src ? src[q] : q;
    split_block<B, TR>(val + (size_t)sb * BSZ, wide, se, ns, dst + (size_t)(out ? out[q] : q) * BSZ, slice_stride,
                       reinterpret_cast<double*>(sh));
  }
}

template <int B, bool TR>
static void launch_split(ifac_ctx* ctx, const double* val, const int32_t* src, int64_t nblk, const int32_t* sblk,
                         const int* sexp, int ns, void* dst) {
  const int grid = (int)std::min<int64_t>(nblk + 1, 152 * 16);
  k_split<B, TR><<<grid, 256, 0, ctx->stream>>>(val, aligned32(val), src, nblk, sblk, sexp, ns,
                                                reinterpret_cast<__nv_bfloat16*>(dst));
  IFAC_CK_LAUNCH();
}

static void split_blocks(ifac_ctx* ctx, int bs, const double* val, const int32_t* src, int64_t nblk, bool tr,
                         const int32_t* sblk, const int* sexp, int ns, void* dst) {
  if (bs == 32) tr ? launch_split<32, true>(ctx, val, src, nblk, sblk, sexp, ns, dst)
                   : launch_split<32, false>(ctx, val, src, nblk, sblk, sexp, ns, dst);
  else if (bs == 64) tr ? launch_split<64, true>(ctx, val, src, nblk, sblk, sexp, ns, dst)
                        : launch_split<64, false>(ctx, val, src, nblk, sblk, sexp, ns, dst);
  else tr ? launch_split<128, true>(ctx, val, src, nblk, sblk, sexp, ns, dst)
          : launch_split<128, false>(ctx, val, src, nblk, sblk, sexp, ns, dst);
}

// Scales and slices of a view (rows rp, blocks src of nblk) in one launch, when
// its block rows are short and many enough for one CTA each; false where the
// two kernels are to be used.  A CTA takes 4 to 6 us for a block of 64, so none
// may get a long row (rows_short): S S with one full block row among 2000 of
// three blocks took 16.0 ms in one kernel and takes 1.5 ms in two.
static bool split_rows_sizes(int nb, int64_t nblk) { return nb >= 2 * 152 && nblk <= 8 * (int64_t)nb; }

static bool split_rows(ifac_ctx* ctx, int bs, const int32_t* rp, const int32_t* src, const int32_t* out, int nb,
                       int64_t nblk, int longest, bool tr, const double* val, int ns, int* eout, unsigned int* l1max,
                       unsigned int* l2max, void* dst) {
  if (!split_rows_sizes(nb, nblk) || !rows_short(nb, nblk, longest)) return false;
  __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(dst);
  const bool wide = aligned32(val);
  const auto go = [&](auto kernel) {
    kernel<<<nb + 1, 256, 0, ctx->stream>>>(rp, src, out, nb, nblk, val, wide, ns, eout, l1max, l2max, d);
    IFAC_CK_LAUNCH();
  };
  if (bs == 32) tr ? go(k_split_rows<32, true>) : go(k_split_rows<32, false>);
  else if (bs == 64) tr ? go(k_split_rows<64, true>) : go(k_split_rows<64, false>);
  else tr ? go(k_split_rows<128, true>) : go(k_split_rows<128, false>);
  return true;
}

// x 2^E rounded to nearest (ties to even), built from the integer's bits;
// results outside the normal range take the FP64 pipe
__device__ __forceinline__ double i64_ldexp(long long x, int E) {
  if (x == 0) return 0.0;
  const unsigned long long sgn = x < 0 ? (1ull << 63) : 0ull;
  const unsigned long long ux = x < 0 ? (unsigned long long)(-x) : (unsigned long long)x;
  int len = 64 - __clzll((long long)ux);
  unsigned long long mant;
  if (len > 53) {
    const int sh = len - 53;
    mant = ux >> sh;
    const unsigned long long rem = ux & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (mant & 1ull))) {
      if (++mant == (1ull << 53)) {
        mant >>= 1;
        ++len;
      }
    }
  } else {
    mant = ux << (53 - len);
  }
  const int field = len - 1 + E + 1023;  // value = mant 2^(len - 53 + E), mant in [2^52, 2^53)
  if (field < 1 || field > 2046) return (double)x * ldexp(1.0, E);
  return __longlong_as_double((long long)(sgn | ((unsigned long long)field << 52) | (mant & 0xfffffffffffffull)));
}

// C_IJ = S_int 2^(e_i + e_j + ea) * am from the fixed-point sums of the
// split kernel (alpha = am 2^ea; am = +-1 when alpha is a signed power of
// two): coalesced reads in hand-over order, a transpose through shared
// memory, row-major FP64 writes, then the FP64 block norms
__global__ void __launch_bounds__(256) k_split_finish(const int32_t* __restrict__ crow,
                                                      const int32_t* __restrict__ cci, int64_t nnzb,
                                                      const longlong2* __restrict__ part, double* __restrict__ cval,
                                                      const int* __restrict__ sige, const int* __restrict__ taue,
                                                      int ea, double am, double* __restrict__ cnorm) {
  __shared__ double tile[BS][BS + 1];
  __shared__ double red[8];
  const bool unit = (am == 1.0 || am == -1.0);
  for (int64_t p = blockIdx.x; p < nnzb; p += gridDim.x) {
    const int I = crow[p], J = cci[p];
    const longlong2* src = part + (size_t)p * (BS * BS / 2);
    for (int i = threadIdx.x; i < BS * BS / 2; i += blockDim.x) {
      const int lane = i & 31, e = (i >> 5) & 15, h = (i >> 9) & 1, qq = i >> 10;
      const int r = qq * 32 + lane, col = h * 32 + 2 * e;
      longlong2 x = src[i];
      if (unit && am < 0.0) {
        x.x = -x.x;
        x.y = -x.y;
      }
      const int er = ea + sige[(size_t)I * BS + r];
      double v0 = i64_ldexp(x.x, er + taue[(size_t)J * BS + col]);
      double v1 = i64_ldexp(x.y, er + taue[(size_t)J * BS + col + 1]);
      if (!unit) {
        v0 *= am;
        v1 *= am;
      }
      tile[r][col] = v0;
      tile[r][col + 1] = v1;
    }
    __syncthreads();
    double* c = cval + (size_t)p * BS * BS;
    double ss = 0.0;
    for (int k = threadIdx.x; k < BS * BS; k += blockDim.x) {
      const double v = tile[k / BS][k % BS];
      c[k] = v;
      ss = fma(v, v, ss);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) red[wid] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += red[w];
      cnorm[p] = sqrt(t);
    }
  }
}

// ---------------------------------------------------------------------------
// Split products on narrow tiles (bs 32, 64, 128).  A tile is 128 x 64
// accumulator elements: 128 / bs block rows of C by 64 columns (two block
// columns at bs 32, one at bs 64, half of one at bs 128, whose two halves the
// same CTA takes one after the other).  Each K block is streamed in chunks of
// at most 64 K elements; a chunk's op(B) slices are resident while its op(A)
// slices stream through a ring.  Every weight class a + b has one FP32
// accumulator in tensor memory (up to 8 classes x 64 columns), side by side,
// as the op(B) slices lie one after the other in shared memory: op(A) slice a
// meets op(B) slices b .. b + 3 in one instruction of 256 columns, whose
// accumulators are the classes a + b .. a + b + 3.  (One instruction of 64
// columns per pair read op(A) from shared memory for every pair: 36 pairs of
// an 8-slice product 4.6 -> 2.9 ms a launch on a 4096-row 3D cluster factor,
// 53% of the measured BF16 rate, and 0.95 ms a launch where it was 1.19 on
// the 262,144-row chain.)  A window of K blocks is as long as every class
// stays exact; after each window the epilogue adds the classes, scaled, into
// 64-bit fixed-point sums held in registers, so a tile may span any number of
// windows.  After the tile's last window the epilogue writes
// S_ij 2^(ea + e_i + e_j) * am in FP64 and the block norms.
// ---------------------------------------------------------------------------
namespace band {
constexpr int MAX_U = 8;                    // weight classes (one unit each): 8 x 64 = 512 columns
// 16 epilogue warps, four per tensor-memory lane quarter, each on 16 of the
// tile's 64 columns: the epilogue's reads of the classes stand between the
// MMAs of consecutive windows (the accumulators fill tensor memory, so they
// are not double-buffered).  Cycles a tile on the 262,144-row chain (two K
// blocks a tile on average): classes into the sums 9.0k -> 4.8k, FP64 result
// and norm 8.7k -> 7.0k, against 10.5k of MMAs; what is left between the MMAs
// and the tensor rate is the op(A) and op(B) traffic from L2 (about 40 bytes
// a clock and SM).
constexpr int EPW = 16;
constexpr int NTB = 32 * (2 + EPW);
constexpr uint32_t TMEM_COLS = 512;
// FP32 accumulate, A = B = BF16, both K-major, M = 128; N is added per
// instruction (64 to 256 columns)
constexpr uint32_t IDESC0 = idesc_of<2, 0, 128>();

template <int B>
struct SB {
  static constexpr int M = 128, N = 64;
  static constexpr int TMB = M / B;                 // block rows per tile (4, 2, 1)
  static constexpr int TNB = B <= N ? N / B : 1;    // block columns per tile (2, 1, 1)
  static constexpr int NSUB = B > N ? B / N : 1;    // column sub-tiles per block column (1, 1, 2)
  static constexpr int BROWS = B < N ? B : N;       // rows of one op(B) box (32, 64, 64)
  // K chunks of 64 elements (32 at bs 32); halving them at bs 64 and 128 was
  // measured slower: the per-slot waits, copies and commits double while the
  // products stay the same
  static constexpr int KC = B < 64 ? B : 64;        // K elements per chunk
  static constexpr int KCH = B / KC;                // chunks per K block (1, 1, 2)
  static constexpr int ATOM = KC * 2;               // bytes of one BF16 row chunk: one swizzle atom (64 or 128)
  static constexpr int SLOT_A = M * ATOM;           // one slice of the tile's op(A) rows: 8, 16, 16 KB
  static constexpr int SLOT_B = N * ATOM;           // one slice of its op(B) columns: 4, 8, 8 KB
  static constexpr int MAXS = 8;                    // slices per operand at most
  // every op(B) slice of a chunk stays in one of two buffers while the op(A)
  // slices stream through a ring: slice a of op(A) meets slices 0 .. ns-1-a
  // of op(B), and its slot is released as soon as those products are issued
  static constexpr int B_BUF = MAXS * SLOT_B;
  static constexpr int RA_FIT = (216 * 1024 - 2 * B_BUF) / SLOT_A;
  static constexpr int RA = RA_FIT < 16 ? RA_FIT : 16;  // op(A) ring slots: 16, 5, 5
  static constexpr int SMEM_BYTES = 2 * B_BUF + RA * SLOT_A + 1024;
  static constexpr int KSTEPS = ATOM / 32;          // MMAs per slice pair and chunk
  static constexpr uint32_t SBO = 8 * ATOM;
  static constexpr uint32_t SWZ = ATOM == 128 ? 2 : 4;
  static constexpr int RECW = TMB + TNB;
  static_assert(SLOT_A % 1024 == 0 && SLOT_B % 1024 == 0, "slots must keep the swizzle alignment");
  static_assert(RA >= 2, "op(A) ring too shallow");
};

// The 64-bit sums of a tile hold units of 2^-f: 2^d of the weight class that
// lies in slot 6; `below` classes of lower weight round into it.
struct FixedSum {
  int below;         // classes below the one that holds the unit
  int d;             // the unit is 2^d of that class, 0 <= d < 7
  float m0, m1, m2;  // 2^-d, 2^(7 - d), 2^(14 - d)
  int s1;            // 21 - d
  int top;           // 2^(10 - d)
  long long offset;  // what class_sums adds beside the classes
};
}  // namespace band

struct BandArgs {
  const int32_t* tiles;    // [2t] tile row (of TMB block rows), [2t+1] tile column (of TNB block columns)
  const int* ntiles;       // device: number of tiles
  const int* tile_nk;      // device: K blocks of each tile
  const int32_t* rec;      // plan: per K block, copy indices of the tile's op(A)_IK, then op(B)_KJ
  const int32_t* rec_off;  // first record of each tile
  const int32_t* cpos;     // per tile, the C positions of its TMB x TNB blocks (-1: not in C)
  double* cval;            // C's values and block norms (FP64)
  double* cnorm;
  const int* sige;         // scale exponents of the scalar rows of op(A) and columns of op(B)
  const int* taue;
  int ea;                  // C_ij = S_ij 2^(ea + e_i + e_j) * am, S_ij the 64-bit fixed-point sum
  double am;               // +-1 (applied to the integer) or the mantissa of alpha
  int nb;
  int ns;                  // slices per operand (1..8)
  int kwin;                // K blocks per window (every weight class exact in one FP32 accumulator)
  int slice_rows_a;        // tensor-map rows between consecutive slices of op(A): (nnzb_A + 1) bs
  int slice_rows_b;
  band::FixedSum fx;       // how the weight classes enter the 64-bit sums
  bool wide;               // C's values start on a 32-byte boundary
  int* err;
  int* ovf;
};

// 32 lanes x 4 columns of tensor memory, without waiting for the values
__device__ __forceinline__ void tmem_ld4_issue(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// the loads issued so far have arrived (the registers pass through the wait,
// so that nothing that uses them moves before it)
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[8][4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0][0]), "+r"(r[0][1]), "+r"(r[0][2]), "+r"(r[0][3]), "+r"(r[1][0]), "+r"(r[1][1]),
                 "+r"(r[1][2]), "+r"(r[1][3]), "+r"(r[2][0]), "+r"(r[2][1]), "+r"(r[2][2]), "+r"(r[2][3]),
                 "+r"(r[3][0]), "+r"(r[3][1]), "+r"(r[3][2]), "+r"(r[3][3])::"memory");
  asm volatile(""
               : "+r"(r[4][0]), "+r"(r[4][1]), "+r"(r[4][2]), "+r"(r[4][3]), "+r"(r[5][0]), "+r"(r[5][1]),
                 "+r"(r[5][2]), "+r"(r[5][3]), "+r"(r[6][0]), "+r"(r[6][1]), "+r"(r[6][2]), "+r"(r[6][3]),
                 "+r"(r[7][0]), "+r"(r[7][1]), "+r"(r[7][2]), "+r"(r[7][3])::"memory");
}

// s[e] + the value of one window's classes x[0..7][e] (highest weight first, a
// factor of 2^7 from slot to slot; integers of magnitude at most 2^24, as FP32
// patterns) in units of slot 6 times 2^d, for four columns e side by side: the
// steps of one column depend on each other.  The carries of the classes and
// the digits that remain are formed in FP32, exactly: adding 1.5 2^23 rounds
// to an integer and leaves it in the low bits, so neither the conversion
// instructions (16 per clock and SM, against 125 FP32 operations and 63
// integer ones) nor a 64-bit shift for every class is needed.  Three digits of
// seven bits go into the 64-bit sum at once; the pattern of 1.5 2^23 that
// comes with them is in fx.offset.
__device__ __forceinline__ void class_sums(long long* s, uint32_t (&r)[8][4], const band::FixedSum& fx) {
  constexpr float M = 12582912.0f;
  const auto carry = [](float v) { return fmaf(v, 0.0078125f, 12582912.0f) - 12582912.0f; };  // round(v / 128)
  float c[4] = {0.0f, 0.0f, 0.0f, 0.0f}, g0[4], g1[4];
  if (fx.below) {
    for (int k = 1; k < fx.below; ++k) {  // (more than one class below the unit: rare)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        r[6][e] = __float_as_uint(__uint_as_float(r[6][e]) + carry(__uint_as_float(r[7][e])));
#pragma unroll
        for (int u = 7; u > 0; --u) r[u][e] = r[u - 1][e];
        r[0][e] = 0u;
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) c[e] = carry(__uint_as_float(r[7][e]));
  }
  // slot u: the carry into the next slot in c, the digit returned
  const auto digit = [&](int u, int e) -> float {
    const float v = __uint_as_float(r[u][e]) + c[e];
    c[e] = carry(v);
    return fmaf(-128.0f, c[e], v);
  };
#pragma unroll
  for (int e = 0; e < 4; ++e) g0[e] = digit(6, e);
  if (fx.d) {  // rounded to the unit
#pragma unroll
    for (int e = 0; e < 4; ++e) g0[e] = fmaf(g0[e], fx.m0, M) - M;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) g0[e] = fmaf(digit(5, e), fx.m1, g0[e] + M);
#pragma unroll
  for (int e = 0; e < 4; ++e) g0[e] = fmaf(digit(4, e), fx.m2, g0[e]);
#pragma unroll
  for (int e = 0; e < 4; ++e) g1[e] = digit(3, e) + M;
#pragma unroll
  for (int e = 0; e < 4; ++e) g1[e] = fmaf(digit(2, e), 128.0f, g1[e]);
#pragma unroll
  for (int e = 0; e < 4; ++e) g1[e] = fmaf(digit(1, e), 16384.0f, g1[e]);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const uint32_t top = (uint32_t)__float2int_rn(__uint_as_float(r[0][e]) + c[e]);
    const uint32_t h = __float_as_uint(g1[e]);
    unsigned long long t = (((unsigned long long)(h >> (32 - fx.s1))) << 32) | (h << fx.s1);
    t += __float_as_uint(g0[e]);
    t += (unsigned long long)(top * (uint32_t)fx.top) << 32;
    s[e] = (long long)((unsigned long long)s[e] + t);
  }
}

// v[e] = s[e] 2^E[e] rounded to nearest even from the integer's bits (results
// outside the normal range: i64_ldexp); `bad` records |s| >= 2^62, which the
// sums' scale rules out (s is complete here; its partial sums are not checked)
__device__ __forceinline__ void fixed_to_f64(const long long (&s)[4], const int (&E)[4], double (&v)[4], bool& bad) {
  bool odd = false;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const uint32_t sg = (uint32_t)(s[e] >> 63);  // 0 or all ones
    const uint32_t xl = (uint32_t)s[e] ^ sg, xh = (uint32_t)(s[e] >> 32) ^ sg;
    const unsigned long long u = (((unsigned long long)xh << 32) | xl) + (sg & 1u);
    const uint32_t h = (uint32_t)(u >> 32), l = (uint32_t)u;
    bad |= (h >> 30) != 0u;
    const bool small = h == 0u;
    const uint32_t a = small ? l : h, b = small ? 0u : l;
    const int lz = __clz((int)a);
    const uint32_t nh = __funnelshift_l(b, a, lz), nl = b << (lz & 31);
    const uint32_t mh = nh >> 11, ml = __funnelshift_r(nl, nh, 11);
    const uint32_t up = ((nl & 0x7ffu) + (ml & 1u)) > 0x400u ? 1u : 0u;
    const int ex = E[e] + (small ? 1023 + 62 - 32 : 1023 + 62) - lz;  // exponent field - 1: mh holds the leading bit
    odd |= (unsigned)ex > 2045u;
    const unsigned long long m = (((unsigned long long)(((uint32_t)ex << 20) + mh)) << 32 | ml) + up;
    const uint32_t zero = a == 0u ? 0u : 0xffffffffu;
    v[e] = __hiloint2double((int)(((uint32_t)(m >> 32) | (sg & 0x80000000u)) & zero), (int)((uint32_t)m & zero));
  }
  if (odd) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = i64_ldexp(s[e], E[e]);
  }
}

template <int B>
__global__ void __launch_bounds__(band::NTB, 1)
    k_gemm_split_band(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                      BandArgs args) {
  using namespace band;
  using L = SB<B>;
  constexpr int N = L::N, TMB = L::TMB, TNB = L::TNB, RA = L::RA;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t afull[RA], aempty[RA], bfull[2], bempty[2];
  __shared__ __align__(8) uint64_t acc_full, acc_empty, drain_bar;
  __shared__ uint32_t tmem_base_slot;
  __shared__ volatile int abort_flag;
  __shared__ double partial[2][4][EPW / 4];
  __shared__ int32_t srec[32 * L::RECW];  // the producer's current chunk of plan records

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bbase = smem_base, abase = smem_base + 2u * (uint32_t)L::B_BUF;
  const int ntiles = *args.ntiles;
  const int ns = args.ns;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < RA; ++s) {
      mbar_init(smem_u32(&afull[s]), 1);
      mbar_init(smem_u32(&aempty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&bfull[s]), 1);
      mbar_init(smem_u32(&bempty[s]), 1);
    }
    mbar_init(smem_u32(&acc_full), 1);
    mbar_init(smem_u32(&acc_empty), EPW);  // one arrival per epilogue warp
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
  // this CTA's tiles: blockIdx.x, blockIdx.x + gridDim.x, ...
  const int mt = ntiles > (int)blockIdx.x ? (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;

  if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    // the warp loads the next chunk of plan records while lane 0 issues the
    // copies of the current one (column sub-tile h = the chunk's repetition).
    // Per K chunk: every op(B) slice into the next buffer, then the op(A)
    // slices one ring slot each.
    int slot = 0, bb = 0;
    uint32_t phase = 0, bphase = 0;
    uint32_t issued_mask = 0, last_parity = 0, b_issued = 0, b_parity = 0;
    bool ok = true;
    RecStream<L::RECW> rs;
    rs.init(args.rec, args.rec_off, args.tile_nk, (int)blockIdx.x, (int)gridDim.x, mt, L::NSUB);
    int32_t cur[L::RECW], nxt[L::RECW];
    int c_it, c_rep, c_j0, c_cnt, n_it, n_rep, n_j0, n_cnt;
    bool have = rs.next(lane, cur, c_it, c_rep, c_j0, c_cnt);
    while (have && ok) {
      if (lane < c_cnt) {
#pragma unroll
        for (int w = 0; w < L::RECW; ++w) srec[lane * L::RECW + w] = cur[w];
      }
      __syncwarp();
      const bool nhave = rs.next(lane, nxt, n_it, n_rep, n_j0, n_cnt);
      if (lane == 0) {
        const int h = c_rep;
        for (int j = 0; j < c_cnt && ok; ++j) {
          const int32_t* r = srec + j * L::RECW;
          for (int c = 0; c < L::KCH && ok; ++c) {
            if (!mbar_wait(smem_u32(&bempty[bb]), bphase ^ 1u, &abort_flag, args.err)) {
              ok = false;
              break;
            }
            const uint32_t fbb = smem_u32(&bfull[bb]);
            mbar_expect_tx(fbb, (uint32_t)(ns * L::SLOT_B));
            b_issued |= 1u << bb;
            b_parity = (b_parity & ~(1u << bb)) | (bphase << bb);
            const uint32_t sb = bbase + (uint32_t)(bb * L::B_BUF);
            for (int k = 0; k < ns; ++k) {
              const int yb = k * args.slice_rows_b;
#pragma unroll
              for (int jb = 0; jb < TNB; ++jb)
                tma_load_2d(sb + k * L::SLOT_B + jb * L::BROWS * L::ATOM, &mapB, c * L::KC,
                            yb + r[TMB + jb] * B + h * N, fbb);
            }
            if (++bb == 2) {
              bb = 0;
              bphase ^= 1u;
            }
            for (int k = 0; k < ns; ++k) {
              if (!mbar_wait(smem_u32(&aempty[slot]), phase ^ 1u, &abort_flag, args.err)) {
                ok = false;
                break;
              }
              const uint32_t fb = smem_u32(&afull[slot]);
              mbar_expect_tx(fb, (uint32_t)L::SLOT_A);
              issued_mask |= 1u << slot;
              last_parity = (last_parity & ~(1u << slot)) | (phase << slot);
              const uint32_t sa = abase + (uint32_t)(slot * L::SLOT_A);
              const int ya = k * args.slice_rows_a;
#pragma unroll
              for (int i = 0; i < TMB; ++i) tma_load_2d(sa + i * B * L::ATOM, &mapA, c * L::KC, ya + r[i] * B, fb);
              if (++slot == RA) {
                slot = 0;
                phase ^= 1u;
              }
            }
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      __syncwarp();  // srec is rewritten next round
#pragma unroll
      for (int w = 0; w < L::RECW; ++w) cur[w] = nxt[w];
      c_it = n_it;
      c_rep = n_rep;
      c_j0 = n_j0;
      c_cnt = n_cnt;
      have = nhave;
    }
    // the copies issued have landed and the MMAs have released every slot
    if (lane == 0) {
      for (int s = 0; s < RA; ++s)
        if (issued_mask & (1u << s)) {
          mbar_wait(smem_u32(&afull[s]), (last_parity >> s) & 1u, &abort_flag, args.err, false);
          mbar_wait(smem_u32(&aempty[s]), (last_parity >> s) & 1u, &abort_flag, args.err, false);
        }
      for (int s = 0; s < 2; ++s)
        if (b_issued & (1u << s)) {
          mbar_wait(smem_u32(&bfull[s]), (b_parity >> s) & 1u, &abort_flag, args.err, false);
          mbar_wait(smem_u32(&bempty[s]), (b_parity >> s) & 1u, &abort_flag, args.err, false);
        }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    if (lane == 0) {
      int slot = 0, bb = 0;  // ring position of the next op(A) slot, op(B) buffer
      uint32_t phase = 0, bphase = 0, acc_phase = 0;
      bool ok = true;
      int nk_next = mt > 0 ? args.tile_nk[blockIdx.x] : 0;  // loaded a tile ahead
      for (int it = 0; it < mt && ok; ++it) {
        const int t = (int)blockIdx.x + it * (int)gridDim.x;
        const int nk = nk_next;
        if (it + 1 < mt) nk_next = args.tile_nk[t + (int)gridDim.x];
        for (int h = 0; h < L::NSUB && ok; ++h) {
          for (int w0 = 0; w0 < nk && ok; w0 += args.kwin) {
            const int w1 = min(nk, w0 + args.kwin);
            // the epilogue has read the previous window's accumulators
            if (!mbar_wait(smem_u32(&acc_empty), acc_phase ^ 1u, &abort_flag, args.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            uint32_t acc0 = 0;  // the window's first products overwrite the accumulators
            for (int j = w0; j < w1 && ok; ++j) {
              for (int c = 0; c < L::KCH && ok; ++c) {
                if (!mbar_wait(smem_u32(&bfull[bb]), bphase, &abort_flag, args.err)) {
                  ok = false;
                  break;
                }
                tc_fence_after();
                // descriptors: the start-address field (bits 0-13, address / 16)
                // of a slot's or a K step's operand is the base descriptor plus
                // its byte offset / 16 (shared addresses stay below 2^18)
                const uint64_t db0 = smem_desc_sw(bbase + (uint32_t)(bb * L::B_BUF), L::SBO, L::SWZ);
                for (int a = 0; a < ns; ++a) {
                  if (!mbar_wait(smem_u32(&afull[slot]), phase, &abort_flag, args.err)) {
                    ok = false;
                    break;
                  }
                  tc_fence_after();
                  const uint64_t da = smem_desc_sw(abase + (uint32_t)(slot * L::SLOT_A), L::SBO, L::SWZ);
                  // slice a of op(A) against slices b, b + 1, ... of op(B), up
                  // to four in one instruction: the slices lie one after the
                  // other in shared memory, and so do the accumulators of the
                  // weight classes a + b, a + b + 1, ...
                  for (int b = 0; b < ns - a; b += 4) {
                    const int nn = min(4, ns - a - b);
                    const uint32_t tacc = tmem + (uint32_t)((a + b) * N);
                    const uint64_t db = db0 + (uint64_t)(b * (L::SLOT_B >> 4));
                    const uint32_t idesc = IDESC0 + (uint32_t)nn * ((uint32_t)(N >> 3) << 17);
#pragma unroll
                    for (int kk = 0; kk < L::KSTEPS; ++kk)
                      mma_kstep<2>(tacc, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc, kk > 0 ? 1u : acc0);
                  }
                  acc0 = 1u;  // slice 0 has started every class
                  mma_commit(smem_u32(&aempty[slot]));  // op(A) slice a is used up
                  if (++slot == RA) {
                    slot = 0;
                    phase ^= 1u;
                  }
                }
                if (!ok) break;
                mma_commit(smem_u32(&bempty[bb]));  // the chunk's op(B) slices are used up
                if (++bb == 2) {
                  bb = 0;
                  bphase ^= 1u;
                }
              }
            }
            if (!ok) break;
            mma_commit(smem_u32(&acc_full));
            acc_phase ^= 1u;
          }
        }
      }
      // every MMA this thread issued completes before tensor memory is released
      mma_commit(smem_u32(&drain_bar));
      mbar_wait(smem_u32(&drain_bar), 0, &abort_flag, args.err, false);
    }
  } else {
    // ------------------------------ epilogue ------------------------------
    constexpr int CW = N / (EPW / 4);        // columns per warp (16)
    const int q = warp & 3;                  // tensor-memory lane quarter
    const int cg = (warp - 2) >> 2;          // columns CW cg .. CW cg + CW - 1 of the tile
    const int rb = (q * 32) / B;             // block row of the tile (a warp's rows lie in one)
    const int rin = (q * 32) % B + lane;     // this thread's row within that block
    const int cb = (cg * CW) / B;            // block column of the tile (at bs <= 64)
    const int et = threadIdx.x - 64;
    uint32_t acc_phase = 0;
    const bool unit = (args.am == 1.0 || args.am == -1.0), neg = args.am < 0.0;
    // the tile's K-step count, its block coordinates, and the C positions of
    // this warp's block and (threads et < TMB TNB) of the block whose norm it
    // writes, loaded a tile ahead
    constexpr int CP = TMB * TNB;
    int nk_n = 0, ti_n = 0, tj_n = 0, p_n = -1, kn_n = -1;
    const auto load_next = [&](int tn) {
      nk_n = args.tile_nk[tn];
      ti_n = args.tiles[2 * tn];
      tj_n = args.tiles[2 * tn + 1];
      p_n = args.cpos[(size_t)tn * CP + rb * TNB + cb];
      if (et < CP) kn_n = args.cpos[(size_t)tn * CP + et];
    };
    if (mt > 0) load_next((int)blockIdx.x);
    const FixedSum fx = args.fx;
    const int slot0 = MAX_U - ns - (fx.below ? 0 : 1);
    for (int it = 0; it < mt; ++it) {
      const int t = (int)blockIdx.x + it * (int)gridDim.x;
      const int nk = nk_n;
      const int I0 = ti_n * TMB, J0 = tj_n * TNB;
      const int I = I0 + rb, J = J0 + cb;
      const int p = p_n;  // position of C_IJ in C (warp-uniform; -1: not in C)
      const int kn = kn_n;
      if (it + 1 < mt) load_next(t + (int)gridDim.x);
      SqAcc4 sq;  // this thread's squares over the tile's column sub-tiles
      bool got = true;
      for (int h = 0; h < L::NSUB; ++h) {
        const int cin = (h * N + cg * CW) % B;  // first column of this warp within block J
        // class_sums leaves its constants' offset in every window's sum
        const long long s0 = -fx.offset * ((nk + args.kwin - 1) / args.kwin);
        long long s[CW];
#pragma unroll
        for (int e = 0; e < CW; ++e) s[e] = s0;
        bool bad = false;
        for (int w0 = 0; w0 < nk; w0 += args.kwin) {
          // (a wait that failed is voted on after the tile: its reads of
          // tensor memory are harmless and the call returns the error)
          got = mbar_wait(smem_u32(&acc_full), acc_phase, &abort_flag, args.err) && got;
          acc_phase ^= 1u;
          __syncwarp();
          tc_fence_after();
          // four columns at a time: every class's value is read behind one
          // wait, in slots: the classes below the sums' unit end at slot 7,
          // the others at slot 6
#pragma unroll
          for (int c4 = 0; c4 < CW / 4; ++c4) {
            uint32_t r[MAX_U][4];
            const uint32_t ta =
                tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cg * CW + c4 * 4) - (uint32_t)(slot0 * N);
#pragma unroll
            for (int u = 0; u < MAX_U; ++u) {
              if (u >= slot0 && u < slot0 + ns) tmem_ld4_issue(ta + (uint32_t)(u * N), r[u]);
              else r[u][0] = r[u][1] = r[u][2] = r[u][3] = 0u;
            }
            tmem_wait_ld(r);
            if (c4 == CW / 4 - 1) {
              // this warp has read its part of the accumulators: the next
              // window's MMAs may overwrite them once every warp has
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&acc_empty));
            }
            class_sums(s + c4 * 4, r, fx);
          }
        }
        // every K of the tile is in these sums: the FP64 result,
        // S_ij 2^(ea + e_i + e_j) * am rounded once, and its squares for the norm
        if (p >= 0) {
          const int er = args.ea + args.sige[(size_t)I * B + rin];
          const int* tj = args.taue + (size_t)J * B + cin;
          double* dst = args.cval + (size_t)p * B * B + (size_t)rin * B + cin;
#pragma unroll
          for (int e = 0; e < CW; e += 4) {
            const int4 tje = __ldg(reinterpret_cast<const int4*>(tj + e));
            const int te[4] = {er + tje.x, er + tje.y, er + tje.z, er + tje.w};
            long long x[4];
            double v[4];
#pragma unroll
            for (int f = 0; f < 4; ++f) x[f] = (unit && neg) ? -s[e + f] : s[e + f];
            fixed_to_f64(x, te, v, bad);
            if (!unit) {
#pragma unroll
              for (int f = 0; f < 4; ++f) v[f] *= args.am;
            }
            sq.add4(v);
            store4(dst + e, v, args.wide);
          }
          if (bad) *args.ovf = 2;
        }
      }
      const double ss = sq.total().warp_total();
      if (lane == 0) partial[it & 1][q][cg] = ss;
      // one barrier per tile (the partials alternate between two buffers):
      // all epilogue warps go on, or all stop
      if (!epi_all<32 * EPW>(got)) break;
      // norms: block (br, bc) of the tile sums the warps of its lane quarters
      // and column groups, in a fixed order
      if (et < CP && kn >= 0) {
        const int br = et / TNB, bc = et % TNB;
        // the lane quarters qq with (32 qq) / B == br and column groups cc
        // with (CW cc) / B == bc, in increasing order
        const int q1 = (br + 1) * B / 32 < 4 ? (br + 1) * B / 32 : 4;
        const int c1 = (bc + 1) * B / CW < EPW / 4 ? (bc + 1) * B / CW : EPW / 4;
        double sum = 0.0;
        for (int qq = br * B / 32; qq < q1; ++qq)
          for (int cc = bc * B / CW; cc < c1; ++cc) sum += partial[it & 1][qq][cc];
        args.cnorm[kn] = sqrt(sum);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(band::TMEM_COLS));
  }
}

// Accumulation units of a split product with ns slices per operand: slice
// pairs (s, t), s + t <= ns + 1, of equal weight 2^(-7 (s + t)) packed
// greedily while sum over the unit of max|q_s| max|q_t| * 64 * kw stays
// <= 2^24, kw = the K blocks a window holds (KW, or the longest tile's K
// steps when fewer), so that every FP32 accumulator sums integers exactly.
struct UnitTable {
  int nunits = 0, npairs = 0;
  int unit_end[MAX_UNITS] = {};  // pairs of unit u: [unit_end[u - 1], unit_end[u])
  int unit_g[MAX_UNITS] = {};    // weight class s + t of unit u
  int si[MAX_PAIRS] = {}, ti[MAX_PAIRS] = {}, pu[MAX_PAIRS] = {};  // slices (1-based) and unit of each pair
};

static UnitTable unit_table(int ns, int kw, int bs) {
  UnitTable t;
  const auto qmax = [](int s) { return s == 1 ? 128 : 64; };
  const int64_t cap = ((int64_t)1 << 24) / ((int64_t)bs * std::max(1, kw));
  for (int g = 2; g <= ns + 1; ++g) {
    int64_t used = 0;
    bool open = false;
    for (int s = 1; s < g; ++s) {
      const int u = g - s;
      if (s > ns || u > ns) continue;
      const int64_t cost = (int64_t)qmax(s) * qmax(u);
      if (open && used + cost > cap) {
        t.unit_end[t.nunits++] = t.npairs;
        used = 0;
        open = false;
      }
      if (!open) {
        if (t.nunits >= MAX_UNITS) fail(IFAC_ERR_UNSUPPORTED, "split product: too many accumulation units");
        t.unit_g[t.nunits] = g;
        open = true;
      }
      if (t.npairs >= MAX_PAIRS) fail(IFAC_ERR_UNSUPPORTED, "split product: too many slice pairs");
      t.si[t.npairs] = s;
      t.ti[t.npairs] = u;
      t.pu[t.npairs] = t.nunits;
      ++t.npairs;
      used += cost;
    }
    if (open) t.unit_end[t.nunits++] = t.npairs;
  }
  return t;
}

// whether a class of kw K blocks and the carry of the class below it (at most
// 2^17) stay within 2^24, as class_sums adds them in FP32
static bool class_carries_fit(int ns, int kw, int bs) {
  for (int g = 2; g <= ns; ++g) {  // class g = s + t, 1-based slices; the last one takes no carry
    const int64_t most = (int64_t)bs * kw * (g == 2 ? 128 * 128 : 2 * 128 * 64 + (int64_t)(g - 3) * 64 * 64);
    if (most + (1 << 17) + 1 > (int64_t)1 << 24) return false;
  }
  return true;
}

template <int B>
static void launch_split_band(ifac_ctx* ctx, const CUtensorMap& mA, const CUtensorMap& mB, const BandArgs& ba,
                              int tiles_bound, int sms) {
  using L = band::SB<B>;
  static std::atomic<unsigned long long> attr{0};
  if (first_on_device(attr, ctx->device))
    IFAC_CK(cudaFuncSetAttribute(k_gemm_split_band<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM_BYTES));
  const int grid = (int)std::min<int64_t>(std::max(tiles_bound, 1), sms);
  k_gemm_split_band<B><<<grid, band::NTB, L::SMEM_BYTES, ctx->stream>>>(mA, mB, ba);
  IFAC_CK_LAUNCH();
}

static void run_split(ifac_ctx* ctx, int ns, const View& arows, bool tA, const ifac_bsr& A, const View& brows,
                      bool tB, const ifac_bsr& B, double alpha, ifac_bsr& C, const int32_t* crow, bool upper,
                      unsigned long long* pairs, OperandCache* ac, OperandCache* bc, const int32_t* avmap,
                      const int32_t* bvmap) {
  Buf<int32_t> asrc, bsrc;  // value positions of op(A) / op(B) view entries under value maps
  using Cf = Cfg<2>;
  const int nb = A.nb, bs = A.bs;
  const int64_t rows = (int64_t)nb * bs;
  if (ns < 3 || ns > 8) fail(IFAC_ERR_UNSUPPORTED, "split product: 3 to 8 slices");
  // a cache filled by an earlier product's op(B) (transposed blocks in the
  // stored order, with that operand's column scales) serves op(A) = that
  // matrix transposed, through the view's source indices, and nothing else
  if (ac && ac->from_b && !(tA && ac->split_ns >= ns)) ac = nullptr;
  const int32_t* amap = (ac && ac->from_b) ? arows.src : nullptr;
  // scales: sigma (rows of op(A)), tau (columns of op(B) = rows of op(B)^T);
  // op(A)'s scales and slices come from the cache when it holds at least ns
  const bool hit = ac && ac->split_ns >= ns;
  const int nsa = hit ? ac->split_ns : (ac ? std::min(8, std::max(ns, ac->want_ns)) : ns);
  Buf<int> sige, taue(ctx, rows);
  // [0] / [1]: scaled 1-norm bounds of op(A) rows / op(B) columns, [2] / [3]: 2-norm bounds
  Buf<unsigned int> l1(ctx, 4);
  IFAC_CK(cudaMemsetAsync(l1.p, 0, 4 * sizeof(unsigned int), ctx->stream));
  // slices: row scale block of an op(A) entry is its CSR row; of an op(B) entry its CSR column
  // (the columns of op(B) are the rows of the other view, made first so that
  // the host has its longest row when op(A)'s slices are under way)
  View bt = view_rows(ctx, B, !tB, nb > 16);
  if (tB) bt.longest = brows.longest_col;
  const size_t bbytes = (size_t)bs * bs * 2;
  Buf<uint8_t> la, lb(ctx, (size_t)ns * (B.nnzb + 1) * bbytes);
  if (!hit) {
    sige = Buf<int>(ctx, rows);
    la = Buf<uint8_t>(ctx, (size_t)nsa * (A.nnzb + 1) * bbytes);
    const int32_t* as = value_src(ctx, arows.src, avmap, A.nnzb, asrc);
    if (!split_rows(ctx, bs, arows.rp, as, nullptr, nb, A.nnzb, arows.longest, tA, A.val, nsa, sige.p, l1.p, l1.p + 2,
                    la.p)) {
      row_scales(ctx, bs, arows.rp, as, nb, A.nnzb, arows.longest, tA, A.val, sige.p, l1.p, l1.p + 2);
      Buf<int32_t> arow(ctx, A.nnzb);
      expand_rows(ctx, arows.rp, nb, arow.p);
      split_blocks(ctx, bs, A.val, as, A.nnzb, tA, arow.p, sige.p, nsa, la.p);
    }
  }
  {
    // (with op(B) = B the view's entries' copies lie in B's stored order)
    if (!tB && nb > 16) bt.longest = read_word(ctx, HW_LONGEST_B);
    Buf<int32_t> btsrc;
    const int32_t* bs_ = value_src(ctx, bt.src, bvmap, B.nnzb, btsrc);
    if (tB || !split_rows(ctx, bs, bt.rp, bs_, bt.src, nb, B.nnzb, bt.longest, true, B.val, ns, taue.p,
                               l1.p + 1, l1.p + 3, lb.p)) {
      row_scales(ctx, bs, bt.rp, bs_, nb, B.nnzb, bt.longest, !tB, B.val, taue.p, l1.p + 1, l1.p + 3);
      split_blocks(ctx, bs, B.val, value_src(ctx, brows.src, bvmap, B.nnzb, bsrc), B.nnzb, !tB, brows.ci, taue.p, ns,
                   lb.p);
    }
  }
  uint8_t* const la_p = hit ? ac->split.p : la.p;
  const int* const sige_p = hit ? ac->sexp.p : sige.p;
  const int* const taue_p = taue.p;
  // one tensor map over all slices of each operand (slice s at row s (nnzb + 1) bs)
  if ((int64_t)ns * (std::max(A.nnzb, B.nnzb) + 1) * bs > (int64_t)0x7fffffff)
    fail(IFAC_ERR_TOO_LARGE, "split product: slice copies exceed the 2^31-row tensor-map range");
  // tile plans: narrow tiles (128 x 64) first.  At bs 64 a product whose
  // tiles all fit one window with at most band::MAX_U units runs on the
  // narrow kernel, every other one on the windowed super-tile kernel; at bs
  // 32 and 128 every product runs on the narrow kernel, window by window.
  // The context's schedule can ask for super-tiles only at bs 64, or narrow
  // tiles (window by window) up to another K length.
  float l1h[4] = {0.f, 0.f, 0.f, 0.f};  // scaled 1- and 2-norm bounds (as l1 above)
  const HostRead l1read{l1h, l1.p, sizeof(l1h)};
  // the default (-1): narrow tiles for every product; with the op(B) slices
  // of a chunk resident and the op(A) slices streamed they are faster than
  // super-tiles on dense products too (3D cluster, n = 16,384: 1.77 s
  // against 2.26 s of split kernel per refinement)
  const int nk_lim = ctx->narrow_kmax_split < 0 ? INT_MAX : ctx->narrow_kmax_split;
  Plan Pb;
  bool banded = bs != 64;
  // block pairs, and block pairs times the ns (ns + 1) / 2 slice pairs
  PairCount pc;
  pc.upper = upper;
  pc.pairs = pairs;
  pc.wpairs = pairs + 1;
  pc.w = ns * (ns + 1) / 2;
  if (bs != 64 || nk_lim > 0) {
    Pb = band_plan(ctx, bs, arows, A, brows, B, C, crow, pc, true, bs == 64 && nk_lim < INT_MAX ? nk_lim : 0, amap,
                   &l1read);
    pc.pairs = pc.wpairs = nullptr;  // counted
    if (bs == 64) banded = Pb.kmax >= 1 && Pb.kmax <= nk_lim;
  } else {
    to_host(ctx, l1h, l1.p, sizeof(l1h));
  }
  Plan P;
  if (!banded) P = make_plan<PAIR * TM, Cf::TN>(ctx, arows, A, brows, B, C, crow, pc, true, 0, amap);
  const int kmax = banded ? Pb.kmax : P.kmax;
  if (hit) {
    l1h[0] = ac->l1;
    l1h[2] = ac->l2;
  } else if (ac) {
    ac->l1 = l1h[0];
    ac->l2 = l1h[2];
    ac->split = std::move(la);
    ac->sexp = std::move(sige);
    ac->split_ns = nsa;
  }
  uint8_t* const lb_p = lb.p;
  if (bc && !tB) {  // op(B) = B in its stored order: keep its slices for a later op(A) = B^T
    bc->reset();
    bc->split = std::move(lb);
    bc->sexp = std::move(taue);
    bc->l1 = l1h[1];
    bc->l2 = l1h[3];
    bc->split_ns = ns;
    bc->from_b = true;
  }
  // window of the narrow kernel: the K blocks (at most 1024 K elements) for
  // which every weight class stays exact in one unit, so that unit u holds
  // the slice pairs (a, b) with a + b = u; the longest tile's K blocks when
  // fewer (one block always fits: 40,960 * 128 <= 2^24 at eight slices)
  int kwin = std::min(1024 / bs, std::max(kmax, 1));
  while (kwin > 1 && (unit_table(ns, kwin, bs).nunits > ns || !class_carries_fit(ns, kwin, bs))) --kwin;
  // the windowed kernel adds into zeroed 64-bit sums that a second kernel
  // converts; the narrow kernel holds each tile's complete sums and writes FP64
  Buf<longlong2> part;
  if (!banded) {
    part = Buf<longlong2>(ctx, (size_t)C.nnzb * (BS * BS / 2));
    IFAC_CK(cudaMemsetAsync(part.p, 0, sizeof(longlong2) * (size_t)C.nnzb * (BS * BS / 2), ctx->stream));
  }
  int ea_alpha = 0;
  const double am = std::frexp(alpha, &ea_alpha) * 2.0;  // alpha = am 2^(ea_alpha - 1), am in [1, 2)
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  // fixed point, scale 2^-f relative to sigma_i tau_j, with every partial sum
  // below 2^62: |sum_ij| <= min(sum_k |a_ik| / sigma_i, sum_k |b_kj| / tau_j)
  // (|a / sigma|, |b / tau| < 1), bounded by the largest scaled row / column
  // 1-norm (FP32, so with a margin), by the scalar inner length K of the
  // longest tile, and (Cauchy-Schwarz) by the product of the largest scaled
  // row and column 2-norms, each widened by 0.0125 sqrt(K) for the slices'
  // rounding (sum_s |q_s| 2^-7s exceeds |a / sigma| by at most 0.0125).  The
  // 2-norm bound is the tight one for dense operands, where every bit of f
  // saved is a rounding the finest accumulation units escape in each window.
  // f <= 56 keeps every weight 2^(f - 7g) of the 7-slice product integral.
  // A sum past 2^62 is an error of the call: the super-tile kernel checks every
  // addition; the narrow kernel's sums wrap modulo 2^64 and are checked when
  // complete, so it would miss one of more than three times the bound.
  int lgK = 0;
  while (((int64_t)1 << lgK) < (int64_t)std::max(kmax, 1) * bs) ++lgK;
  const double rk = 0.0125 * std::sqrt((double)std::max(kmax, 1) * bs);
  const double l2b = ((double)l1h[2] + rk) * ((double)l1h[3] + rk);
  const double l1b = std::min(std::min((double)l1h[0], (double)l1h[1]), l2b) * 1.125 + 2.0;
  int lgB = 0;
  while (std::ldexp(1.0, lgB) < l1b && lgB < 62) ++lgB;
  const int fbits = std::min(56, 62 - std::min(lgK, lgB));
  // units: a window of kw K blocks (every window of every tile has at most kw
  // blocks, so each FP32 accumulator sums integers of magnitude <= 2^24
  // exactly)
  const UnitTable ut = banded ? unit_table(ns, kwin, bs) : unit_table(ns, std::min(KW, std::max(kmax, 1)), bs);
  prof_begin(ctx, 2);
  if (banded) {
    BandArgs ba{};
    ba.tiles = Pb.tiles.p;
    ba.ntiles = Pb.coff.p + Pb.nchunk;
    ba.tile_nk = Pb.tnk.p;
    ba.rec = Pb.rec.p;
    ba.rec_off = Pb.off.p;
    ba.cpos = Pb.cpos.p;
    ba.cval = C.val;
    ba.cnorm = C.norms;
    ba.sige = sige_p;
    ba.taue = taue_p;
    // (a unit below the last class's would hold zeros only)
    const int fband = std::min(fbits, SPLIT_BITS * (ns + 1));
    ba.ea = ea_alpha - 1 - fband;
    ba.am = am;
    ba.nb = nb;
    ba.ns = ns;
    ba.kwin = kwin;
    ba.slice_rows_a = (int)(A.nnzb + 1) * bs;
    ba.slice_rows_b = (int)(B.nnzb + 1) * bs;
    if (ut.nunits != ns) fail(IFAC_ERR_UNSUPPORTED, "split product: a weight class needs two units");
    // the last class's weight is 2^-7(ns + 1): the unit 2^-f is 2^(7 below + d) of it
    const int drop = SPLIT_BITS * (ns + 1) - fband;
    ba.fx.below = drop / SPLIT_BITS;
    ba.fx.d = drop % SPLIT_BITS;
    ba.fx.m0 = std::ldexp(1.0f, -ba.fx.d);
    ba.fx.m1 = std::ldexp(1.0f, 7 - ba.fx.d);
    ba.fx.m2 = std::ldexp(1.0f, 14 - ba.fx.d);
    ba.fx.s1 = 21 - ba.fx.d;
    ba.fx.top = 1 << (10 - ba.fx.d);
    ba.fx.offset = 0x4B400000ll * (1 + (1ll << ba.fx.s1));
    ba.wide = (reinterpret_cast<uintptr_t>(C.val) & 31u) == 0;
    ba.err = ctx->dev_err;
    ba.ovf = ctx->dev_err;
    const int kc = bs < 64 ? bs : 64;  // K elements per chunk (band::SB<bs>::KC)
    const CUtensorMap mA = make_map_box(bs, la_p, (int64_t)ns * (A.nnzb + 1), kc, bs);
    const CUtensorMap mB = make_map_box(bs, lb_p, (int64_t)ns * (B.nnzb + 1), kc, bs < 64 ? bs : 64);
    if (bs == 32) launch_split_band<32>(ctx, mA, mB, ba, Pb.ntiles, sms);
    else if (bs == 64) launch_split_band<64>(ctx, mA, mB, ba, Pb.ntiles, sms);
    else launch_split_band<128>(ctx, mA, mB, ba, Pb.ntiles, sms);
  } else {
    const CUtensorMap mA = make_map<2>(la_p, (int64_t)ns * (A.nnzb + 1));
    const CUtensorMap mB = make_map<2>(lb_p, (int64_t)ns * (B.nnzb + 1));
    static std::atomic<unsigned long long> attr{0};
    if (first_on_device(attr, ctx->device))
      IFAC_CK(cudaFuncSetAttribute(k_gemm_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cf::SMEM_BYTES));
    TileArgs args{};
    args.tiles = P.tiles.p;
    args.ntiles = P.coff.p + P.nchunk;
    args.tile_nk = P.tnk.p;
    args.nwin = cdiv(std::max(kmax, 1), KW);
    args.nb = nb;
    args.rec = P.rec.p;
    args.rec_off = P.off.p;
    args.crp = C.row_ptr;
    args.cci = C.col_idx;
    args.cval = C.val;
    args.cnorm = C.norms;
    args.alpha = 1.0;
    args.err = ctx->dev_err;
    args.split = 1;
    args.cpart = part.p;
    args.stall = 0;
    args.wait_limit = WAIT_LIMIT;
    args.nunits = ut.nunits;
    for (int u = 0; u < ut.nunits; ++u) {
      args.unit_end[u] = ut.unit_end[u];
      args.unit_sh[u] = fbits - SPLIT_BITS * ut.unit_g[u];
    }
    for (int p = 0; p < ut.npairs; ++p) {
      args.pair_ya[p] = (ut.si[p] - 1) * (int)(A.nnzb + 1) * BS;
      args.pair_yb[p] = (ut.ti[p] - 1) * (int)(B.nnzb + 1) * BS;
    }
    args.ovf = ctx->dev_err;
    const int64_t pairs_grid = std::min<int64_t>(std::max(P.ntiles, 1), sms / PAIR);
    k_gemm_tc<2><<<(unsigned)(pairs_grid * PAIR), NTHREADS, Cf::SMEM_BYTES, ctx->stream>>>(mA, mB, args);
    IFAC_CK_LAUNCH();
  }
  prof_end(ctx);
  ++ctx->split_launches;
  if (!banded) {
    k_split_finish<<<(int)std::min<int64_t>(C.nnzb, 152 * 16), 256, 0, ctx->stream>>>(
        crow, C.col_idx, C.nnzb, part.p, C.val, sige_p, taue_p, ea_alpha - 1 - fbits, am, C.norms);
    IFAC_CK_LAUNCH();
  }
}

// Failure-path self-test of the bounded waits: one pair of CTAs over a
// one-tile product (1 x 1 blocks of a 64-row matrix) whose producer and MMA
// issuer do no work, so the epilogue's accumulator wait expires after
// wait_limit polls.  Nothing is copied or multiplied; every CTA releases its
// tensor memory and returns, and the host sees the device error flag.
static void stall_selftest(ifac_ctx* ctx, long long wait_limit) {
  using Cf = Cfg<2>;
  Buf<uint8_t> zeros(ctx, (size_t)2 * BS * BS * 2);
  IFAC_CK(cudaMemsetAsync(zeros.p, 0, zeros.n, ctx->stream));
  const CUtensorMap m = make_map<2>(zeros.p, 2);
  // tiles {0, 0}; one tile; one K step; plan records all zero; C pattern: one block
  Buf<int32_t> small(ctx, 32);
  const int32_t host[32] = {0, 0, /*ntiles*/ 1, /*nk*/ 1, /*rec_off*/ 0, 1, /*crp*/ 0, 1, /*cci*/ 0};
  IFAC_CK(cudaMemcpyAsync(small.p, host, sizeof(host), cudaMemcpyHostToDevice, ctx->stream));
  Buf<double> cval(ctx, (size_t)BS * BS + 1);
  TileArgs args{};
  args.tiles = small.p;
  args.ntiles = small.p + 2;
  args.tile_nk = small.p + 3;
  args.nwin = 1;
  args.nb = 1;
  args.rec = small.p + 9;  // zeros
  args.rec_off = small.p + 4;
  args.crp = small.p + 6;
  args.cci = small.p + 8;
  args.cval = cval.p;
  args.cnorm = cval.p + BS * BS;
  args.alpha = 1.0;
  args.err = ctx->dev_err;
  args.split = 0;
  args.stall = 1;
  args.wait_limit = wait_limit;
  static std::atomic<unsigned long long> attr{0};
  if (first_on_device(attr, ctx->device))
    IFAC_CK(cudaFuncSetAttribute(k_gemm_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cf::SMEM_BYTES));
  k_gemm_tc<2><<<PAIR, NTHREADS, Cf::SMEM_BYTES, ctx->stream>>>(m, m, args);
  IFAC_CK_LAUNCH();
  IFAC_CK(cudaStreamSynchronize(ctx->stream));
}

}  // namespace tc

void tc_wait_timeout_selftest(ifac_ctx* ctx, long long wait_limit) { tc::stall_selftest(ctx, wait_limit); }

void gemm_numeric_tc(ifac_ctx* ctx, int prec, const View& arows, bool tA, const ifac_bsr& A, const View& brows,
                     bool tB, const ifac_bsr& B, double alpha, ifac_bsr& C, const int32_t* crow, bool upper,
                     unsigned long long* pairs_dev, OperandCache* acache, OperandCache* bcache,
                     const OperandCache* bpre, const int32_t* avmap, const int32_t* bvmap, bool out32, bool b32) {
  if (C.nnzb == 0) return;
  if ((out32 || b32) && prec != IFAC_TF32 && prec != IFAC_BF16)
    fail(IFAC_ERR_INVALID, "FP32 values: TF32/BF16 products only");
  if (A.bs != 32 && A.bs != 64 && A.bs != 128) fail(IFAC_ERR_UNSUPPORTED, "tensor-core block products: bs 32, 64 or 128");
  if (!B.val && !(bpre && bpre->b_ready)) fail(IFAC_ERR_INVALID, "tensor-core product: op(B) has no values");
  if (prec == IFAC_BF16)
    tc::run<2>(ctx, arows, tA, A, brows, tB, B, alpha, C, crow, upper, pairs_dev, acache, bcache, bpre, avmap, bvmap,
               out32, b32);
  else if (prec == IFAC_TF32)
    tc::run<4>(ctx, arows, tA, A, brows, tB, B, alpha, C, crow, upper, pairs_dev, acache, bcache, bpre, avmap, bvmap,
               out32, b32);
  else if (prec == IFAC_FP64_SPLIT)
    tc::run_split(ctx, ctx->split_slices, arows, tA, A, brows, tB, B, alpha, C, crow, upper, pairs_dev, acache,
                  bcache, avmap, bvmap);
  else fail(IFAC_ERR_UNSUPPORTED, "unknown precision");
}

// the mixed schedule's P at m = 2 as a low-precision op(B) copy (k_poly2_lp)
void poly2_lp(ifac_ctx* ctx, int elt, const ifac_bsr& U, const ifac_bsr& D, double b1, double b2,
              const ifac_bsr& P, const int32_t* prow, void* out, const int32_t* umap, bool u32) {
  if (U.bs != 64) fail(IFAC_ERR_UNSUPPORTED, "correction operand: bs 64");
  const size_t bb = (size_t)64 * 64 * elt;
  IFAC_CK(cudaMemsetAsync(static_cast<uint8_t*>(out) + (size_t)P.nnzb * bb, 0, bb, ctx->stream));
  if (P.nnzb == 0) return;
  const int grid = (int)std::min<int64_t>(P.nnzb, 152 * 8);
  const float* u32v = reinterpret_cast<const float*>(U.val);
  if (elt == 2 && u32)
    tc::k_poly2_lp<2, float><<<grid, 256, 0, ctx->stream>>>(prow, P.col_idx, P.nnzb, U.row_ptr, U.col_idx, u32v, umap,
                                                             D.row_ptr, D.col_idx, D.val, (float)b1, (float)b2, out);
  else if (elt == 2)
    tc::k_poly2_lp<2, double><<<grid, 256, 0, ctx->stream>>>(prow, P.col_idx, P.nnzb, U.row_ptr, U.col_idx, U.val,
                                                              umap, D.row_ptr, D.col_idx, D.val, (float)b1, (float)b2,
                                                              out);
  else if (u32)
    tc::k_poly2_lp<4, float><<<grid, 256, 0, ctx->stream>>>(prow, P.col_idx, P.nnzb, U.row_ptr, U.col_idx, u32v, umap,
                                                             D.row_ptr, D.col_idx, D.val, (float)b1, (float)b2, out);
  else
    tc::k_poly2_lp<4, double><<<grid, 256, 0, ctx->stream>>>(prow, P.col_idx, P.nnzb, U.row_ptr, U.col_idx, U.val,
                                                              umap, D.row_ptr, D.col_idx, D.val, (float)b1, (float)b2,
                                                              out);
  IFAC_CK_LAUNCH();
}

}  // namespace ifac
