// pattern.cu -- block-pattern (symbolic) work on the device.
//
// Patterns are handled as bitmaps: one bit per (block row, block column),
// W = ceil(nb/32) 32-bit words per block row.  The pattern of a product
// op(A) op(B) is, row by row, the OR of the op(B)-row bitmaps selected by the
// stored blocks of the op(A) row (every (I, J) with some K such that both
// blocks are stored); the pattern of a sum is the OR of the operands' bitmaps.
// Enumerating set bits in word order yields sorted column lists directly, so
// no sort is needed.  Row pointers come from an exclusive scan of popcounts.
//
// What bounds it is launches: at a few thousand rows each of these kernels
// runs for 2 us.  So a small pattern (rule_small) is one CTA from the bitmaps
// in shared memory to the column lists, and a larger one is a bitmap kernel, a
// count kernel whose last CTA scans (scan_tail) and a fill kernel; totals
// reach the host through mapped memory.  Before, each was up to nine launches
// (clear, scatter, OR, count, scan, copy to the host, fill).  FP64 product of
// the 1000-row chain 171 -> 119 us; refinement of the 4096-row chain 5.0 -> 3.5
// ms (500 launches -> 162).
#include "internal.cuh"
#include "scan_tail.cuh"

namespace ifac {

int words_per_row(int nb) { return (nb + 31) / 32; }

namespace {

constexpr int NT = 256;         // threads of the row kernels (one warp per block row)
constexpr int SMALL_NB = 512;   // block rows of a one-CTA pattern: two bitmaps of 32 KB
constexpr int SMALL_IN = 16384;  // and blocks of an operand: 64 KB of staged lists

// one operand's pattern as a bitmap source, transposed or not
struct Source {
  const int32_t* rp;
  const int32_t* ci;
  int trans;
};

struct Job {
  Source s[3];
  int nsrc;
  int diag;             // the diagonal blocks as well
  int nb, W;
  int cap;              // one-CTA kernel: what the lists hold; a longer pattern is only counted
  const int32_t* arp;   // a product: rows of op(A) (the sources are op(B)); null: the union of the sources
  const int32_t* aci;
  int upper;            // only columns >= the row
  int32_t* rp;
  int32_t* ci;
  int32_t* row;
  // a transposed view: the position of each entry's block in the source matrix
  const int32_t* frp;
  const int32_t* fci;
  int32_t* src;
  int32_t* total;       // host word, or null
  // host words (or null) for the blocks of the longest row of lrp, or of the
  // pattern itself (lrp null)
  const int32_t* lrp[2];
  int32_t* longest[2];
};

__device__ __forceinline__ uint32_t upper_bits(uint32_t v, int row, int w) {
  if (w < (row >> 5)) return 0u;
  return w == (row >> 5) ? v & ~((1u << (row & 31)) - 1u) : v;
}

// entry (r, c) of A^T: the position of block (c, r) in A's sorted row c
__device__ __forceinline__ int find_src(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int r, int c) {
  int lo = rp[c], hi = rp[c + 1];
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (ci[mid] < r) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// the set bits of word w of row r at positions pos, pos + 1, ...
__device__ __forceinline__ void emit(const Job& j, uint32_t word, int r, int w, int pos) {
  while (word) {
    const int c = w * 32 + __ffs((int)word) - 1;
    j.ci[pos] = c;
    if (j.row) j.row[pos] = r;
    ++pos;
    word &= word - 1;
  }
}

// A whole small pattern in one CTA.  Every phase takes all rows at once (a
// group of 1024 / nb threads each), and a product's op(A) lists are staged in
// shared memory first: a loop over rows would pay the latency of global memory
// for each (nb = 512: 20 us that way).
__global__ void __launch_bounds__(1024) k_pattern_small(Job j, int nnza) {
  extern __shared__ uint32_t sh[];
  __shared__ int32_t wsum[32], wlen[2][32];
  const int WP = j.W | 1, nw = j.nb * WP;           // odd row stride: no bank conflicts across rows
  uint32_t* bm = sh;                                // [nb * WP] the sources
  int32_t* off = reinterpret_cast<int32_t*>(bm + nw);  // [nb + 1]
  uint32_t* out = j.arp ? reinterpret_cast<uint32_t*>(off + j.nb + 1) : bm;  // [nb * WP] the pattern
  int32_t* arp = reinterpret_cast<int32_t*>(out + nw);  // product: [nb + 1], [nnza]
  int32_t* aci = arp + j.nb + 1;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int lg = 5;  // log2 of the threads that share a row
  while ((j.nb << lg) > 1024 && lg > 0) --lg;
  const int G = 1 << lg, grow = tid >> lg, glane = tid & (G - 1);
  const bool live = grow < j.nb;
  for (int i = tid; i < nw; i += 1024) bm[i] = 0u;
  if (j.arp) {
    for (int i = tid; i <= j.nb; i += 1024) arp[i] = j.arp[i];
    for (int i = tid; i < nnza; i += 1024) aci[i] = j.aci[i];
  }
  __syncthreads();
  if (live) {
    for (int k = 0; k < j.nsrc; ++k) {
      const int p1 = j.s[k].rp[grow + 1];
#pragma unroll 4
      for (int p = j.s[k].rp[grow] + glane; p < p1; p += G) {
        const int c = j.s[k].ci[p], br = j.s[k].trans ? c : grow, bc = j.s[k].trans ? grow : c;
        atomicOr(&bm[br * WP + (bc >> 5)], 1u << (bc & 31));
      }
    }
    if (j.diag && glane == 0) atomicOr(&bm[grow * WP + (grow >> 5)], 1u << (grow & 31));
  }
  __syncthreads();
  if (j.arp) {
    if (live)
      for (int w = glane; w < j.W; w += G) {
        uint32_t acc = 0;
        for (int p = arp[grow]; p < arp[grow + 1]; ++p) acc |= bm[aci[p] * WP + w];
        out[grow * WP + w] = j.upper ? upper_bits(acc, grow, w) : acc;
      }
    __syncthreads();
  }
  int c = 0;
  if (tid < j.nb)
    for (int w = 0; w < j.W; ++w) c += __popc(out[tid * WP + w]);
  int x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[wid] = x;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (j.longest[i]) {
      const int len = tid >= j.nb ? 0 : j.lrp[i] ? j.lrp[i][tid + 1] - j.lrp[i][tid] : c;
      const int m = (int)__reduce_max_sync(0xffffffffu, (unsigned)len);
      if (lane == 0) wlen[i][wid] = m;
    }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (j.longest[i] && wid == i) {
      const int m = (int)__reduce_max_sync(0xffffffffu, (unsigned)wlen[i][lane]);
      if (lane == 0) *j.longest[i] = m;
    }
  const int run = (int)__reduce_add_sync(0xffffffffu, (unsigned)(lane < wid ? wsum[lane] : 0)) + x - c;
  if (tid < j.nb) {
    off[tid] = run;
    j.rp[tid] = run;
    if (tid == j.nb - 1) {
      off[j.nb] = j.rp[j.nb] = run + c;
      if (j.total) *j.total = run + c;
    }
  }
  __syncthreads();
  if (!live || off[j.nb] > j.cap) return;
  const auto before = [&](int r, int w) {  // set bits of row r in the words before w
    int n = off[r];
    for (int v = 0; v < w; ++v) n += __popc(out[r * WP + v]);
    return n;
  };
  for (int w = glane; w < j.W; w += G) {
    const uint32_t word = out[grow * WP + w];
    if (word) emit(j, word, grow, w, before(grow, w));
  }
  if (j.src) {  // (a transposed view: each stored block finds its own place)
    const int p1 = j.frp[grow + 1];
    for (int p = j.frp[grow] + glane; p < p1; p += G) {
      const int r = j.fci[p], w = grow >> 5;
      j.src[before(r, w) + __popc(out[r * WP + w] & ((1u << (grow & 31)) - 1u))] = p;
    }
  }
}

// the sources' bits in a cleared bitmap (one warp per block row)
__global__ void __launch_bounds__(NT) k_scatter(Job j, uint32_t* __restrict__ bm) {
  const int row = (int)((blockIdx.x * (size_t)NT + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (row >= j.nb) return;
  for (int k = 0; k < j.nsrc; ++k)
    for (int p = j.s[k].rp[row] + lane; p < j.s[k].rp[row + 1]; p += 32) {
      const int c = j.s[k].ci[p], r = j.s[k].trans ? c : row, col = j.s[k].trans ? row : c;
      atomicOr(&bm[(size_t)r * j.W + (col >> 5)], 1u << (col & 31));
    }
  if (j.diag && lane == 0) atomicOr(&bm[(size_t)row * j.W + (row >> 5)], 1u << (row & 31));
}

// the product's rows, out[I] = OR over K in row I of op(A) of bm[K] (or bm
// itself), their counts and the row pointers; ticket[1] and [2] are zero between launches
__global__ void __launch_bounds__(NT) k_rows_scan(Job j, const uint32_t* __restrict__ bm, uint32_t* __restrict__ out,
                                                  int32_t* __restrict__ cnt, unsigned* __restrict__ ticket) {
  __shared__ int32_t wlen[2][NT / 32];
  const int row = (int)((blockIdx.x * (size_t)NT + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  int c = 0;
  if (row < j.nb) {
    const int p0 = j.arp ? j.arp[row] : 0, p1 = j.arp ? j.arp[row + 1] : 0;
    for (int w = lane; w < j.W; w += 32) {
      uint32_t acc = 0;
      if (j.arp) {
        for (int p = p0; p < p1; ++p) acc |= bm[(size_t)j.aci[p] * j.W + w];
        if (j.upper) acc = upper_bits(acc, row, w);
        out[(size_t)row * j.W + w] = acc;
      } else {
        acc = bm[(size_t)row * j.W + w];
      }
      c += __popc(acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) cnt[row] = c;
  }
  int* const lmax = reinterpret_cast<int*>(ticket + 1);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (j.longest[i] && lane == 0)
      wlen[i][threadIdx.x >> 5] = row >= j.nb ? 0 : j.lrp[i] ? j.lrp[i][row + 1] - j.lrp[i][row] : c;
  if (j.longest[0] || j.longest[1]) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (j.longest[i] && threadIdx.x == i) {  // one atomic for each CTA
        int len = 0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) len = max(len, wlen[i][w]);
        atomicMax(lmax + i, len);
      }
  }
  const bool last = scan_tail<NT>(cnt, j.rp, j.nb, ticket, j.total);
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (last && j.longest[i] && threadIdx.x == i) *j.longest[i] = atomicExch(lmax + i, 0);
}

// enumerate the set bits of each row in increasing column (warp per row)
__global__ void __launch_bounds__(NT) k_row_fill(Job j, const uint32_t* __restrict__ bm) {
  const int row = (int)((blockIdx.x * (size_t)NT + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (row >= j.nb) return;
  int pos = j.rp[row];
  for (int base = 0; base < j.W; base += 32) {
    const int w = base + lane;
    const uint32_t word = w < j.W ? bm[(size_t)row * j.W + w] : 0u;
    const int c = __popc(word);
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    emit(j, word, row, w, pos + x - c);
    if (j.src)
      for (uint32_t u = word, q = (uint32_t)(pos + x - c); u; u &= u - 1u, ++q)
        j.src[q] = find_src(j.frp, j.fci, row, w * 32 + __ffs((int)u) - 1);
    pos += __shfl_sync(0xffffffffu, x, 31);
  }
}

int row_grid(int nb) { return cdiv((int64_t)nb * 32, NT); }

// One CTA does a pattern of up to SMALL_NB block rows whose operands hold up
// to 16,384 blocks and whose result at most 32,768 (about 10 us there: what
// three kernels with all their warps take); beyond that the rows go over the
// whole GPU.
bool rule_small(int nb, int64_t in_blocks, int64_t out_bound) {
  return nb <= SMALL_NB && in_blocks <= SMALL_IN && out_bound <= 32768;
}

void launch_small(ifac_ctx* ctx, const Job& j, int64_t nnza) {
  const size_t nw = (size_t)j.nb * (j.W | 1), smem = 4 * (nw + j.nb + 1 + (j.arp ? nw + j.nb + 1 + (size_t)nnza : 0));
  // (a kernel has 48 KB without asking, its static shared memory included; set
  // at every launch above 32 KB, so that no other thread can launch before it)
  if (smem > 32 * 1024)
    IFAC_CK(cudaFuncSetAttribute(k_pattern_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 4 * (2 * (SMALL_NB * (SMALL_NB / 32 + 1) + SMALL_NB + 1) + SMALL_IN)));
  k_pattern_small<<<1, 1024, smem, ctx->stream>>>(j, (int)nnza);
  IFAC_CK_LAUNCH();
}

// A list that a result keeps, in a caller's memory: one of the exact size in
// place of one taken by a bound, where that saves more than 64 KB.
template <typename T>
void shrink(ifac_ctx* ctx, Buf<T>& b, int64_t n) {
  if (!ctx->custom_alloc || (b.n - (size_t)n) * sizeof(T) <= 65536) return;
  Buf<T> c(ctx, n);
  if (n > 0) IFAC_CK(cudaMemcpyAsync(c.p, b.p, sizeof(T) * n, cudaMemcpyDeviceToDevice, ctx->stream));
  b = std::move(c);
}

// The pattern of a job: known >= 0 the number of its blocks where the host
// knows it (a transposed view), so nothing is read back; guess what it will be
// about.  The one-CTA kernel writes lists of `room` blocks and goes out once more
// where they are too short.  j's longest[] are set by the caller.
Pattern run_job(ifac_ctx* ctx, Job j, int64_t in_blocks, int64_t guess, int64_t room, int64_t known,
                Buf<int32_t>* src, int64_t nnza = 0) {
  Pattern P;
  j.W = words_per_row(j.nb);
  P.rp = Buf<int32_t>(ctx, j.nb + 1);
  j.rp = P.rp.p;
  j.total = known < 0 ? host_word(ctx, HW_NNZ) : nullptr;
  const auto alloc = [&](int64_t n) {
    P.ci = Buf<int32_t>(ctx, n);
    P.row = Buf<int32_t>(ctx, n);
    j.ci = P.ci.p;
    j.row = P.row.p;
    if (src) {
      *src = Buf<int32_t>(ctx, n);
      j.src = src->p;
    }
  };
  if (rule_small(j.nb, in_blocks, guess)) {
    j.cap = (int)room;
    alloc(room);
    launch_small(ctx, j, nnza);
    P.nnzb = known >= 0 ? known : read_word(ctx, HW_NNZ);
    if (P.nnzb > j.cap) {
      j.cap = (int)P.nnzb;
      j.total = nullptr;
      j.longest[0] = j.longest[1] = nullptr;
      alloc(P.nnzb);
      launch_small(ctx, j, nnza);
    }
    shrink(ctx, P.ci, P.nnzb);
    return P;
  }
  const size_t words = (size_t)j.nb * j.W;
  Buf<uint32_t> bm(ctx, words), rows(ctx, j.arp ? words : 1);
  Buf<int32_t> cnt(ctx, j.nb);
  IFAC_CK(cudaMemsetAsync(bm.p, 0, sizeof(uint32_t) * words, ctx->stream));
  k_scatter<<<row_grid(j.nb), NT, 0, ctx->stream>>>(j, bm.p);
  IFAC_CK_LAUNCH();
  k_rows_scan<<<row_grid(j.nb), NT, 0, ctx->stream>>>(j, bm.p, rows.p, cnt.p, ctx->ticket);
  IFAC_CK_LAUNCH();
  P.nnzb = known >= 0 ? known : read_word(ctx, HW_NNZ);
  alloc(P.nnzb);
  if (P.nnzb > 0) {
    k_row_fill<<<row_grid(j.nb), NT, 0, ctx->stream>>>(j, j.arp ? rows.p : bm.p);
    IFAC_CK_LAUNCH();
  }
  return P;
}

void add_source(Job& j, const int32_t* rp, const int32_t* ci, int64_t nnzb, bool trans) {
  if (nnzb > 0) j.s[j.nsrc++] = Source{rp, ci, trans ? 1 : 0};
}

}  // namespace

Pattern pattern_from_bitmap(ifac_ctx* ctx, const uint32_t* bm, int nb) {
  Job j{};
  j.nb = nb;
  j.W = words_per_row(nb);
  Pattern P;
  P.rp = Buf<int32_t>(ctx, nb + 1);
  j.rp = P.rp.p;
  j.total = host_word(ctx, HW_NNZ);
  Buf<int32_t> cnt(ctx, nb);
  k_rows_scan<<<row_grid(nb), NT, 0, ctx->stream>>>(j, bm, nullptr, cnt.p, ctx->ticket);
  IFAC_CK_LAUNCH();
  P.nnzb = read_word(ctx, HW_NNZ);
  P.ci = Buf<int32_t>(ctx, P.nnzb);
  P.row = Buf<int32_t>(ctx, P.nnzb);
  j.ci = P.ci.p;
  j.row = P.row.p;
  if (P.nnzb > 0) {
    k_row_fill<<<row_grid(nb), NT, 0, ctx->stream>>>(j, bm);
    IFAC_CK_LAUNCH();
  }
  return P;
}

// ---------------------------------------------------------------------------
// transposed views
// ---------------------------------------------------------------------------
// out[q] for block q = (row[q], ci[q]) of A: the position of its transpose
__global__ void k_find_src(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int64_t nnz,
                           const int32_t* __restrict__ row, int32_t* __restrict__ out) {
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q < nnz) out[q] = find_src(rp, ci, row[q], ci[q]);
}

void transposed_positions(ifac_ctx* ctx, const ifac_bsr& A, const int32_t* row, int32_t* out) {
  if (A.nnzb == 0) return;
  k_find_src<<<cdiv(A.nnzb, 256), 256, 0, ctx->stream>>>(A.row_ptr, A.col_idx, A.nnzb, row, out);
  IFAC_CK_LAUNCH();
}

View view_rows(ifac_ctx* ctx, const ifac_bsr& A, bool trans, bool want_longest) {
  View v;
  if (!trans) {
    v.rp = A.row_ptr;
    v.ci = A.col_idx;
    v.src = nullptr;
    return v;
  }
  Job j{};
  j.nb = A.nb;
  add_source(j, A.row_ptr, A.col_idx, A.nnzb, true);
  j.frp = A.row_ptr;
  j.fci = A.col_idx;
  if (want_longest) j.longest[0] = host_word(ctx, HW_LONGEST_B);
  Pattern P = run_job(ctx, j, A.nnzb, A.nnzb, A.nnzb, A.nnzb, &v.own_src);  // A^T has A's blocks
  v.own_rp = std::move(P.rp);
  v.own_ci = std::move(P.ci);
  v.rp = v.own_rp.p;
  v.ci = v.own_ci.p;
  v.src = v.own_src.p;
  return v;
}

// ---------------------------------------------------------------------------
// product and union patterns
// ---------------------------------------------------------------------------
Pattern product_pattern(ifac_ctx* ctx, const View& arows, int64_t nnza, const ifac_bsr& B, bool transB, int nb,
                        bool upper, bool want_longest) {
  Job j{};
  j.nb = nb;
  add_source(j, B.row_ptr, B.col_idx, B.nnzb, transB);
  j.arp = arows.rp;
  j.aci = arows.ci;
  j.upper = upper ? 1 : 0;
  // a row of op(A) with k blocks meets about k nnz(B) / nb of op(B)
  const int64_t full = (int64_t)nb * nb, guess = std::min(full, nnza * std::max<int64_t>(1, B.nnzb / nb));
  // (twice that and at least 64 KB, so that uneven operands seldom need more)
  const int64_t room = std::min(full, std::max<int64_t>(16384, 2 * nnza * ((B.nnzb + nb - 1) / nb)));
  const bool want_a = want_longest, want_b = want_longest && transB;
  if (want_a) {
    j.lrp[0] = arows.rp;
    j.longest[0] = host_word(ctx, HW_LONGEST_A);
  }
  if (want_b) {
    j.lrp[1] = B.row_ptr;
    j.longest[1] = host_word(ctx, HW_LONGEST_B);
  }
  Pattern P = run_job(ctx, j, std::max(nnza, B.nnzb), guess, room, -1, nullptr, nnza);
  if (want_a) P.longest_a = read_word(ctx, HW_LONGEST_A);  // (written with the total)
  if (want_b) P.longest_b = read_word(ctx, HW_LONGEST_B);
  return P;
}

Pattern union_pattern(ifac_ctx* ctx, const ifac_bsr& A, const ifac_bsr* B, bool diag) {
  Job j{};
  j.nb = A.nb;
  add_source(j, A.row_ptr, A.col_idx, A.nnzb, false);
  if (B) add_source(j, B->row_ptr, B->col_idx, B->nnzb, false);
  j.diag = diag ? 1 : 0;
  const int64_t in = A.nnzb + (B ? B->nnzb : 0);
  const int64_t cap = std::min<int64_t>(in + (diag ? A.nb : 0), (int64_t)A.nb * A.nb);
  return run_job(ctx, j, in, cap, cap, -1, nullptr);
}

Pattern sym_pattern(ifac_ctx* ctx, const ifac_bsr& U, const ifac_bsr* B, bool diag) {
  Job j{};
  j.nb = U.nb;
  add_source(j, U.row_ptr, U.col_idx, U.nnzb, false);
  add_source(j, U.row_ptr, U.col_idx, U.nnzb, true);
  if (B) add_source(j, B->row_ptr, B->col_idx, B->nnzb, false);
  j.diag = diag ? 1 : 0;
  const int64_t in = 2 * U.nnzb + (B ? B->nnzb : 0);
  const int64_t cap = std::min<int64_t>(in + (diag ? U.nb : 0), (int64_t)U.nb * U.nb);
  return run_job(ctx, j, in, cap, cap, -1, nullptr);
}

__global__ void k_expand_rows(const int32_t* __restrict__ rp, int nb, int32_t* __restrict__ row) {
  int r = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (r >= nb) return;
  for (int p = rp[r] + lane; p < rp[r + 1]; p += 32) row[p] = r;
}

void expand_rows(ifac_ctx* ctx, const int32_t* rp, int nb, int32_t* row) {
  k_expand_rows<<<cdiv((int64_t)nb * 32, 256), 256, 0, ctx->stream>>>(rp, nb, row);
  IFAC_CK_LAUNCH();
}

// ---------------------------------------------------------------------------
// block selection / truncation with order-preserving compaction
// ---------------------------------------------------------------------------
// whether block p stays: by mask, or (keep null) by !(norm < tau) -- NaN norms
// are kept, as in the oracle
__device__ __forceinline__ bool stays(const uint8_t* __restrict__ keep, const double* __restrict__ norms, double tau,
                                      int p) {
  return keep ? keep[p] != 0 : !(norms[p] < tau);
}

// kept blocks per block row, and their row pointers
__global__ void __launch_bounds__(NT)
    k_keep_scan(const int32_t* __restrict__ rp, int nb, const uint8_t* __restrict__ keep,
                const double* __restrict__ norms, double tau, int32_t* __restrict__ cnt, int32_t* __restrict__ rp_new,
                unsigned* __restrict__ ticket, int32_t* __restrict__ total) {
  const int row = (int)((blockIdx.x * (size_t)NT + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (row < nb) {
    int c = 0;
    for (int p = rp[row] + lane; p < rp[row + 1]; p += 32) c += stays(keep, norms, tau, p) ? 1 : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0) cnt[row] = c;
  }
  scan_tail<NT>(cnt, rp_new, nb, ticket, total);
}

// dest[p]: the new position of block p (-1: dropped), if dest; vmap[new
// position] = p, if vmap
__global__ void __launch_bounds__(NT)
    k_keep_dest(const int32_t* __restrict__ rp, int nb, const uint8_t* __restrict__ keep,
                const double* __restrict__ norms, double tau, const int32_t* __restrict__ rp_new,
                const int32_t* __restrict__ ci, int32_t* __restrict__ ci_new, double* __restrict__ norms_new,
                int32_t* __restrict__ dest, int32_t* __restrict__ vmap) {
  const int row = (int)((blockIdx.x * (size_t)NT + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (row >= nb) return;
  int pos = rp_new[row];
  for (int base = rp[row]; base < rp[row + 1]; base += 32) {
    const int p = base + lane;
    const bool in = p < rp[row + 1], k = in && stays(keep, norms, tau, p);
    const unsigned m = __ballot_sync(0xffffffffu, k);
    const int d = k ? pos + __popc(m & ((1u << lane) - 1u)) : -1;
    if (in && dest) dest[p] = d;
    if (k) {
      ci_new[d] = ci[p];
      norms_new[d] = norms[p];
      if (vmap) vmap[d] = p;
    }
    pos += __popc(m);
  }
}

// The same for up to SMALL_KEEP blocks, in one CTA (1024 blocks take 1.5 us; at
// 12,000 the two kernels above, 10 us, are faster): kept blocks stay in CSR
// order, so a block's new position is the number of kept ones before it.
constexpr int SMALL_KEEP = 4096;

__global__ void __launch_bounds__(1024)
    k_keep_small(const int32_t* __restrict__ rp, int nb, int nnz, const uint8_t* __restrict__ keep,
                 const double* __restrict__ norms, double tau, const int32_t* __restrict__ ci,
                 int32_t* __restrict__ rp_new, int32_t* __restrict__ ci_new, double* __restrict__ norms_new,
                 int32_t* __restrict__ dest, int32_t* __restrict__ vmap, int32_t* __restrict__ total) {
  extern __shared__ int32_t before[];  // [nnz + 1] kept blocks before block p
  __shared__ int wsum[2][32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int carry = 0;
  for (int base = 0, par = 0; base < nnz; base += 1024, par ^= 1) {
    const int p = base + tid;
    const bool k = p < nnz && stays(keep, norms, tau, p);
    const unsigned m = __ballot_sync(0xffffffffu, k);
    if (lane == 0) wsum[par][wid] = __popc(m);
    __syncthreads();
    const int c = wsum[par][lane];  // every warp adds up the warps' counts
    int x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    const int d = carry + __shfl_sync(0xffffffffu, x - c, wid) + __popc(m & ((1u << lane) - 1u));
    if (p < nnz) {
      before[p] = d;
      if (dest) dest[p] = k ? d : -1;
    }
    if (k) {
      ci_new[d] = ci[p];
      norms_new[d] = norms[p];
      if (vmap) vmap[d] = p;
    }
    carry += __shfl_sync(0xffffffffu, x, 31);
  }
  if (tid == 0) {
    before[nnz] = carry;
    *total = carry;
  }
  __syncthreads();
  for (int r = tid; r <= nb; r += 1024) rp_new[r] = before[rp[r]];
}

__global__ void k_copy_blocks(const double* __restrict__ src, const int32_t* __restrict__ dest, int64_t nblk,
                              int bsz, bool wide, double* __restrict__ dst) {
  for (int64_t p = blockIdx.x; p < nblk; p += gridDim.x) {
    int d = dest[p];
    if (d < 0) continue;
    if (wide && (bsz & 1) == 0) {  // aligned values and even block size: every block starts 16-byte aligned
      const double2* s = reinterpret_cast<const double2*>(src + (size_t)p * bsz);
      double2* t = reinterpret_cast<double2*>(dst + (size_t)d * bsz);
      for (int e = threadIdx.x; e < bsz / 2; e += blockDim.x) t[e] = s[e];
    } else {
      for (int e = threadIdx.x; e < bsz; e += blockDim.x) dst[(size_t)d * bsz + e] = src[(size_t)p * bsz + e];
    }
  }
}

// The kept blocks' pattern and norms, in A's order, with their values left
// out; dest / vmap as in k_keep_dest.  The lists are sized for every block, so
// that both kernels go out before the count is read.
struct Kept {
  Buf<int32_t> rp, ci, map;
  Buf<double> norms;
  int64_t n = 0;
};

static Kept keep_pattern(ifac_ctx* ctx, const ifac_bsr& A, const uint8_t* keep, double tau, bool want_vmap) {
  Kept k;
  const int nb = A.nb;
  k.rp = Buf<int32_t>(ctx, nb + 1);
  if (A.nnzb == 0) {
    IFAC_CK(cudaMemsetAsync(k.rp.p, 0, sizeof(int32_t) * (nb + 1), ctx->stream));
    k.ci = Buf<int32_t>(ctx, 1);
    k.norms = Buf<double>(ctx, 1);
    return k;
  }
  k.ci = Buf<int32_t>(ctx, A.nnzb);
  k.norms = Buf<double>(ctx, A.nnzb);
  k.map = Buf<int32_t>(ctx, A.nnzb);
  const auto finish = [&] {
    k.n = read_word(ctx, HW_KEPT);
    shrink(ctx, k.ci, k.n);
    shrink(ctx, k.norms, k.n);
  };
  if (A.nnzb <= SMALL_KEEP) {
    k_keep_small<<<1, 1024, 4 * ((size_t)A.nnzb + 1), ctx->stream>>>(A.row_ptr, nb, (int)A.nnzb, keep, A.norms, tau, A.col_idx, k.rp.p,
                                                 k.ci.p, k.norms.p, want_vmap ? nullptr : k.map.p,
                                                 want_vmap ? k.map.p : nullptr, host_word(ctx, HW_KEPT));
    IFAC_CK_LAUNCH();
    finish();
    return k;
  }
  Buf<int32_t> cnt(ctx, nb);
  k_keep_scan<<<row_grid(nb), NT, 0, ctx->stream>>>(A.row_ptr, nb, keep, A.norms, tau, cnt.p, k.rp.p, ctx->ticket,
                                                    host_word(ctx, HW_KEPT));
  IFAC_CK_LAUNCH();
  k_keep_dest<<<row_grid(nb), NT, 0, ctx->stream>>>(A.row_ptr, nb, keep, A.norms, tau, k.rp.p, A.col_idx, k.ci.p,
                                                    k.norms.p, want_vmap ? nullptr : k.map.p,
                                                    want_vmap ? k.map.p : nullptr);
  IFAC_CK_LAUNCH();
  finish();
  return k;
}

// a new matrix of the kept blocks, in order
static Mat gather_kept(ifac_ctx* ctx, const ifac_bsr& A, Kept&& k) {
  Mat R(ctx);
  R.m.n = A.n;
  R.m.bs = A.bs;
  R.m.nb = A.nb;
  R.m.nnzb = k.n;
  R.m.row_ptr = k.rp.release();
  R.m.col_idx = k.ci.release();
  R.m.norms = k.norms.release();
  R.m.val = static_cast<double*>(dalloc(ctx, sizeof(double) * (size_t)(k.n ? k.n : 1) * A.bs * A.bs));
  if (k.n > 0) {
    const int blocks = (int)std::min<int64_t>(A.nnzb, 152 * 16);
    k_copy_blocks<<<blocks, 256, 0, ctx->stream>>>(A.val, k.map.p, A.nnzb, A.bs * A.bs, aligned16(A.val), R.m.val);
    IFAC_CK_LAUNCH();
  }
  return R;
}

Mat select_blocks(ifac_ctx* ctx, const ifac_bsr& A, const uint8_t* keep) {
  return gather_kept(ctx, A, keep_pattern(ctx, A, keep, 0.0, false));
}

Mat select_norms(ifac_ctx* ctx, const ifac_bsr& A, double tau) {
  return gather_kept(ctx, A, keep_pattern(ctx, A, nullptr, tau, false));
}

Mat compact(ifac_ctx* ctx, Mat&& full, double tau, bool nocopy) {
  if (full.m.nnzb == 0 || !(tau > 0)) return std::move(full);
  Kept k = keep_pattern(ctx, full.m, nullptr, tau, nocopy);
  if (k.n == full.m.nnzb) return std::move(full);  // nothing dropped: no copy
  if (!nocopy) return gather_kept(ctx, full.m, std::move(k));
  // the kept blocks stay in full's value array, which the result takes over
  Mat R(ctx);
  R.m.n = full.m.n;
  R.m.bs = full.m.bs;
  R.m.nb = full.m.nb;
  R.m.nnzb = k.n;
  R.m.row_ptr = k.rp.release();
  R.m.col_idx = k.ci.release();
  R.m.norms = k.norms.release();
  R.vmap = std::move(k.map);
  R.m.val = full.m.val;
  full.m.val = nullptr;
  return R;
}

}  // namespace ifac
