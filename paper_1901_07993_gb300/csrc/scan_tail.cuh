// scan_tail.cuh -- the exclusive scan of the counts that a kernel's CTAs have
// just written, done by whichever CTA finishes last, with the total also
// written to a word of mapped memory that the host polls.  One launch in place
// of a count kernel, a single-CTA scan and a device-to-host copy: each costs
// about 2 us on the device and 3 us of host time, and a block-sparse product at
// a few thousand rows is made of little else.
#pragma once

#include <cstdint>

namespace ifac {

// Called by every thread of every CTA of the grid after the CTA's counts are
// written; NT = blockDim.x.  ticket: a device word that is zero between
// launches (the last CTA resets it).  out[i] = sum of cnt[0 .. i), out[n] and
// *total (nullable) the sum of all.  True in the CTA that did the scan.
template <int NT>
__device__ __forceinline__ bool scan_tail(const int32_t* cnt, int32_t* out, int n, unsigned* ticket, int32_t* total) {
  constexpr int K = 16, NW = NT / 32;
  __shared__ int32_t wsum[NW];
  __shared__ int32_t carry;
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    carry = 0;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  for (int base = 0; base < n; base += NT * K) {
    const int i0 = base + tid * K;
    int v[K], t = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      v[k] = i0 + k < n ? __ldcg(cnt + i0 + k) : 0;
      t += v[k];
    }
    int x = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    int run = carry + x - t;
#pragma unroll
    for (int w = 0; w < NW; ++w) run += w < wid ? wsum[w] : 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (i0 + k < n) out[i0 + k] = run;
      run += v[k];
    }
    __syncthreads();
    if (tid == NT - 1) carry = run;
    __syncthreads();
  }
  if (tid == 0) {
    out[n] = carry;
    if (total) *total = carry;
    *ticket = 0u;
  }
  return true;
}

}  // namespace ifac
