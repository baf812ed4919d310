// Device-wide inclusive scans with an associative (not necessarily
// commutative) operator on 32-bit values: one tile of kGTile elements per
// block, tiles chained by decoupled look-back (device_util.cuh).  Src and Dst
// are functors that produce element i and consume the scanned value of i.
#pragma once

#include <stdint.h>

#include "apo_internal.cuh"
#include "device_util.cuh"

namespace apo {

// Inclusive scan over n elements (in reverse index order when kReverse), one
// kGTile-element tile per block.  Elements pass through shared memory, so
// that memory is read and written in order while a thread scans kGI
// consecutive ones (padded by a word per kGI: no bank conflicts).  A tile
// waits for a look-back as long as there are tiles in flight, hence 4,096
// elements per tile.
constexpr int kGT = 256, kGI = 16, kGTile = kGT * kGI;
__device__ __forceinline__ int g_pad(int q) { return q + q / kGI; }
template <bool kReverse, class Src, class Op, class Dst>
__global__ void __launch_bounds__(kGT) k_seg_scan(Src src, Dst dst, uint32_t n, Op op, uint32_t ident,
                                                  uint64_t *status, uint32_t *tile_ctr, uint32_t epoch,
                                                  uint32_t *err) {
  __shared__ uint32_t s_tile, s_pre;
  __shared__ uint32_t scr[kGT / 32];
  __shared__ uint32_t sv[kGTile + kGT];
  const int tid = threadIdx.x;
  if (tid == 0) s_tile = atomicAdd(tile_ctr, 1u);
  __syncthreads();
  const uint32_t t = s_tile;
  const uint64_t base = (uint64_t)t * kGTile;
#pragma unroll
  for (int j = 0; j < kGI; ++j) {
    const int q = j * kGT + tid;
    const uint64_t i = base + q;
    sv[g_pad(q)] = i < n ? src(kReverse ? (uint32_t)(n - 1 - i) : (uint32_t)i) : ident;
  }
  __syncthreads();
  uint32_t v[kGI];
#pragma unroll
  for (int i = 0; i < kGI; ++i) v[i] = sv[g_pad(tid * kGI + i)];
#pragma unroll
  for (int i = 1; i < kGI; ++i) v[i] = op(v[i - 1], v[i]);
  uint32_t tot;
  const uint32_t ex = block_exclusive<kGT / 32>(v[kGI - 1], op, ident, scr, &tot);
  if (tid < 32) {
    if (tid == 0) lb_store(&status[t], lb_pack(t == 0 ? kLbInclusive : kLbAggregate, epoch, tot));
    uint32_t pre = ident;
    if (t > 0) {
      pre = lb_exclusive_warp(status, 1, t, epoch, op, ident, err);
      if (tid == 0) lb_store(&status[t], lb_pack(kLbInclusive, epoch, op(pre, tot)));
    }
    if (tid == 0) s_pre = pre;
  }
  __syncthreads();
  const uint32_t r = op(s_pre, ex);
#pragma unroll
  for (int i = 0; i < kGI; ++i) sv[g_pad(tid * kGI + i)] = op(r, v[i]);
  __syncthreads();
#pragma unroll 4
  for (int j = 0; j < kGI; ++j) {
    const int q = j * kGT + tid;
    const uint64_t i = base + q;
    if (i < n) dst(kReverse ? (uint32_t)(n - 1 - i) : (uint32_t)i, sv[g_pad(q)]);
  }
}

template <bool kReverse, class Src, class Op, class Dst>
int seg_scan(apo_ctx *c, Src src, Dst dst, uint32_t n, Op op, uint32_t ident, cudaStream_t s) {
  if (n == 0) return APO_OK;
  const int tiles = ceil_div(n, kGTile);
  APO_TRY(ensure_lookback(c, tiles));
  uint32_t *ctr = c->ps.counters + kCtrMisc + kMiscCompactTiles;
  APO_CUDA_TRY(cudaMemsetAsync(ctr, 0, sizeof(uint32_t), s));
  Launch lp_(c, kKSegScan, n, s);
  k_seg_scan<kReverse><<<tiles, kGT, 0, s>>>(src, dst, n, op, ident, c->ps.lookback, ctr, next_epoch(c),
                                             c->ps.err);
  APO_CUDA_TRY(cudaGetLastError());
  return APO_OK;
}

}  // namespace apo
