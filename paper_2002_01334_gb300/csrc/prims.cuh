// Device primitives: exclusive scan of uint32 and a stable LSD radix sort of (uint64 key,
// uint32 value) pairs, written for this library (no library kernels).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace lpb {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// block-wide exclusive scan of one value per thread; returns the block total in *total
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *smem, uint32_t *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) smem[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    uint32_t w = lane < nw ? smem[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) smem[lane] = w;
  }
  __syncthreads();
  const uint32_t before = (warp > 0 ? smem[warp - 1] : 0u) + x - v;
  *total = smem[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before;
}

__global__ void k_scan_tiles(const uint32_t *in, uint32_t *out, uint32_t *tile_sums, int64_t n) {
  __shared__ uint32_t sm[32];
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  uint32_t v[SCAN_ITEMS];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    v[k] = (base + k < n) ? in[base + k] : 0u;
    s += v[k];
  }
  uint32_t tot;
  uint32_t run = block_exclusive_scan(s, sm, &tot);
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = tot;
}

// single block: exclusive scan of the tile sums in place, total to *total
__global__ void k_scan_sums(uint32_t *sums, int64_t m, uint32_t *total) {
  __shared__ uint32_t sm[32];
  uint32_t carry = 0;
  for (int64_t c = 0; c < m; c += blockDim.x) {
    const int64_t i = c + threadIdx.x;
    const uint32_t v = i < m ? sums[i] : 0u;
    uint32_t tot;
    const uint32_t ex = block_exclusive_scan(v, sm, &tot);
    if (i < m) sums[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void k_scan_add(uint32_t *out, const uint32_t *sums, int64_t n) {
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  const uint32_t add = sums[blockIdx.x];
  for (int k = threadIdx.x; k < SCAN_TILE; k += blockDim.x)
    if (base + k < n) out[base + k] += add;
}

// one block for short arrays: chunks of blockDim * SCAN_ITEMS with a running carry; the exclusive
// scan of in[0..n) into out (in place allowed), the total into *total (may be null)
__global__ void k_scan_one(const uint32_t *in, uint32_t *out, int64_t n, uint32_t *total) {
  __shared__ uint32_t sm[32];
  uint32_t carry = 0;
  const int64_t chunk = (int64_t)blockDim.x * SCAN_ITEMS;
  for (int64_t c0 = 0; c0 < n; c0 += chunk) {
    const int64_t base = c0 + (int64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      v[k] = (base + k < n) ? in[base + k] : 0u;
      s += v[k];
    }
    uint32_t tot;
    uint32_t run = carry + block_exclusive_scan(s, sm, &tot);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      if (base + k < n) out[base + k] = run;
      run += v[k];
    }
    carry += tot;
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

// ---------------------------------------------------------------------------------------
// Several arrays per launch.  The target groups of an evaluation build the same structures from their own
// points; one launch serves all of them (job = blockIdx.y), because at the small end an evaluation is
// a chain of launches (360 for the trees of four groups at N = 3,000, 1.7 of 7.6 ms).
// ---------------------------------------------------------------------------------------
constexpr int MAXJOB = 16;  // target groups: 2 L, L <= 8

struct ScanJob {
  const uint32_t *in;
  uint32_t *out, *sums;  // sums: one per tile
  int64_t n;
};
struct ScanJobs {
  ScanJob j[MAXJOB];
};
// exclusive scans, one block per array, chunks with a running carry
__global__ void k_scan_one_b(const __grid_constant__ ScanJobs J) {
  const ScanJob &j = J.j[blockIdx.x];
  __shared__ uint32_t sm[32];
  uint32_t carry = 0;
  const int64_t chunk = (int64_t)blockDim.x * SCAN_ITEMS;
  for (int64_t c0 = 0; c0 < j.n; c0 += chunk) {
    const int64_t base = c0 + (int64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      v[k] = (base + k < j.n) ? j.in[base + k] : 0u;
      s += v[k];
    }
    uint32_t tot;
    uint32_t run = carry + block_exclusive_scan(s, sm, &tot);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      if (base + k < j.n) j.out[base + k] = run;
      run += v[k];
    }
    carry += tot;
  }
}
__global__ void k_scan_tiles_b(const __grid_constant__ ScanJobs J) {
  const ScanJob &j = J.j[blockIdx.y];
  __shared__ uint32_t sm[32];
  if ((int64_t)blockIdx.x * SCAN_TILE >= j.n) return;
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  uint32_t v[SCAN_ITEMS];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    v[k] = (base + k < j.n) ? j.in[base + k] : 0u;
    s += v[k];
  }
  uint32_t tot;
  uint32_t run = block_exclusive_scan(s, sm, &tot);
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    if (base + k < j.n) j.out[base + k] = run;
    run += v[k];
  }
  if (threadIdx.x == 0) j.sums[blockIdx.x] = tot;
}
__global__ void k_scan_sums_b(const __grid_constant__ ScanJobs J) {
  const ScanJob &j = J.j[blockIdx.x];
  __shared__ uint32_t sm[32];
  const int64_t m = (j.n + SCAN_TILE - 1) / SCAN_TILE;
  uint32_t carry = 0;
  for (int64_t c = 0; c < m; c += blockDim.x) {
    const int64_t i = c + threadIdx.x;
    const uint32_t v = i < m ? j.sums[i] : 0u;
    uint32_t tot;
    const uint32_t ex = block_exclusive_scan(v, sm, &tot);
    if (i < m) j.sums[i] = carry + ex;
    carry += tot;
  }
}
__global__ void k_scan_add_b(const __grid_constant__ ScanJobs J) {
  const ScanJob &j = J.j[blockIdx.y];
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  if (base >= j.n) return;
  const uint32_t add = j.sums[blockIdx.x];
  for (int k = threadIdx.x; k < SCAN_TILE; k += blockDim.x)
    if (base + k < j.n) j.out[base + k] += add;
}

// ---------------------------------------------------------------------------------------
// Stable LSD radix sort of (uint64 key, uint32 value), 8-bit digits, one launch per step for all jobs.
// Tile = 256 threads x 8 rounds; within a tile the items are visited round-major (item =
// round*256 + thread), so ranks follow the input order.
// ---------------------------------------------------------------------------------------
constexpr int RS_THREADS = 256;
constexpr int RS_ROUNDS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS;

struct SortJob {
  const uint64_t *k;
  const uint32_t *v;
  uint64_t *ok;
  uint32_t *ov;
  uint32_t *hist, *offs;
  int64_t n;
  int nblocks, lo, bits;
};
struct SortJobs {
  SortJob j[MAXJOB];
};

__global__ void k_radix_hist(const __grid_constant__ SortJobs J, int pass) {
  const SortJob &j = J.j[blockIdx.y];
  if ((int)blockIdx.x >= j.nblocks) return;
  const int shift = j.lo + 8 * pass;
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * RS_TILE;
  for (int r = 0; r < RS_ROUNDS; ++r) {
    const int64_t i = base + r * RS_THREADS + threadIdx.x;
    if (i < j.n) atomicAdd(&h[(j.k[i] >> shift) & 255u], 1u);
  }
  __syncthreads();
  j.hist[(int64_t)threadIdx.x * j.nblocks + blockIdx.x] = h[threadIdx.x];
}

__global__ void k_radix_scatter(const __grid_constant__ SortJobs J, int pass) {
  const SortJob &j = J.j[blockIdx.y];
  if ((int)blockIdx.x >= j.nblocks) return;
  const int shift = j.lo + 8 * pass;
  __shared__ uint32_t cnt[RS_THREADS / 32][256];
  __shared__ uint32_t base_d[256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  base_d[threadIdx.x] = j.offs[(int64_t)threadIdx.x * j.nblocks + blockIdx.x];
  for (int w = 0; w < RS_THREADS / 32; ++w) cnt[w][threadIdx.x] = 0;
  __syncthreads();
  const int64_t tbase = (int64_t)blockIdx.x * RS_TILE;
  for (int r = 0; r < RS_ROUNDS; ++r) {
    const int64_t i = tbase + r * RS_THREADS + threadIdx.x;
    const bool valid = i < j.n;
    const uint64_t k = valid ? j.k[i] : 0ull;
    const uint32_t v = valid ? j.v[i] : 0u;
    const uint32_t d = valid ? (uint32_t)((k >> shift) & 255u) : 256u;  // 256: padding, ranked last
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const uint32_t lt = peers & ((1u << lane) - 1u);
    const uint32_t rank = __popc(lt);
    if (valid && lt == 0u) cnt[warp][d] = __popc(peers);
    __syncthreads();
    {  // exclusive prefix over warps for digit threadIdx.x, advancing the running base
      const int dd = threadIdx.x;
      uint32_t run = base_d[dd];
      for (int w = 0; w < RS_THREADS / 32; ++w) {
        const uint32_t t = cnt[w][dd];
        cnt[w][dd] = run;
        run += t;
      }
      base_d[dd] = run;
    }
    __syncthreads();
    if (valid) {
      const uint32_t pos = cnt[warp][d] + rank;
      j.ok[pos] = k;
      j.ov[pos] = v;
    }
    __syncthreads();
    for (int w = 0; w < RS_THREADS / 32; ++w) cnt[w][threadIdx.x] = 0;
    __syncthreads();
  }
}

// every pass of a short array in one block: warp w holds the contiguous items [w n/32, (w+1) n/32)
// (rounded to 32), counts its digits, and scatters them in order after a scan over (digit, warp).
// Bound by the latency of its passes (about 1 us a pass and thousand items); above RS_SMALL items the
// three-launch form is faster.  The sorted arrays end in (k, v) after an even number of passes, else in
// (ok, ov).
constexpr int64_t RS_SMALL = 8192;
__global__ void __launch_bounds__(1024) k_radix_small(const __grid_constant__ SortJobs J) {
  const SortJob &j = J.j[blockIdx.x];
  __shared__ uint32_t cnt[32][256];
  __shared__ uint32_t sm[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t per = ((j.n + 31) / 32 + 31) / 32 * 32, b0 = warp * per, b1 = min(b0 + per, j.n);
  uint64_t *k0 = const_cast<uint64_t *>(j.k), *k1 = j.ok;
  uint32_t *v0 = const_cast<uint32_t *>(j.v), *v1 = j.ov;
  for (int shift = j.lo; shift < j.bits; shift += 8) {
    for (int e = threadIdx.x; e < 32 * 256; e += 1024) (&cnt[0][0])[e] = 0;
    __syncthreads();
    for (int64_t i = b0; i < b1; i += 32) {
      const bool valid = i + lane < b1;
      const uint32_t d = valid ? (uint32_t)((k0[i + lane] >> shift) & 255u) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      if (valid && (peers & ((1u << lane) - 1u)) == 0u) cnt[warp][d] += __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    uint32_t mine = 0;  // items of digit threadIdx.x
    if (threadIdx.x < 256)
      for (int w = 0; w < 32; ++w) mine += cnt[w][threadIdx.x];
    uint32_t tot;
    uint32_t run = block_exclusive_scan(mine, sm, &tot);
    if (threadIdx.x < 256)
      for (int w = 0; w < 32; ++w) {
        const uint32_t t = cnt[w][threadIdx.x];
        cnt[w][threadIdx.x] = run;
        run += t;
      }
    __syncthreads();
    for (int64_t i = b0; i < b1; i += 32) {
      const bool valid = i + lane < b1;
      const uint64_t k = valid ? k0[i + lane] : 0ull;
      const uint32_t v = valid ? v0[i + lane] : 0u;
      const uint32_t d = valid ? (uint32_t)((k >> shift) & 255u) : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const uint32_t lt = peers & ((1u << lane) - 1u);
      const uint32_t base = valid ? cnt[warp][d] : 0u;
      __syncwarp();
      if (valid) {
        k1[base + __popc(lt)] = k;
        v1[base + __popc(lt)] = v;
        if (lt == 0u) cnt[warp][d] = base + __popc(peers);
      }
      __syncwarp();
    }
    __syncthreads();  // the block's global writes are visible to it
    uint64_t *tk = k0; k0 = k1; k1 = tk;
    uint32_t *tv = v0; v0 = v1; v1 = tv;
  }
}

}  // namespace lpb
