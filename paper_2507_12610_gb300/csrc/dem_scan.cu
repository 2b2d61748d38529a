// Exclusive prefix sum of a u32 array in two kernels: per-block totals, the
// last block to finish scanning the totals, then a per-block scan that adds its
// offset (and, if asked, clears the input for its next use, which spares a pass
// that clears it).  Integer and order-fixed, so the result is exact and
// deterministic.  The kernels return at once unless the control block says the
// lists are being rebuilt.
#include "dem_internal.cuh"

namespace dem {

namespace {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;  // per thread
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* warp_tot,
                                                         uint32_t* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    uint32_t w = lane < nw ? warp_tot[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    if (lane < nw) warp_tot[lane] = wi - w;
    if (lane == nw - 1) *total = wi;
  }
  __syncthreads();
  return incl - v + warp_tot[wid];
}

// A thread's kScanItems consecutive values from `base` (zeros past n), as
// 128-bit loads where they all exist (base is a multiple of kScanItems).
__device__ __forceinline__ uint32_t load_items(const uint32_t* in, int64_t base, int64_t n,
                                               uint32_t (&v)[kScanItems]) {
  uint32_t s = 0;
  if (base + kScanItems <= n) {
    const uint4* q = reinterpret_cast<const uint4*>(in + base);
#pragma unroll
    for (int k = 0; k < kScanItems / 4; ++k) {
      const uint4 x = q[k];
      v[4 * k] = x.x;
      v[4 * k + 1] = x.y;
      v[4 * k + 2] = x.z;
      v[4 * k + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = base + k < n ? in[base + k] : 0u;
  }
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) s += v[k];
  return s;
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_reduce(const Ctl* ctl, const uint32_t* in, int64_t n, uint32_t* block_sums,
              uint32_t* done) {
  if (!ctl->rebuild || ctl->status) return;
  __shared__ uint32_t warp_tot[32];
  __shared__ uint32_t total;
  __shared__ bool last;
  uint32_t v[kScanItems];
  const uint32_t s =
      load_items(in, (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems, n, v);
  block_exclusive_scan(s, warp_tot, &total);
  if (threadIdx.x == 0) {
    block_sums[blockIdx.x] = total;
    __threadfence();
    // wraps to zero at the last block, ready for the next scan
    last = atomicInc(done, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int64_t nblocks = gridDim.x;
  uint32_t carry = 0;
  for (int64_t b0 = 0; b0 < nblocks; b0 += kScanThreads) {
    const int64_t i = b0 + threadIdx.x;
    const uint32_t x = i < nblocks ? __ldcg(block_sums + i) : 0u;
    const uint32_t ex = block_exclusive_scan(x, warp_tot, &total);
    if (i < nblocks) block_sums[i] = carry + ex;
    carry += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) block_sums[nblocks] = carry;
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_down(const Ctl* ctl, uint32_t* in, uint32_t* out, int64_t n, const uint32_t* block_sums,
            int64_t nblocks, bool clear) {
  if (!ctl->rebuild || ctl->status) return;
  __shared__ uint32_t warp_tot[32];
  __shared__ uint32_t total;
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  const uint32_t s = load_items(in, base, n, v);
  uint32_t ex = block_exclusive_scan(s, warp_tot, &total) + block_sums[blockIdx.x];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {  // to exclusive offsets
    const uint32_t x = v[k];
    v[k] = ex;
    ex += x;
  }
  if (base + kScanItems <= n) {
    uint4* q = reinterpret_cast<uint4*>(out + base);
    uint4* z = reinterpret_cast<uint4*>(in + base);
#pragma unroll
    for (int k = 0; k < kScanItems / 4; ++k) {
      q[k] = make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
      if (clear) z[k] = make_uint4(0u, 0u, 0u, 0u);
    }
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
      if (base + k < n) {
        out[base + k] = v[k];
        if (clear) in[base + k] = 0u;
      }
  }
  if (blockIdx.x == nblocks - 1 && threadIdx.x == 0) out[n] = block_sums[nblocks];
}

}  // namespace

int64_t scan_block_sums_size(int64_t n) { return (n + kScanTile - 1) / kScanTile + 1; }

// out has n + 1 entries; out[n] is the total.  in and out start on 16-byte
// boundaries.
void launch_scan(cudaStream_t st, const Ctl* ctl, uint32_t* in, uint32_t* out, int64_t n,
                 uint32_t* block_sums, uint32_t* done, bool clear) {
  const int64_t nb = (n + kScanTile - 1) / kScanTile;
  k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, st>>>(ctl, in, n, block_sums, done);
  k_scan_down<<<(unsigned)nb, kScanThreads, 0, st>>>(ctl, in, out, n, block_sums, nb, clear);
}

}  // namespace dem
