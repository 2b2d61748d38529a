// dem_contact_forces_noalloc: contact force and torque sums of a particle
// state with no friction history, computed without allocating any memory.
//
// Its scratch (cell keys, arrival slots, cell counts and offsets, the sorted
// order) lives in one file-scope device array of fixed size, so the call needs
// neither cudaMalloc nor any other allocator.  Host code only ever sees that
// array's name as a host-side stand-in, never a device address: the device
// address is obtained once per device with cudaGetSymbolAddress and passed to
// the kernels.
//
// The arithmetic is the same as the FP64 step of the library for a first
// step (zero springs, particle pairs only, partners summed in ascending index),
// and this file is compiled without multiply-add contraction like that step.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "dem_internal.cuh"
#include "dem_law.cuh"
#include "dem_math.cuh"

namespace dem {
namespace {

constexpr int64_t kNoAllocMaxParticles = 131072;  // 2^17
constexpr int64_t kNoAllocMaxCells = 262144;      // 2^18
constexpr int kTile = 4096;                       // scan tile (elements per block)
constexpr int64_t kMaxTiles = kNoAllocMaxCells / kTile + 1;
constexpr int kMaxTouching = 64;                  // touching partners per particle
constexpr uint32_t kMaxPerCell = 64;              // particles per grid cell

// scratch layout (u32 words)
constexpr int64_t kOffKey = 0;
constexpr int64_t kOffLocal = kOffKey + kNoAllocMaxParticles;
constexpr int64_t kOffOrder = kOffLocal + kNoAllocMaxParticles;
constexpr int64_t kOffCount = kOffOrder + kNoAllocMaxParticles;
constexpr int64_t kOffStart = kOffCount + kNoAllocMaxCells;
constexpr int64_t kOffTiles = kOffStart + kNoAllocMaxCells + 1;
constexpr int64_t kOffStatus = kOffTiles + kMaxTiles + 1;
// 16-byte records: position (float, from the box corner) and radius of each
// sorted slot; 1/R and 1/m (double) of each particle
constexpr int64_t kOffPos = (kOffStatus + 1 + 3) / 4 * 4;
constexpr int64_t kOffInv = kOffPos + 4 * kNoAllocMaxParticles;
constexpr int64_t kScratchWords = kOffInv + 4 * kNoAllocMaxParticles;

// ~7.6 MB, held by every device that loads the library until the process exits
__device__ __align__(256) uint32_t g_noalloc_scratch[kScratchWords];

struct Grid {
  double lo[3], hi[3];
  double inv_h;
  float margin;  // above the rounding of a float distance in the box
  int32_t nc[3];
  int32_t ncells;
};

__device__ __forceinline__ uint32_t cell_of(const Grid& g, double x, double y, double z) {
  int c[3];
  const double p[3] = {x, y, z};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double f = floor((p[a] - g.lo[a]) * g.inv_h);
    int ci = f < 0.0 ? 0 : (f >= (double)g.nc[a] ? g.nc[a] - 1 : (int)f);
    c[a] = ci;
  }
  return (uint32_t)((c[2] * g.nc[1] + c[1]) * g.nc[0] + c[0]);
}

__global__ void na_clear(uint32_t* s, int64_t ncells) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ncells;
       i += (int64_t)gridDim.x * blockDim.x)
    s[kOffCount + i] = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0) s[kOffStatus] = 0u;
}

__device__ __forceinline__ void na_fail(uint32_t* s, uint32_t code) {
  atomicCAS(&s[kOffStatus], 0u, code);
}

// Cell of each particle.  A radius outside (0, r_max], a non-finite or
// out-of-domain position (DEM_ERR_INVALID) or a cell holding more than
// kMaxPerCell particles (DEM_ERR_CAPACITY) sets the status word; the later
// kernels then return at once, so a wrong domain or radius bound cannot make
// the call walk one crowded cell for a long time.
__global__ void na_bin(uint32_t* s, Grid g, const double* R, const double* x, int64_t n,
                       double r_max) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double px = x[3 * i], py = x[3 * i + 1], pz = x[3 * i + 2], r = R[i];
  const double p3[3] = {px, py, pz};
  bool ok = r > 0.0 && r <= r_max;
#pragma unroll
  for (int a = 0; a < 3; ++a) ok = ok && p3[a] >= g.lo[a] && p3[a] <= g.hi[a];  // false for NaN
  uint32_t c = 0;
  if (ok) {
    c = cell_of(g, px, py, pz);
    const uint32_t k = atomicAdd(&s[kOffCount + c], 1u);
    if (k >= kMaxPerCell) na_fail(s, (uint32_t)DEM_ERR_CAPACITY);
    s[kOffLocal + i] = k;
  } else {
    na_fail(s, (uint32_t)DEM_ERR_INVALID);
    s[kOffLocal + i] = 0u;
  }
  s[kOffKey + i] = c;
}

// Exclusive scan of the cell counts: tile totals (one block per tile of
// kTile cells), an exclusive scan of the totals (one warp), then every tile
// scanned in shared memory (256 threads, kTile / 256 consecutive cells each).
// The result is the same whatever the launch shape (integer sums).
constexpr int kScanThreads = 256;
constexpr int kPerThread = kTile / kScanThreads;

__device__ __forceinline__ uint32_t warp_excl_scan(uint32_t v, uint32_t& total) {
  const int lane = threadIdx.x & 31;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - v;
}

__global__ void __launch_bounds__(kScanThreads) na_scan_tiles(uint32_t* s, int64_t ncells) {
  __shared__ uint32_t part[kScanThreads];
  const int64_t base = (int64_t)blockIdx.x * kTile;
  uint32_t sum = 0;
  for (int k = threadIdx.x; k < kTile; k += blockDim.x) {
    const int64_t i = base + k;
    if (i < ncells) sum += s[kOffCount + i];
  }
  part[threadIdx.x] = sum;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) s[kOffTiles + blockIdx.x] = part[0];
}

// one warp: exclusive scan of the tile totals, 32 at a time with a carry
__global__ void na_scan_top(uint32_t* s, int64_t ntiles) {
  uint32_t carry = 0;
  for (int64_t t0 = 0; t0 < ntiles; t0 += 32) {
    const int64_t t = t0 + threadIdx.x;
    const uint32_t v = t < ntiles ? s[kOffTiles + t] : 0u;
    uint32_t total;
    const uint32_t ex = warp_excl_scan(v, total);
    if (t < ntiles) s[kOffTiles + t] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) s[kOffTiles + ntiles] = carry;
}

__global__ void __launch_bounds__(kScanThreads) na_scan_down(uint32_t* s, int64_t ncells,
                                                             int64_t ntiles) {
  __shared__ uint32_t wsum[kScanThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)threadIdx.x * kPerThread;
  uint32_t v[kPerThread];
  uint32_t mine = 0;
#pragma unroll
  for (int k = 0; k < kPerThread; ++k) {
    v[k] = base + k < ncells ? s[kOffCount + base + k] : 0u;
    mine += v[k];
  }
  // exclusive prefix of the threads' sums within the block
  uint32_t wtotal;
  const uint32_t ex = warp_excl_scan(mine, wtotal);
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) wsum[warp] = wtotal;
  __syncthreads();
  uint32_t before = 0;
  for (int k = 0; k < warp; ++k) before += wsum[k];
  uint32_t acc = s[kOffTiles + blockIdx.x] + before + ex;
#pragma unroll
  for (int k = 0; k < kPerThread; ++k) {
    if (base + k < ncells) s[kOffStart + base + k] = acc;
    acc += v[k];
  }
  if (blockIdx.x == ntiles - 1 && threadIdx.x == 0) s[kOffStart + ncells] = s[kOffTiles + ntiles];
}

__global__ void na_scatter(uint32_t* s, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || s[kOffStatus] != 0u) return;
  s[kOffOrder + s[kOffStart + s[kOffKey + i]] + s[kOffLocal + i]] = (uint32_t)i;
}

// The sorted slots: by cell, within a cell by particle index (a particle's rank
// among its cell's), in the array that held the arrival indices; with the
// slot's float position and the particle's inverse radius and mass.
__global__ void na_rank(uint32_t* s, Grid g, const double* R, const double* x, double rho,
                        int64_t n) {
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n || s[kOffStatus] != 0u) return;
  const uint32_t i = s[kOffOrder + a];
  const uint32_t c = s[kOffKey + i];
  uint32_t t = s[kOffStart + c];
  const uint32_t e = s[kOffStart + c + 1];
  for (uint32_t k = t; k < e; ++k)
    if (s[kOffOrder + k] < i) ++t;
  s[kOffLocal + t] = i;
  const double Ri = R[i], m = 4.0 / 3.0 * M_PI * rho * Ri * Ri * Ri;
  reinterpret_cast<float4*>(s + kOffPos)[t] =
      make_float4((float)(x[3 * (int64_t)i] - g.lo[0]), (float)(x[3 * (int64_t)i + 1] - g.lo[1]),
                  (float)(x[3 * (int64_t)i + 2] - g.lo[2]), (float)Ri);
  reinterpret_cast<double2*>(s + kOffInv)[i] = make_double2(1.0 / Ri, 1.0 / m);
}

struct ForceArgs {
  const double* R;
  const double* x;
  const double* v;
  const double* w;
  double* F;
  double* T;
  int64_t n;
  LawConst<double> c;
};

__device__ __forceinline__ V3<double> ld3(const double* a, int64_t i) {
  return mk(a[3 * i], a[3 * i + 1], a[3 * i + 2]);
}

// Whether particles i < j touch; the offset, its length and the overlap.
__device__ __forceinline__ bool touching(const ForceArgs& a, int64_t i, int64_t j, V3<double>& d,
                                         double& dist, double& delta) {
  d = ld3(a.x, i) - ld3(a.x, j);
  const double S = a.R[i] + a.R[j];
  const double d2 = dot(d, d);
  if (d2 > S * S * (1.0 + 1e-10)) return false;
  dist = sqrt(d2);
  delta = S - dist;
  return delta >= 0.0 && dist > 0.0;
}

// Force and torque on particle t from its contact with u, the pair evaluated
// in canonical orientation with zero springs; false if they do not touch.
__device__ __forceinline__ bool pair_force(const ForceArgs& a, const double2* inv, int64_t t,
                                           int64_t u, double c6[6]) {
  const bool t_is_i = t < u;
  const int64_t i = t_is_i ? t : u, j = t_is_i ? u : t;
  V3<double> d;
  double dist, delta;
  if (!touching(a, i, j, d, dist, delta)) return false;
  const V3<double> nh = (1.0 / dist) * d;
  const double Ri = a.R[i], Rj = a.R[j];
  const double2 vi = inv[i], vj = inv[j];
  const double Rs = 1.0 / (vi.x + vj.x);
  const double ms = 1.0 / (vi.y + vj.y);
  const double ri = Ri - delta / 2.0, rj = Rj - delta / 2.0;
  const V3<double> wi = ld3(a.w, i), wj = ld3(a.w, j);
  V3<double> us = mk(0.0, 0.0, 0.0), ur = us;
  double ut = 0.0;
  const LawOut<double> o = contact_law<double, true>(
      a.c, nh, delta, Rs, ms, ri, rj, 1.0 / (1.0 / ri + 1.0 / rj), ld3(a.v, i) - ld3(a.v, j),
      ri * wi + rj * wj, wi - wj, us, ur, ut);
  if (t_is_i) {
    c6[0] = o.f.x; c6[1] = o.f.y; c6[2] = o.f.z;
    c6[3] = o.ti.x; c6[4] = o.ti.y; c6[5] = o.ti.z;
  } else {
    c6[0] = -o.f.x; c6[1] = -o.f.y; c6[2] = -o.f.z;
    c6[3] = o.tj.x; c6[4] = o.tj.y; c6[5] = o.tj.z;
  }
  return true;
}

// Calls f(slot) for the slots of the 27 cells around cell (cx, cy, cz), the
// three cells of a row along x as one range.
template <typename Fn>
__device__ __forceinline__ void for_near_slots(const uint32_t* s, const Grid& g, uint32_t cell,
                                               Fn f) {
  const int cx = (int)(cell % (uint32_t)g.nc[0]);
  const int cy = (int)((cell / (uint32_t)g.nc[0]) % (uint32_t)g.nc[1]);
  const int cz = (int)(cell / ((uint32_t)g.nc[0] * (uint32_t)g.nc[1]));
  const int x0 = cx > 0 ? cx - 1 : 0, x1 = cx + 1 < g.nc[0] ? cx + 1 : g.nc[0] - 1;
  for (int z = cz > 0 ? cz - 1 : 0; z <= cz + 1 && z < g.nc[2]; ++z)
    for (int y = cy > 0 ? cy - 1 : 0; y <= cy + 1 && y < g.nc[1]; ++y) {
      const uint32_t row = (uint32_t)((z * g.nc[1] + y) * g.nc[0]);
      const uint32_t e = s[kOffStart + row + x1 + 1];
      for (uint32_t k = s[kOffStart + row + x0]; k < e; ++k) f(k);
    }
}

// A warp owns PPW consecutive sorted slots.  Each owner lane collects its
// particle's partners that may touch it by a single-precision test with a
// margin (the FP64 pipe takes 16 cycles for a warp instruction, so the ~76
// candidates of a particle must not go through it), ascending by index; then
// the lanes take the warp's collected contacts 32 at a time through the
// double-precision test and the law, all lanes busy, and add them in order, one
// lane per (particle, component).  The kernel is bound by the FP64 pipe (both
// particles of a pair evaluate it: there is no memory for results to hand
// over).  100,000 spheres of a settled drum: a call 896 -> 345 us;
// 2,000 spheres 248 -> 109 us.
// Blocks of one warp, with fewer particles in small calls, spread the warps
// over the SMs and shorten their chains, as in the FP64 step.
template <int PPW>
__global__ void __launch_bounds__(32, 16) na_forces(uint32_t* s, Grid g, ForceArgs a) {
  __shared__ uint32_t near_s[kMaxTouching][32];  // [k][owner lane], ascending per lane
  __shared__ uint32_t seg[33];
  __shared__ uint32_t own_s[32];
  __shared__ double contrib[32][6];
  __shared__ double acc[32][6];
  if (s[kOffStatus] != 0u) return;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x;
  const int64_t slot = (int64_t)blockIdx.x * PPW + lane;
  const bool own = lane < PPW && slot < a.n;
  const float4* pos = reinterpret_cast<const float4*>(s + kOffPos);
  const double2* inv = reinterpret_cast<const double2*>(s + kOffInv);
  const uint32_t* order = s + kOffLocal;
  const int64_t t = own ? (int64_t)order[slot] : 0;
  uint32_t cnt = 0;
  if (own) {
    const float4 X = pos[slot];
    for_near_slots(s, g, s[kOffKey + t], [&](uint32_t k) {
      const float4 Y = pos[k];
      const float dx = X.x - Y.x, dy = X.y - Y.y, dz = X.z - Y.z;
      const float S = X.w + Y.w + g.margin;
      if (dx * dx + dy * dy + dz * dz > S * S * 1.0001f || (int64_t)k == slot) return;
      if (cnt < (uint32_t)kMaxTouching) {
        const uint32_t u = order[k];
        uint32_t j = cnt;
        while (j > 0 && near_s[j - 1][lane] > u) {
          near_s[j][lane] = near_s[j - 1][lane];
          --j;
        }
        near_s[j][lane] = u;
      }
      ++cnt;
    });
  }
  // more than kMaxTouching that may touch: the exact test picks those that do
  if (cnt > (uint32_t)kMaxTouching) {
    cnt = 0;
    for_near_slots(s, g, s[kOffKey + t], [&](uint32_t k) {
      const int64_t u = (int64_t)order[k];
      V3<double> d;
      double dist, delta;
      if (u == t || !touching(a, t < u ? t : u, t < u ? u : t, d, dist, delta)) return;
      if (cnt < (uint32_t)kMaxTouching) {
        uint32_t j = cnt++;
        while (j > 0 && near_s[j - 1][lane] > (uint32_t)u) {
          near_s[j][lane] = near_s[j - 1][lane];
          --j;
        }
        near_s[j][lane] = (uint32_t)u;
      } else {
        na_fail(s, (uint32_t)DEM_ERR_CAPACITY);
      }
    });
  }
  uint32_t incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(full, incl, o);
    if (lane >= o) incl += v;
  }
  seg[lane + 1] = incl;
  if (lane == 0) seg[0] = 0;
  own_s[lane] = (uint32_t)t;
#pragma unroll
  for (int c = 0; c < 6; ++c) acc[lane][c] = 0.0;
  const uint32_t E = __shfl_sync(full, incl, 31);
  __syncwarp();
  for (uint32_t e0 = 0; e0 < E; e0 += 32) {
    const uint32_t e = e0 + lane;
    bool hit = false;
    if (e < E) {
      int tl = 0;
#pragma unroll
      for (int step = PPW / 2; step > 0; step >>= 1)
        if (seg[tl + step] <= e) tl += step;
      double c6[6];
      hit = pair_force(a, inv, (int64_t)own_s[tl], (int64_t)near_s[e - seg[tl]][tl], c6);
      if (hit) {
#pragma unroll
        for (int c = 0; c < 6; ++c) contrib[lane][c] = c6[c];
      }
    }
    const unsigned hits = __ballot_sync(full, hit);
    __syncwarp();
    // particles pa .. pb have contacts in this batch
    const uint32_t last = (e0 + 32 < E ? e0 + 32 : E) - 1u;
    int pa = 0, pb = 0;
#pragma unroll
    for (int step = PPW / 2; step > 0; step >>= 1) {
      if (seg[pa + step] <= e0) pa += step;
      if (seg[pb + step] <= last) pb += step;
    }
    const int njobs = (pb - pa + 1) * 6;
    for (int j = lane; j < njobs; j += 32) {
      const int pp = pa + j / 6, c = j % 6;
      const uint32_t x0 = seg[pp] > e0 ? seg[pp] : e0;
      const uint32_t x1 = seg[pp + 1] < e0 + 32 ? seg[pp + 1] : e0 + 32;
      double h = acc[pp][c];
      for (uint32_t x = x0; x < x1; ++x)
        if (hits >> (x - e0) & 1u) h = h + contrib[x - e0][c];
      acc[pp][c] = h;
    }
    __syncwarp();
  }
  if (own) {
    for (int c = 0; c < 3; ++c) {
      a.F[3 * t + c] = acc[lane][c];
      a.T[3 * t + c] = acc[lane][3 + c];
    }
  }
}

std::mutex g_setup_mutex;
constexpr int kMaxDevices = 64;
uint32_t* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (set-up on the
// first call per device).
int scratch_for_current_device(uint32_t** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return DEM_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || p == nullptr) {
      cudaGetLastError();
      return DEM_ERR_CUDA;
    }
    g_scratch_ptr[dev] = static_cast<uint32_t*>(p);
  }
  *out = g_scratch_ptr[dev];
  return DEM_OK;
}

double beta_host(double e_n) {
  if (e_n <= 0.0) return 1.0;
  if (e_n >= 1.0) return 0.0;
  const double l = std::log(e_n);
  const double r = M_PI / l;
  return 1.0 / std::sqrt(1.0 + r * r);
}

}  // namespace
}  // namespace dem

using namespace dem;

extern "C" int dem_contact_forces_noalloc(const dem_params* params, int64_t n, double r_max,
                                          const double* R, const double* x, const double* v,
                                          const double* w, double* F, double* T,
                                          void* stream) {
  if (!params || !R || !x || !v || !w || !F || !T) return DEM_ERR_INVALID;
  if (n < 1 || n > kNoAllocMaxParticles) return DEM_ERR_INVALID;
  if (!(r_max > 0) || !std::isfinite(r_max)) return DEM_ERR_INVALID;
  const double E = params->E, nu = params->nu;
  if (!(E > 0) || !(nu > -1.0 && nu <= 0.5) || !(params->rho > 0) || !(params->e_n >= 0) ||
      !(params->e_n <= 1) || params->mu_s < 0 || params->mu_r < 0 || params->mu_t < 0 ||
      !(params->dt > 0))
    return DEM_ERR_INVALID;
  Grid g{};
  const double h = 2.0 * r_max;
  int64_t ncells = 1;
  for (int a = 0; a < 3; ++a) {
    const double lo = params->domain_lo[a], hi = params->domain_hi[a];
    if (!(lo < hi) || !std::isfinite(lo) || !std::isfinite(hi)) return DEM_ERR_INVALID;
    const double c = std::ceil((hi - lo) / h);
    if (!(c >= 1) || c > (double)kNoAllocMaxCells) return DEM_ERR_INVALID;
    g.lo[a] = lo;
    g.hi[a] = hi;
    g.nc[a] = (int32_t)c;
    ncells *= (int64_t)c;
    if (ncells > kNoAllocMaxCells) return DEM_ERR_INVALID;
  }
  g.inv_h = 1.0 / h;
  // float positions from the corner: a distance is off by a few units in the
  // last place of the box's largest extent (2^-24 of it, rounded to nearest)
  g.margin = (float)(1e-6 * std::max({g.hi[0] - g.lo[0], g.hi[1] - g.lo[1], g.hi[2] - g.lo[2]}));
  g.ncells = (int32_t)ncells;
  uint32_t* s = nullptr;
  int rc = scratch_for_current_device(&s);
  if (rc != DEM_OK) return rc;
  ForceArgs fa;
  fa.R = R; fa.x = x; fa.v = v; fa.w = w; fa.F = F; fa.T = T; fa.n = n;
  const double G = E / (2.0 * (1.0 + nu));
  fa.c = LawConst<double>{1.0 / ((1.0 - nu * nu) / E + (1.0 - nu * nu) / E),
                          1.0 / ((2.0 - nu) / G + (2.0 - nu) / G), beta_host(params->e_n),
                          params->mu_s, params->mu_r, params->mu_t, params->dt, 0.0};
  fa.c.cs_cn = std::sqrt(fa.c.Gs / (5.0 * fa.c.Es));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t ntiles = (ncells + kTile - 1) / kTile;
  const unsigned nb = (unsigned)((n + 127) / 128);
  na_clear<<<(unsigned)std::min<int64_t>((ncells + 255) / 256, 1024), 256, 0, st>>>(s, ncells);
  na_bin<<<nb, 128, 0, st>>>(s, g, R, x, n, r_max);
  na_scan_tiles<<<(unsigned)ntiles, kScanThreads, 0, st>>>(s, ncells);
  na_scan_top<<<1, 32, 0, st>>>(s, ntiles);
  na_scan_down<<<(unsigned)ntiles, kScanThreads, 0, st>>>(s, ncells, ntiles);
  na_scatter<<<nb, 128, 0, st>>>(s, n);
  na_rank<<<nb, 128, 0, st>>>(s, g, R, x, params->rho, n);
  if (n <= 8192)
    na_forces<8><<<(unsigned)((n + 7) / 8), 32, 0, st>>>(s, g, fa);
  else if (n <= 40960)
    na_forces<16><<<(unsigned)((n + 15) / 16), 32, 0, st>>>(s, g, fa);
  else
    na_forces<32><<<(unsigned)((n + 31) / 32), 32, 0, st>>>(s, g, fa);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return DEM_ERR_CUDA;
  uint32_t status = 0;
  if (cudaMemcpyAsync(&status, s + kOffStatus, sizeof status, cudaMemcpyDeviceToHost, st) !=
          cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    cudaGetLastError();
    return DEM_ERR_CUDA;
  }
  return (int)status;
}
