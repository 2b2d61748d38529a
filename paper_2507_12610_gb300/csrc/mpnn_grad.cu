// Backward layers of the message-passing surrogate (declared in include/mpnn.h):
// the matrix kernels take their rows through the graph's indices and the relu
// masks that the forward layers left, and write what the next kernel reads.
//
// Gradients of the states keep the order of the layer-by-layer kernels of mpnn.cu
// (each product chain in ascending chunks of 16, each sum in the graph's order),
// so they have the same bits.  Layer by layer a round wrote the gathered inputs
// twice (once transposed), the masked gradients three times and a 1,792-byte input
// gradient for every edge; here it writes the masked gradient once, the 1,024
// bytes that the nodes sum and the edge state's gradient.
#include <algorithm>

#include "../../include/mpnn.h"
#include "mpnn_mma.cuh"

namespace {

using namespace mpnn;

// eight bf16 with those kept whose bit in `bits` is set
__device__ __forceinline__ uint4 masked(uint4 v, uint32_t bits) {
  auto two = [](uint32_t w, uint32_t b) {
    return w & ((b & 1u ? 0x0000ffffu : 0u) | (b & 2u ? 0xffff0000u : 0u));
  };
  return make_uint4(two(v.x, bits), two(v.y, bits >> 2), two(v.z, bits >> 4), two(v.w, bits >> 6));
}

// ---- gradients of a layer's inputs ------------------------------------------------

enum Kind { kDecode, kUpdate, kMessage };

struct InputGradArgs {
  int64_t rows;           // rows of the product
  const uint16_t* dZ;     // [rows][K] bf16; messages: the receivers' [n][128]
  const int32_t* dst;     // messages: the receiver of each edge
  const uint32_t* mask;   // messages: [rows][4]; decode: the last update's [rows][4]
  const uint16_t* W;      // [inputs][K] bf16
  float* dh;              // decode: written; update: added to; [rows][128]
  uint16_t* zb;           // decode, update: bf16 out [rows][128]; messages: see last
  float* dX;              // messages: [rows][256], the receiver's and sender's parts
  float* de;              // messages: [rows][128], the edge state's gradient so far
  const uint16_t* eb;     // messages: the edge states
  uint16_t* zm;           // messages: the edges' gradients [rows][128], written
  int first, last;        // messages: de starts at 0; zb = bf16(de where eb > 0) ends it
};

constexpr int kTile = 64;
constexpr int kGroups = 2;

template <Kind K>
struct InputGrad {
  static constexpr int kIn = K == kDecode ? 64 : 128;                // length of the chain
  static constexpr int kCols = K == kDecode ? 1 : K == kUpdate ? 2 : 3;  // x 128 inputs
  static constexpr uint32_t kRow = K == kDecode ? kRow64 : kRowH;
  static constexpr uint32_t kTiles = kCols * 128 * kRow;  // the rows follow the weights
  static constexpr uint32_t kBytes = kTiles + kGroups * kTile * kRow;
};

// dX = dZ W^T, 64 rows a tile, 8 warps of 32 x 32 over 128 inputs at a time; two
// groups of 8 warps share the weights in shared memory and walk over tiles, each
// its own.  Bound by what it writes (messages: 1,280 B an edge and the read and
// write of 512): a training step on 12 hopper scenes (16,000 nodes) 51 us a round, the
// products of the layer-by-layer step with their gathers and copies 480 us.
template <Kind K>
__global__ void __launch_bounds__(kGroups * kGroupThreads, 1) k_input_grad(InputGradArgs a) {
  using L = InputGrad<K>;
  extern __shared__ __align__(16) uint8_t smem[];
  const int grp = threadIdx.x / kGroupThreads, tid = threadIdx.x % kGroupThreads;
  const int lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const int wm = warp >> 2, wn = warp & 3;
  const uint32_t base = smem_addr(smem);
  uint8_t* const tile_p = smem + L::kTiles + grp * kTile * L::kRow;
  const uint32_t tile = smem_addr(tile_p);
  constexpr int kPieces = L::kIn / 8;
  for (int k = threadIdx.x; k < L::kCols * 128 * kPieces; k += kGroups * kGroupThreads) {
    const int r = k / kPieces, c = k % kPieces;
    cp16(base + (uint32_t)r * L::kRow + 16u * c, a.W + (int64_t)r * L::kIn + 8 * c);
  }
  cp_commit();
  cp_wait<0>();
  __syncthreads();
  const int64_t step = (int64_t)gridDim.x * kGroups * kTile;
  for (int64_t r0 = ((int64_t)grp * gridDim.x + blockIdx.x) * kTile; r0 < a.rows; r0 += step) {
    group_sync(grp);  // the last tile's products have read the stage
#pragma unroll
    for (int k = tid; k < kTile * kPieces; k += kGroupThreads) {
      const int r = k / kPieces, c = k % kPieces;
      const int64_t row = r0 + r;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (row < a.rows) {
        if (K == kMessage) {
          v = masked(*reinterpret_cast<const uint4*>(a.dZ + (int64_t)a.dst[row] * kH + 8 * c),
                     a.mask[row * 4 + (c >> 2)] >> (8 * (c & 3)));
          *reinterpret_cast<uint4*>(a.zm + row * kH + 8 * c) = v;
        } else {
          v = *reinterpret_cast<const uint4*>(a.dZ + row * L::kIn + 8 * c);
        }
      }
      *reinterpret_cast<uint4*>(tile_p + (uint32_t)r * L::kRow + 16u * c) = v;
    }
    group_sync(grp);
#pragma unroll
    for (int q = 0; q < L::kCols; ++q) {
      float acc[2][4][4];
      zero(acc);
      mma_chain<L::kIn / 16>(
          acc, tile + a_lane(lane, L::kRow) + (uint32_t)(wm * 32) * L::kRow, L::kRow,
          base + b_lane(lane, L::kRow) + (uint32_t)(128 * q + wn * 32) * L::kRow, L::kRow);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int64_t row = r0 + wm * 32 + 16 * i + 8 * h + g;
          if (row >= a.rows) continue;
          uint32_t bits = 0u;
          if (K == kDecode) bits = a.mask[row * 4 + wn];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int c = wn * 32 + 8 * j + 2 * t4;
            float2 v = make_float2(0.f + acc[i][j][2 * h], 0.f + acc[i][j][2 * h + 1]);
            if (K == kDecode) {
              *reinterpret_cast<float2*>(a.dh + row * kH + c) = v;
              const uint32_t b = bits >> (8 * j + 2 * t4);
              *reinterpret_cast<uint32_t*>(a.zb + row * kH + c) =
                  pack_bf16(b & 1u ? v.x : 0.f, b & 2u ? v.y : 0.f);
            } else if (K == kUpdate && q == 0) {
              float2* p = reinterpret_cast<float2*>(a.dh + row * kH + c);
              const float2 o = *p;
              *p = make_float2(o.x + v.x, o.y + v.y);
            } else if (K == kUpdate) {
              *reinterpret_cast<uint32_t*>(a.zb + row * kH + c) = pack_bf16(v.x, v.y);
            } else if (q < 2) {
              *reinterpret_cast<float2*>(a.dX + row * 256 + 128 * q + c) = v;
            } else {
              float2* p = reinterpret_cast<float2*>(a.de + row * kH + c);
              if (!a.first) {
                const float2 o = *p;
                v = make_float2(o.x + v.x, o.y + v.y);
              }
              if (a.last) {
                const uint32_t e = *reinterpret_cast<const uint32_t*>(a.eb + row * kH + c);
                *reinterpret_cast<uint32_t*>(a.zb + row * kH + c) =
                    pack_bf16(__uint_as_float(e << 16) > 0.f ? v.x : 0.f,
                              __uint_as_float(e & 0xffff0000u) > 0.f ? v.y : 0.f);
              } else {
                *p = v;
              }
            }
          }
        }
    }
  }
}

template <Kind K>
int launch_input_grad(const InputGradArgs& a, cudaStream_t st) {
  using L = InputGrad<K>;
  auto* k = &k_input_grad<K>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::kBytes) !=
      cudaSuccess) {
    cudaGetLastError();
    return DEM_ERR_CUDA;
  }
  const int64_t tiles = (a.rows + kTile - 1) / kTile;
  k<<<(unsigned)std::min<int64_t>(tiles, kSms), kGroups * kGroupThreads, L::kBytes, st>>>(a);
  return launch_status();
}

// ---- gradients summed over a node's edges -------------------------------------------

// dh = (dh + sum over the edges it receives) + sum over those it sends, ascending,
// then zb = bf16(dh) where the relu before it was positive: by the bits of mask, or
// (mask NULL) where hb > 0.  A warp a node, four columns a lane, four edges in flight.
__global__ void __launch_bounds__(256)
k_node_grad(int64_t n, int64_t npad, const int64_t* __restrict__ off,
            const int32_t* __restrict__ perm, const float* __restrict__ dX,
            const uint32_t* __restrict__ mask, const uint16_t* __restrict__ hb,
            float* __restrict__ dh, uint16_t* __restrict__ zb) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= npad) return;
  float4 s[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
  if (i < n) {
    const int64_t e0 = off[i], e1 = off[i + 1];
    for (int64_t k = e0; k < e1; k += 4) {
      float4 v[2][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u < e1) {
          v[0][u] = *reinterpret_cast<const float4*>(dX + (k + u) * 256 + 4 * lane);
          v[1][u] =
              *reinterpret_cast<const float4*>(dX + (int64_t)perm[k + u] * 256 + 128 + 4 * lane);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u < e1)
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            s[p].x += v[p][u].x;
            s[p].y += v[p][u].y;
            s[p].z += v[p][u].z;
            s[p].w += v[p][u].w;
          }
    }
  }
  float4* d = reinterpret_cast<float4*>(dh + i * kH + 4 * lane);
  float4 o = *d;
  o = make_float4(o.x + s[0].x, o.y + s[0].y, o.z + s[0].z, o.w + s[0].w);
  o = make_float4(o.x + s[1].x, o.y + s[1].y, o.z + s[1].z, o.w + s[1].w);
  *d = o;
  uint32_t bits;
  if (mask) {
    bits = mask[i * 4 + (lane >> 3)] >> (4 * (lane & 7));
  } else {
    const uint2 b = *reinterpret_cast<const uint2*>(hb + i * kH + 4 * lane);
    bits = (__uint_as_float(b.x << 16) > 0.f ? 1u : 0u) |
           (__uint_as_float(b.x & 0xffff0000u) > 0.f ? 2u : 0u) |
           (__uint_as_float(b.y << 16) > 0.f ? 4u : 0u) |
           (__uint_as_float(b.y & 0xffff0000u) > 0.f ? 8u : 0u);
  }
  *reinterpret_cast<uint2*>(zb + i * kH + 4 * lane) =
      make_uint2(pack_bf16(bits & 1u ? o.x : 0.f, bits & 2u ? o.y : 0.f),
                 pack_bf16(bits & 4u ? o.z : 0.f, bits & 8u ? o.w : 0.f));
}

// ---- gradients of the weights --------------------------------------------------------

struct WeightGradArgs {
  int64_t rows, per;             // rows, and rows of a split (a multiple of 16)
  const uint16_t *X0, *X1, *X2;  // input segments, rows of 128 (one input block: of 16)
  const int32_t *idx0, *idx1;    // row of a segment for row r, NULL: r
  const uint16_t* dZ;            // [rows][N]
  int N, kp;                     // columns and rows of G
  float* work;                   // [splits][kp][N]
};

// M inputs x N outputs a block: warps, 16-row and 16-column tiles of a warp
template <int M, int N>
struct WeightGrad {
  static constexpr int kMW = M == 16 ? 1 : N == 64 ? 2 : 4, kNW = 8 / kMW;
  static constexpr int kMT = M / kMW / 16, kNT = N / kNW / 16;
  static constexpr int kStages = 4;
  static constexpr uint32_t kRowX = M == 64 ? kRow64 : kRow16;
  static constexpr uint32_t kRowZ = 2 * N + 16;
  static constexpr uint32_t kZ = kTile * kRowX, kStage = kZ + kTile * kRowZ;
  static constexpr uint32_t kBytes = kStages * kStage;
};

// Part of G = [X_0, X_1, .., 1]^T dZ: block (split, input block, output block) sums
// its rows' products for M inputs (the last input block's also the constant row) and
// N outputs, 64 rows a stage, four stages in flight.  Both operands lie in rows of
// the reduction, so the fragments come by transposing ldmatrix loads: no transposed
// copies.  Splits and chunks are those of mpnn_gemm_split on the transposed operands, so the sums have
// its bits; hence few splits, each a chain of at least 4,096 rows, and small blocks
// to spread a split over the chip: bound by mma.sync's 512 FMA a cycle and SM where
// the blocks fill it, else by a stage's latency.  12 hopper scenes: a message layer
// 58 us (66 us a layer on average with 64 x 128 blocks), an update layer 34 (53) us; with
// the transposes and conversions that it replaces a training step took 1,900 us more.
template <int M, int N>
__global__ void __launch_bounds__(256, M == 64 && N == 64 ? 3 : 2) k_weight_grad(WeightGradArgs a) {
  using L = WeightGrad<M, N>;
  extern __shared__ __align__(16) uint8_t smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3, q = lane >> 3;
  const int wm = warp / L::kNW, wn = warp % L::kNW;
  const uint32_t base = smem_addr(smem);
  const int in0 = M * blockIdx.y, seg = in0 >> 7;  // first input; its segment
  const int out0 = N * blockIdx.z;                 // first output
  const bool ones = M == 64 && blockIdx.y + 1 == gridDim.y && wm == 0;
  constexpr int kLd = M == 64 ? kH : 16;
  const uint16_t* const X = (seg == 0 ? a.X0 : seg == 1 ? a.X1 : a.X2) + (in0 & 127);
  const int32_t* const idx = seg == 0 ? a.idx0 : seg == 1 ? a.idx1 : nullptr;
  const int64_t rb = (int64_t)blockIdx.x * a.per;
  const int64_t re = rb + a.per < a.rows ? rb + a.per : a.rows;
  const int nst = rb < re ? (int)((re - rb + kTile - 1) / kTile) : 0;
  constexpr int kXW = M / 8, kXP = (kTile * kXW + 255) / 256;  // pieces a row, a thread
  constexpr int kZW = N / 8, kZP = kTile * kZW / 256;
  int64_t from[kXP];  // rows of X of the next stage to load
  auto rows_of = [&](int s) {
#pragma unroll
    for (int u = 0; u < kXP; ++u) {
      const int64_t row = rb + (int64_t)s * kTile + (tid + 256 * u) / kXW;
      from[u] = row < re ? (idx ? (int64_t)idx[row] : row) : -1;
    }
  };
  auto load = [&](int s) {
    if (s < nst) {
      const uint32_t st = base + (uint32_t)(s % L::kStages) * L::kStage;
#pragma unroll
      for (int u = 0; u < kXP; ++u) {
        const int k = tid + 256 * u, r = k / kXW, c = k % kXW;
        if (k < kTile * kXW)
          cp16(st + (uint32_t)r * L::kRowX + 16u * c, X + (from[u] < 0 ? 0 : from[u]) * kLd + 8 * c,
               from[u] >= 0);
      }
#pragma unroll
      for (int u = 0; u < kZP; ++u) {
        const int k = tid + 256 * u, r = k / kZW, c = k % kZW;
        const int64_t row = rb + (int64_t)s * kTile + r;
        const bool in = row < re;
        cp16(st + L::kZ + (uint32_t)r * L::kRowZ + 16u * c, a.dZ + (in ? row : 0) * a.N + out0 + 8 * c,
             in);
      }
      rows_of(s + 1);
    }
    cp_commit();
  };
  float acc[L::kMT][2 * L::kNT][4], one[2 * L::kNT][4];
#pragma unroll
  for (int j = 0; j < 2 * L::kNT; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      one[j][r] = 0.f;
#pragma unroll
      for (int i = 0; i < L::kMT; ++i) acc[i][j][r] = 0.f;
    }
  rows_of(0);
#pragma unroll
  for (int s = 0; s < L::kStages - 1; ++s) load(s);
  for (int s = 0; s < nst; ++s) {
    cp_wait<L::kStages - 2>();
    __syncthreads();  // stage s is there, and the reads of stage s - 1 are over
    load(s + L::kStages - 1);
    const uint32_t st = base + (uint32_t)(s % L::kStages) * L::kStage;
    // a small block's few products would wait for each chunk's loads: all of a
    // stage's fragments first, where they fit the registers
    constexpr bool kAhead = L::kMT == 1;
    constexpr int kCh = kTile / 16, kHeld = kAhead ? kCh : 1;
    uint32_t A[kHeld][L::kMT][4], B[kHeld][L::kNT][4];
    auto fragments = [&](int ch, uint32_t (&Ac)[L::kMT][4], uint32_t (&Bc)[L::kNT][4]) {
      // matrices of a transposing load: A by (k, m) halves, B by (k, n) halves
      const uint32_t xa = st + 32u * (wm * L::kMT) + 16u * (q & 1) +
                          (uint32_t)(16 * ch + (lane & 7) + 8 * (q >> 1)) * L::kRowX;
      const uint32_t za = st + L::kZ + 32u * (wn * L::kNT) + 16u * (q >> 1) +
                          (uint32_t)(16 * ch + (lane & 7) + 8 * (q & 1)) * L::kRowZ;
#pragma unroll
      for (int j = 0; j < L::kNT; ++j) ldsm4_t(Bc[j], za + 32u * j);
#pragma unroll
      for (int i = 0; i < L::kMT; ++i) ldsm4_t(Ac[i], xa + 32u * i);
    };
    if (kAhead)
#pragma unroll
      for (int ch = 0; ch < kCh; ++ch) fragments(ch, A[ch % kHeld], B[ch % kHeld]);
#pragma unroll
    for (int ch = 0; ch < kCh; ++ch) {
      const int at = ch % kHeld;
      if (!kAhead) fragments(ch, A[at], B[at]);
#pragma unroll
      for (int i = 0; i < L::kMT; ++i)
#pragma unroll
        for (int j = 0; j < 2 * L::kNT; ++j)
          mma_bf16(acc[i][j], A[at][i][0], A[at][i][1], A[at][i][2], A[at][i][3],
                   B[at][j >> 1][2 * (j & 1)], B[at][j >> 1][2 * (j & 1) + 1]);
      if (ones) {
        const uint32_t u = g == 0 ? 0x3F803F80u : 0u;
#pragma unroll
        for (int j = 0; j < 2 * L::kNT; ++j)
          mma_bf16(one[j], u, 0u, u, 0u, B[at][j >> 1][2 * (j & 1)],
                   B[at][j >> 1][2 * (j & 1) + 1]);
      }
    }
  }
  float* const out = a.work + ((int64_t)blockIdx.x * a.kp + in0) * a.N + out0 +
                     16 * wn * L::kNT + 2 * t4;
#pragma unroll
  for (int j = 0; j < 2 * L::kNT; ++j) {
#pragma unroll
    for (int i = 0; i < L::kMT; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        *reinterpret_cast<float2*>(out + (16 * (wm * L::kMT + i) + 8 * h + g) * a.N + 8 * j) =
            make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
    if (ones && g == 0)
      *reinterpret_cast<float2*>(out + M * a.N + 8 * j) = make_float2(one[j][0], one[j][1]);
  }
}

template <int M, int N>
int launch_weight_grad(const WeightGradArgs& a, int splits, int blocks, cudaStream_t st) {
  using L = WeightGrad<M, N>;
  auto* k = &k_weight_grad<M, N>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::kBytes) !=
      cudaSuccess) {
    cudaGetLastError();
    return DEM_ERR_CUDA;
  }
  k<<<dim3((unsigned)splits, (unsigned)blocks, (unsigned)(a.N / N)), 256, L::kBytes, st>>>(a);
  return launch_status();
}

// G = sum of the splits in ascending order; rows past the inputs are zero.
__global__ void __launch_bounds__(256)
k_weight_sum(int64_t used, int64_t all, int splits, const float* __restrict__ work,
             float* __restrict__ G) {
  const int64_t i = ((int64_t)blockIdx.x * 256 + threadIdx.x);
  if (i >= all) return;
  float v = 0.f;
  if (i < used) {
#pragma unroll 8
    for (int z = 0; z < splits; ++z) v += work[z * all + i];
  }
  G[i] = v;
}

}  // namespace

extern "C" {

int mpnn_grad_decode(int64_t npad, const uint16_t* dyb, const uint16_t* Wdec,
                     const uint32_t* mask, float* dh, uint16_t* zb, void* stream) {
  if (npad <= 0 || !dyb || !Wdec || !mask || !dh || !zb || !aligned16(dyb, Wdec, dh, zb))
    return DEM_ERR_INVALID;
  InputGradArgs a{};
  a.rows = npad;
  a.dZ = dyb;
  a.W = Wdec;
  a.mask = mask;
  a.dh = dh;
  a.zb = zb;
  return launch_input_grad<kDecode>(a, static_cast<cudaStream_t>(stream));
}

int mpnn_grad_update(int64_t npad, const uint16_t* zb, const uint16_t* Wu, float* dh,
                     uint16_t* dMb, void* stream) {
  if (npad <= 0 || !zb || !Wu || !dh || !dMb || !aligned16(zb, Wu, dh, dMb))
    return DEM_ERR_INVALID;
  InputGradArgs a{};
  a.rows = npad;
  a.dZ = zb;
  a.W = Wu;
  a.dh = dh;
  a.zb = dMb;
  return launch_input_grad<kUpdate>(a, static_cast<cudaStream_t>(stream));
}

int mpnn_grad_messages(int64_t E, const int32_t* dst, const uint16_t* dMb, const uint32_t* mask,
                       const uint16_t* Wm, const uint16_t* eb, int32_t first, int32_t last,
                       uint16_t* zm, float* dX, float* de, uint16_t* zeb, void* stream) {
  if (E < 0 || (E > 0 && (!dst || !dMb || !mask || !Wm || !eb || !zm || !dX || !de || !zeb)) ||
      !aligned16(dMb, Wm, eb, zm, dX, de, zeb))
    return DEM_ERR_INVALID;
  if (E == 0) return DEM_OK;
  InputGradArgs a{};
  a.rows = E;
  a.dZ = dMb;
  a.dst = dst;
  a.mask = mask;
  a.W = Wm;
  a.dX = dX;
  a.de = de;
  a.eb = eb;
  a.zm = zm;
  a.zb = zeb;
  a.first = first;
  a.last = last;
  return launch_input_grad<kMessage>(a, static_cast<cudaStream_t>(stream));
}

int mpnn_grad_nodes(int64_t n, int64_t npad, const int64_t* off, const int32_t* perm,
                    const float* dX, const uint32_t* mask, const uint16_t* hb, float* dh,
                    uint16_t* zb, void* stream) {
  if (n <= 0 || npad < n || !off || !perm || !dX || (!mask && !hb) || !dh || !zb ||
      !aligned16(dX, hb, dh, zb))
    return DEM_ERR_INVALID;
  const int64_t blocks = (npad + 7) / 8;
  if (blocks > 0x7fffffff) return DEM_ERR_INVALID;
  k_node_grad<<<(unsigned)blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      n, npad, off, perm, dX, mask, hb, dh, zb);
  return launch_status();
}

int mpnn_grad_weights(int64_t rows, int64_t K, int32_t segments, const uint16_t* X0,
                      const int32_t* idx0, const uint16_t* X1, const int32_t* idx1,
                      const uint16_t* X2, const uint16_t* dZ, int32_t N, int32_t kp,
                      int32_t splits, float* work, float* G, void* stream) {
  // segments 0: one of 16 inputs; else 128 inputs each and a constant after them
  if (rows < 0 || K < rows || K % 16 || segments < 0 || segments > 3 ||
      (segments == 1 ? N != 64 && N != 128 : N != 128) ||
      (segments == 0 ? kp < 16 : kp < 128 * segments + 1) || splits < 1 || splits > 65535 ||
      !X0 || (segments > 1 && !X1) || (segments > 2 && !X2) || !dZ || !work || !G ||
      !aligned16(X0, X1, X2, dZ, work))
    return DEM_ERR_INVALID;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t per = ((K / 16 + splits - 1) / splits) * 16;  // as mpnn_gemm_split's
  const WeightGradArgs a{rows, per, X0, X1, X2, idx0, idx1, dZ, N, kp, work};
  // the wider block reads its operands less often; it needs a block for every SM
  // (4 to 48 blocks in its place: 53 us a layer, 34 with the narrow ones)
  const bool wide = (int64_t)splits * 2 * segments * (N / 64) >= kSms;
  const int rc = segments == 0 ? launch_weight_grad<16, 128>(a, splits, 1, st)
                 : wide        ? launch_weight_grad<64, 64>(a, splits, 2 * segments, st)
                               : launch_weight_grad<64, 32>(a, splits, 2 * segments, st);
  if (rc != DEM_OK) return rc;
  const int64_t all = (int64_t)kp * N;
  const int64_t used = segments == 0 ? 16 * N : (int64_t)(128 * segments + 1) * N;
  k_weight_sum<<<(unsigned)((all + 255) / 256), 256, 0, st>>>(used, all, splits, work, G);
  return launch_status();
}

}  // extern "C"
