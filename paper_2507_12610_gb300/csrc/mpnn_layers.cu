// Fused layers of the message-passing surrogate (declared in include/mpnn.h):
// the network of width 128 with its gathers, concatenations, residuals and
// segment sums inside the matrix kernels.
//
// Values are those of the layer-by-layer kernels of mpnn.cu: every product
// chain takes its k in the same ascending chunks of 16, every sum the same
// order, every stored value the same rounding.  What changes is what travels
// through memory: layer by layer, a round writes and reads the 800-byte message
// inputs and 512-byte messages of every edge; here an edge costs its two ends'
// 256-byte states: the sender's from L2, its own from memory.
//
// The messages run on tcgen05.mma, whose chains over k in chunks of 16 give the
// bits of the mma.sync chains of mpnn.cu (tested); mma.sync itself runs at about
// 311 TFLOP/s on this chip, a sixth of tcgen05, and would bound them.
#include <algorithm>

#include "../../include/mpnn.h"
#include "mpnn_mma.cuh"
#include "mpnn_tc.cuh"

namespace {

using namespace mpnn;

constexpr uint32_t kRowK = 560;    // bytes of a staged row of 272 bf16 (35 pieces)
constexpr uint32_t kRowDec = 304;  // ... of 144 bf16 (19 pieces)

// rows x cols bf16 (columns c0 .. c0 + cols of a row-major matrix of row
// length ld) into shared memory, rows `row` bytes apart, by all threads
__device__ __forceinline__ void stage(uint32_t dst, uint32_t row, const uint16_t* src, int64_t ld,
                                      int c0, int rows, int cols) {
  const int pieces = cols / 8;
  for (int k = threadIdx.x; k < rows * pieces; k += blockDim.x) {
    const int r = k / pieces, c = k - r * pieces;
    cp16(dst + (uint32_t)r * row + 16u * (uint32_t)c, src + (int64_t)r * ld + c0 + 8 * c);
  }
}

// ---- edges ----------------------------------------------------------------------

// Edge states e = relu(ef W_e), bf16: one chunk of 16, made once for all rounds
// (the 256 bytes an edge are read again in each; making them inside the message
// kernel instead held its pipeline up by a trip through TMEM).  A warp keeps the
// weights' fragments of all 128 columns in registers and takes 16 edges at a
// time, operands straight from global memory, the next ones loaded ahead; bound by
// the writes (1.05 M edges, 304 MB: 58 us; without the loads ahead and with more
// blocks than fit 83).
constexpr int kEdgeThreads = 256;

__global__ void __launch_bounds__(kEdgeThreads)
k_edges(int64_t E, const uint16_t* __restrict__ ef, const uint16_t* __restrict__ We,
        uint16_t* __restrict__ eb) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  uint32_t b[16][2];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint16_t* w = We + (8 * j + g) * 16 + 2 * t4;
    b[j][0] = *reinterpret_cast<const uint32_t*>(w);
    b[j][1] = *reinterpret_cast<const uint32_t*>(w + 8);
  }
  const int64_t nw = (int64_t)gridDim.x * (kEdgeThreads / 32);
  const int64_t tiles = (E + 15) / 16;
  int64_t t = (int64_t)blockIdx.x * (kEdgeThreads / 32) + (threadIdx.x >> 5);
  uint32_t f[4];  // the next tile's features
  const auto load = [&] {
    const int64_t r0 = min(16 * t + g, E - 1), r8 = min(16 * t + g + 8, E - 1);
    const uint32_t* f0 = reinterpret_cast<const uint32_t*>(ef + r0 * 16) + t4;
    const uint32_t* f8 = reinterpret_cast<const uint32_t*>(ef + r8 * 16) + t4;
    f[0] = f0[0];
    f[1] = f8[0];
    f[2] = f0[4];
    f[3] = f8[4];
  };
  if (t < tiles) load();
  while (t < tiles) {
    const int64_t r0 = 16 * t + g, r8 = r0 + 8;
    const uint32_t a0 = f[0], a1 = f[1], a2 = f[2], a3 = f[3];
    t += nw;
    if (t < tiles) load();
#pragma unroll
    for (int q = 0; q < 4; ++q) {  // 32 columns at a time
      float acc[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[j][r] = 0.f;
        mma_bf16(acc[j], a0, a1, a2, a3, b[4 * q + j][0], b[4 * q + j][1]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        // four lanes hold a row's 32 columns in pairs: exchange them so that each
        // lane writes 16 bytes; in step s a lane gets its pairs from lane t4 ^ s
        uint32_t p[4], o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          p[j] = pack_bf16(relu0(acc[j][2 * h]), relu0(acc[j][2 * h + 1]));
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const uint32_t give = t4 == 0 ? p[s] : t4 == 1 ? p[1 ^ s] : t4 == 2 ? p[2 ^ s] : p[3 ^ s];
          const uint32_t got = __shfl_xor_sync(0xffffffffu, give, s);
          const int at = t4 ^ s;
          o[0] = at == 0 ? got : o[0];
          o[1] = at == 1 ? got : o[1];
          o[2] = at == 2 ? got : o[2];
          o[3] = at == 3 ? got : o[3];
        }
        const int64_t row = h ? r8 : r0;
        if (row < E)
          *reinterpret_cast<uint4*>(eb + row * kH + 32 * q + 8 * t4) =
              make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  }
}

// ---- messages -------------------------------------------------------------------

// One round of messages: m_e = relu([h_dst, h_src, e_e, 1] W_m) for every edge
// and M_i = sum over the edges e received by i, ascending.
struct MessageArgs {
  int64_t n, E;
  const int64_t* off;
  const int32_t* src;
  const int32_t* dst;
  const uint16_t* hb;  // [npad][128]
  const uint16_t* eb;  // [E][128]
  const uint16_t* Wm;  // [128][400]
  const float* P1;     // [npad][128] h W_m over the receiver's columns
  uint16_t* Mb;        // [npad][128] rows 0 .. n-1 written
  uint32_t* mask;      // [E][4] or NULL: bit c of row e: message component c > 0
  int tries;           // of a wait
  int32_t* status;     // or NULL: DEM_ERR_TIMEOUT if a wait ran out
};

// One block an SM owns a range of nodes (of about the same cost for every block:
// the start and sum warps work by node, so a node counts as kNodeCost edges; with
// 1 the blocks of a bed's loose top took twice as long as the others) and takes
// their edges 128 at a time: two tiles of
// operands in shared memory, four of accumulators in TMEM.  Products are taken
// transposed: TMEM lane c holds message component c of the tile's edges
// (columns), so that one thread has a component of consecutive edges and sums a
// node's messages in order in a register, without a transposition through shared
// memory.  Per tile:
//   4 producer warps  copy the senders' and the edges' states into shared memory;
//   8 start warps     store the receiver's third of the product into the
//                     accumulators, each group of 4 half of the edges (it is the
//                     same for all edges of a node: it comes from the node kernel,
//                     and the chain over k begins with the receiver's columns, so
//                     the start is exact and saves 8 of 25 chunks);
//   one thread        issues the 17 chunks of the senders, edges and constant;
//   12 sum warps      take the messages from TMEM, relu, and sum them node by node,
//                     each group of 4 every third tile: a group leaves its tile's
//                     first node to the end, when the sum of that node's edges in
//                     the tile before has come from the group before.  (A sum and
//                     its place in the ring of kCarry are taken before the ring comes
//                     round: tile t + 8 starts after tile t + 4 has left its
//                     accumulators, and the group of t + 4 took t + 1 before it.)
// The weights stay in shared memory (72 KB).  Measured on a settled bed of 100,000
// nodes and 1,054,942 edges: 125 us, against 1,230 us for the gather, product and
// sum kernels it replaces (20,000 nodes: 27 us).  Bound by the issue slots (60 %
// busy) that the start and sum warps take for runs of about ten edges, then by the
// L2 reads of both states (52 us of HBM traffic, 20 us of products).  With two
// groups of sum warps 157 us (20,000: 37), with three and two comparisons a column
// 151; the rest is the search for a block's first node.
constexpr int kTileE = 128;
constexpr int kSumGroups = 3;
// first warps of the roles (each on a multiple of 4: a warp reaches the 32 TMEM
// lanes of its number mod 4)
constexpr int kStartWarp = 4 * kSumGroups, kCopyWarp = kStartWarp + 8, kIssueWarp = kCopyWarp + 4;
constexpr int kMsgThreads = 32 * (kIssueWarp + 1);
constexpr uint32_t kPanel = 128 * 128;  // 128 rows of 64 bf16
constexpr uint32_t kPlain = 128 * 32;   // 128 rows of 16 bf16
// stages: senders (2 panels), edge states (2 panels)
constexpr uint32_t kStBytes = 4 * kPanel;
constexpr uint32_t kMsgW = 2 * kStBytes, kMsgWc = kMsgW + 4 * kPanel, kMsgXc = kMsgWc + kPlain,
                   kMsgBytes = kMsgXc + kPlain + 1024;
constexpr int64_t kNodeCost = 8;
constexpr int kRuns = 8;   // nodes whose rows a start group loads together
constexpr int kCarry = 8;  // sums handed from tile to tile, in turn

struct MsgShared {
  uint64_t full[2], mdone[4], ready[4], dfree[4], carried[kCarry];
  uint32_t tmem;
  int node[2];
  int failed;
  int2 start[8][65];          // runs of edges of one node, by start warp
  int2 run[kStartWarp][kTileE + 2];  // ... by sum warp
  float carry[kCarry][128];   // open sum at the end of a tile
};

// piece c (16 bytes) of row r of a pair of swizzled panels
__device__ __forceinline__ uint32_t panel_at(int r, int c) {
  return (uint32_t)(c >> 3) * kPanel + (uint32_t)r * 128u + 16u * (uint32_t)((c & 7) ^ (r & 7));
}

// Receivers of 64 edges (32 q + lane of them) and of the edge before each.
struct Receivers {
  int dst[2], before[2];
  __device__ __forceinline__ void load(const int32_t* d, int64_t from, int64_t e_begin,
                                       int64_t e_end, int lane) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int64_t e = min(from + 32 * q + lane, e_end - 1);
      dst[q] = d[e];
      before[q] = d[max(e - 1, e_begin)];
    }
  }
};

// The accumulators' start of 64 edges: each node's row of P1 once, into its
// edges' columns.  load() lists the runs of edges of one node in `run` (first
// edge, receiver) and loads the first kRuns rows; fill() stores them (columns at d
// of the warp's lanes, component c).
struct Start {
  float p[kRuns];
  int at[kRuns + 1];
  int nrun;
  __device__ __forceinline__ void rows(const MessageArgs& a, const int2* run, int r0, int c) {
#pragma unroll
    for (int i = 0; i < kRuns; ++i) {
      const int2 r = run[min(r0 + i, nrun)];
      at[i] = r.x;
      p[i] = a.P1[(int64_t)r.y * kH + c];
    }
    at[kRuns] = run[min(r0 + kRuns, nrun)].x;
  }
  __device__ __forceinline__ void load(const MessageArgs& a, const Receivers& R, int2* run, int c,
                                       int lane) {
    nrun = 0;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const bool first = (q == 0 && lane == 0) || R.before[q] != R.dst[q];
      const uint32_t bits = __ballot_sync(0xffffffffu, first);
      if (first)
        run[nrun + __popc(bits & ((1u << lane) - 1u))] = make_int2(32 * q + lane, R.dst[q]);
      nrun += __popc(bits);
    }
    if (lane == 0) run[nrun] = make_int2(64, 0);
    __syncwarp();
    rows(a, run, 0, c);
  }
  __device__ __forceinline__ void fill(const MessageArgs& a, const int2* run, uint32_t d, int c) {
    for (int r0 = 0;;) {
#pragma unroll
      for (int i = 0; i < kRuns; ++i)
        if (r0 + i < nrun) tc_fill(d + at[i], __float_as_uint(p[i]), at[i + 1] - at[i]);
      r0 += kRuns;
      if (r0 >= nrun) return;
      rows(a, run, r0, c);
    }
  }
};

// Keep: write the message masks of a training pass (a template: the test for it
// cost the sum warps a branch at every edge).
template <bool Keep>
__global__ void __launch_bounds__(kMsgThreads, 1) k_message(MessageArgs a) {
  extern __shared__ __align__(16) uint8_t smem_any[];
  __shared__ MsgShared S;
  uint8_t* const smem = smem_any + ((1024u - (smem_addr(smem_any) & 1023u)) & 1023u);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t base = smem_addr(smem);
  const auto bar = [&](uint64_t* b) { return smem_addr(b); };
  // weights: W_m columns 128 .. 383 (senders, edges) in panels, 384 .. 399 (the
  // constant) plain; the constant's input [1, 0 x 15] of every row
  for (int k = tid; k < 128 * 34; k += kMsgThreads) {
    const int r = k / 34, c = k - 34 * r;
    const uint16_t* src = a.Wm + (int64_t)r * 400 + 128 + 8 * c;
    cp16(c < 32 ? base + kMsgW + (uint32_t)(c >> 4) * 2u * kPanel + panel_at(r, c & 15)
                : base + kMsgWc + (uint32_t)(c - 32) * 2048u + 16u * r,
         src);
  }
  for (int k = tid; k < 128 * 2; k += kMsgThreads)
    *reinterpret_cast<uint4*>(smem + kMsgXc + (k >> 7) * 2048 + 16 * (k & 127)) =
        make_uint4(k < 128 ? 0x3F80u : 0u, 0u, 0u, 0u);
  cp_commit();
  if (warp < 2) {
    // first node whose edges and nodes before it reach the share; a warp probes 32
    // nodes at a time (one by one the dependent loads were most of the 8 us before
    // the first tile)
    const int64_t share = (a.E + kNodeCost * a.n) * (int64_t)(blockIdx.x + warp) / gridDim.x;
    int64_t lo = 0, hi = a.n;
    while (lo < hi) {
      const int64_t chunk = (hi - lo + 31) / 32, at = lo + lane * chunk;
      const bool before = at < hi && a.off[at] + kNodeCost * at < share;
      const int k = __popc(__ballot_sync(0xffffffffu, before));
      hi = k < 32 ? min(hi, lo + k * chunk) : hi;
      lo = k > 0 ? lo + (k - 1) * chunk + 1 : lo;
    }
    if (lane == 0) S.node[warp] = (int)(blockIdx.x + warp == gridDim.x ? a.n : lo);
  }
  if (tid == 64) {
    for (int b = 0; b < 2; ++b) mbar_init(bar(&S.full[b]), 128);
    for (int b = 0; b < 4; ++b) {
      mbar_init(bar(&S.mdone[b]), 1);
      mbar_init(bar(&S.ready[b]), 256);
      mbar_init(bar(&S.dfree[b]), 128);
    }
    for (int b = 0; b < kCarry; ++b) mbar_init(bar(&S.carried[b]), 128);
    S.failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kIssueWarp) tc_alloc(smem_addr(&S.tmem), 512);
  cp_wait<0>();
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = S.tmem;  // columns 128 b: accumulators of tiles b mod 4
  const int i0 = S.node[0], i1 = S.node[1];
  const int64_t e_begin = a.off[i0], e_end = a.off[i1];
  const int ntile = (int)((e_end - e_begin + kTileE - 1) / kTileE);
  volatile int* failed = &S.failed;

  if (warp == kIssueWarp) {
    // ---- issuer
    if (lane == 0) {
      const uint32_t idesc = tc_idesc(128, 128);
      int t = 0;
      for (; t < ntile; ++t) {
        const int b = t & 1, d = t & 3;
        if (!mbar_wait(bar(&S.full[b]), (t >> 1) & 1, failed, a.tries)) break;
        if (!mbar_wait(bar(&S.ready[d]), (t >> 2) & 1, failed, a.tries)) break;
        tc_fence_after();
        const uint32_t x = base + (uint32_t)b * kStBytes;
#pragma unroll
        for (int ch = 0; ch < 16; ++ch) {
          const uint32_t o = (uint32_t)(ch >> 2) * kPanel + 32u * (ch & 3);
          tc_mma(tmem + 128u * d, desc_sw128(base + kMsgW + o), desc_sw128(x + o), idesc, true);
        }
        tc_mma(tmem + 128u * d, desc_plain(base + kMsgWc, 2048u),
               desc_plain(base + kMsgXc, 2048u), idesc, true);
        tc_commit(bar(&S.mdone[d]));
      }
      // a block that gave up has nobody who waited for the last products: they must
      // not outlive the stages and TMEM
      if (t > 0) mbar_drain(bar(&S.mdone[(t - 1) & 3]), ((t - 1) >> 2) & 1);
    }
    __syncwarp();
  } else if (warp >= kCopyWarp) {
    // ---- producers: warp w copies rows 32 w .. 32 w + 31 of a tile, two a step
    const int w = warp - kCopyWarp;
    int next = ntile > 0 ? a.src[min(e_begin + 32 * w + lane, e_end - 1)] : 0;
    for (int t = 0; t < ntile; ++t) {
      const int b = t & 1;
      if (t > 0) {  // the copies of the tile before have landed
        cp_wait<0>();
        fence_async_smem();
        mbar_arrive(bar(&S.full[b ^ 1]));
      }
      // the products of tile t - 2 have read the stage
      const bool ok = t < 2 || mbar_wait(bar(&S.mdone[(t - 2) & 3]), ((t - 2) >> 2) & 1, failed,
                                         a.tries);
      if (!__all_sync(0xffffffffu, ok)) break;
      const int64_t t0 = e_begin + (int64_t)t * kTileE;
      const int idx = next;
      const uint32_t st = base + (uint32_t)b * kStBytes;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int r = 2 * j + (lane >> 4), c = lane & 15;
        const int s = __shfl_sync(0xffffffffu, idx, r);
        const uint32_t at = st + panel_at(32 * w + r, c);
        cp16(at, a.hb + (int64_t)s * kH + 8 * c);
        cp16(at + 2u * kPanel, a.eb + min(t0 + 32 * w + r, e_end - 1) * kH + 8 * c);
      }
      cp_commit();
      if (t + 1 < ntile) next = a.src[min(t0 + kTileE + 32 * w + lane, e_end - 1)];
    }
    cp_wait<0>();
    fence_async_smem();
    if (ntile > 0) mbar_arrive(bar(&S.full[(ntile - 1) & 1]));
  } else if (warp >= kStartWarp) {
    // ---- start warps: thread = component, group = half of the tile's edges
    const int half = (warp - kStartWarp) >> 2, c = tid & 127;
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    int2* const run = S.start[warp - kStartWarp];
    Receivers R;
    if (ntile > 0) R.load(a.dst, e_begin + 64 * half, e_begin, e_end, lane);
    for (int t = 0; t < ntile; ++t) {
      const int d = t & 3;
      const int64_t t0 = e_begin + (int64_t)t * kTileE;
      Start st;
      st.load(a, R, run, c, lane);
      if (t + 1 < ntile) R.load(a.dst, t0 + kTileE + 64 * half, e_begin, e_end, lane);
      const bool ok = t < 4 || mbar_wait(bar(&S.dfree[d]), ((t - 4) >> 2) & 1, failed, a.tries);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      st.fill(a, run, tmem + lanes + 128u * d + 64u * half, c);
      tc_wait_st();
      tc_fence_before();
      mbar_arrive(bar(&S.ready[d]));
    }
  } else {
    // ---- sum warps: thread = component, group = every third tile
    const int group = warp >> 2, c = tid & 127;
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    int2* const run = S.run[warp];
    int dst[4], after[4];  // receivers of edges 32 q + lane and of the edges after them
    const auto receivers = [&](int64_t t0) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t e = t0 + 32 * q + lane;
        dst[q] = e < e_end ? a.dst[e] : -1;
        after[q] = e + 1 < e_end ? a.dst[e + 1] : -1;
      }
    };
    if (group < ntile) receivers(e_begin + group * kTileE);
    for (int t = group; t < ntile; t += kSumGroups) {
      const int d = t & 3;
      const int64_t t0 = e_begin + (int64_t)t * kTileE;
      // the tile's runs of edges of one node: (edge after the last, receiver); a
      // run that goes on in the next tile has receiver -1
      int nrun = 0;
      const int m = (int)min((int64_t)kTileE, e_end - t0);
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool last = dst[q] >= 0 && dst[q] != after[q];
        const uint32_t bits = __ballot_sync(0xffffffffu, last);
        if (last)
          run[nrun + __popc(bits & ((1u << lane) - 1u))] = make_int2(32 * q + lane + 1, dst[q]);
        nrun += __popc(bits);
      }
      if (lane < 2) run[nrun + lane] = make_int2(m, -1);
      __syncwarp();
      if (t + kSumGroups < ntile) receivers(t0 + kSumGroups * kTileE);
      const bool ok = mbar_wait(bar(&S.mdone[d]), (t >> 2) & 1, failed, a.tries);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const uint32_t acc = tmem + lanes + 128u * d;
      // sum of edges pos .. end - 1, added to s in order
      const auto add = [&](float s, int pos, int end) {
        while (pos < end) {
          // 16 columns, of which pos .. end - 1 count; the last 16 of the tile at
          // most (TMEM ends with the last tile's columns)
          const int from = min(pos, kTileE - 16);
          uint32_t v[16];
          tc_ld16(v, acc + (uint32_t)from);
          // the columns that count, as bits: one test sets seven predicates, where two
          // comparisons a column took half of the sum warps' instructions
          const int stop = min(end - from, 16);
          const uint32_t in = ((1u << stop) - 1u) & ~((1u << (pos - from)) - 1u);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float x = fmaxf(__uint_as_float(v[j]), 0.f);
            if (in >> j & 1u) s += x;
            if (Keep) {
              const uint32_t bits = __ballot_sync(0xffffffffu, x > 0.f);
              if (lane == j && (in >> j & 1u))
                a.mask[(t0 + from + j) * 4 + (warp & 3)] = bits;
            }
          }
          pos = from + 16;
        }
        return s;
      };
      const int2 r0 = run[0];
      int2 r = run[1];
      float open = 0.f;  // sum of the node that goes on in the next tile
      for (int pos = r0.x, i = 2; pos < m; ++i) {
        const int2 next = run[i];
        const float s = add(0.f, pos, r.x);
        if (r.y >= 0)
          a.Mb[(int64_t)r.y * kH + c] = to_bf16(s);
        else
          open = s;
        pos = r.x;
        r = next;
      }
      const bool whole = r0.x == m && r0.y < 0;  // one node from end to end
      if (!whole) {
        S.carry[t & (kCarry - 1)][c] = open;
        mbar_arrive(bar(&S.carried[t & (kCarry - 1)]));
      }
      float s = 0.f;
      if (t > 0) {
        const bool came = mbar_wait(bar(&S.carried[(t - 1) & (kCarry - 1)]),
                                    ((t - 1) / kCarry) & 1, failed, a.tries);
        if (!__all_sync(0xffffffffu, came)) break;
        s = S.carry[(t - 1) & (kCarry - 1)][c];
      }
      s = add(s, 0, r0.x);
      tc_fence_before();
      mbar_arrive(bar(&S.dfree[d]));
      if (whole) {
        S.carry[t & (kCarry - 1)][c] = s;
        mbar_arrive(bar(&S.carried[t & (kCarry - 1)]));
      } else if (r0.y >= 0) {
        a.Mb[(int64_t)r0.y * kH + c] = to_bf16(s);
      }
    }
    // nodes without edges
    for (int i = i0 + tid; i < i1; i += 128 * kSumGroups)
      if (a.off[i] == a.off[i + 1])
        for (int k = 0; k < kH / 8; ++k)
          reinterpret_cast<uint4*>(a.Mb + (int64_t)i * kH)[k] = make_uint4(0u, 0u, 0u, 0u);
  }
  tc_fence_before();
  __syncthreads();
  if (S.failed) {  // a wait ran out: no sums that look like results
    if (tid == 0 && a.status) *a.status = DEM_ERR_TIMEOUT;
    for (int64_t k = tid; k < (int64_t)(i1 - i0) * kH; k += kMsgThreads)
      a.Mb[(int64_t)i0 * kH + k] = 0x7FC0u;
  }
  if (warp == kIssueWarp) {
    tc_fence_after();
    tc_dealloc(tmem, 512);
  }
}

// ---- nodes ----------------------------------------------------------------------

// Encode: h = relu(nf W_n).  Update: h += relu([h, M, 1] W_u).  Then the bf16
// copy of h and either P1 = h W_m over the receiver's columns of the next
// round's message layer, or the decoder's outputs y = [h, 1] W_d.
struct NodeArgs {
  int64_t n, npad;
  const uint16_t* nf;     // encode: [npad][16]
  const uint16_t* hb_in;  // update: [npad][128]
  const uint16_t* Mb;     // update: [npad][128]
  const uint16_t* W;      // encode: [128][16]; update: [128][272]
  const uint16_t* W2;     // next message layer [128][400], or the decoder [64][144]
  float* h;               // [npad][128], updated in place (encode: written)
  uint16_t* hb;           // [npad][128]
  float* out;             // P1 [npad][128] or y [npad][64]
  uint32_t* mask;         // [npad][4] or NULL: bit c: update component c > 0
  int32_t* status;        // or NULL; encode: cleared; decode: NaN outputs if it is set
};

constexpr int kTileN = 64;
constexpr int kNodeGroups = 2;
constexpr uint32_t kNodeW = 0, kNodeW2 = kNodeW + 128 * kRowK, kNodeTiles = kNodeW2 + 128 * kRowH;
constexpr uint32_t kNodeH = 0, kNodeM = kNodeH + kTileN * kRowH, kNodeTile = kNodeM + kTileN * kRowH;
constexpr uint32_t kNodeBytes = kNodeTiles + kNodeGroups * kNodeTile;

// 64 nodes a tile, 8 warps of 32 x 32; a block of two such groups shares the
// weights in shared memory and walks over tiles, each group its own (their loads
// and barriers fill each other's gaps: 100,000 nodes 77 us, 97 us with one group;
// 230 MB, 34 us, is the floor).  A tile a block first: few tiles use all SMs.
template <bool Encode, bool Decode>
__global__ void __launch_bounds__(kNodeGroups * kGroupThreads, 1) k_node(NodeArgs a) {
  extern __shared__ __align__(16) uint8_t smem_any[];
  const int grp = threadIdx.x / kGroupThreads, tid = threadIdx.x % kGroupThreads;
  const int lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const int wm = warp >> 2, wn = warp & 3;
  if (Encode && a.status && blockIdx.x == 0 && threadIdx.x == 0) *a.status = DEM_OK;
  const bool failed = Decode && a.status && *a.status != DEM_OK;
  const uint32_t base = smem_addr(smem_any);  // the weights
  uint8_t* const smem = smem_any + kNodeTiles + grp * kNodeTile;  // the group's tile
  const uint32_t tile = smem_addr(smem);
  constexpr uint32_t kRowW = Encode ? kRow16 : kRowK;
  if (Encode)
    stage(base + kNodeW, kRow16, a.W, 16, 0, 128, 16);
  else
    stage(base + kNodeW, kRowK, a.W, 272, 0, 128, 272);
  if (Decode)
    stage(base + kNodeW2, kRowDec, a.W2, 144, 0, 64, 144);
  else
    stage(base + kNodeW2, kRowH, a.W2, 400, 0, 128, kH);
  cp_commit();
  cp_wait<0>();
  __syncthreads();
  const int64_t step = (int64_t)gridDim.x * kNodeGroups * kTileN;
  for (int64_t r0 = ((int64_t)grp * gridDim.x + blockIdx.x) * kTileN; r0 < a.npad; r0 += step) {
    group_sync(grp);  // the last tile's products have read the stage
    if (Encode) {
      if (tid < 2 * kTileN)
        cp16(tile + kNodeH + (uint32_t)(tid >> 1) * kRow16 + 16u * (tid & 1),
             a.nf + (r0 + (tid >> 1)) * 16 + 8 * (tid & 1));
    } else {
      for (int k = tid; k < kTileN * 16; k += kGroupThreads) {
        const int r = k >> 4, c = k & 15;
        const bool in = r0 + r < a.n;  // rows past n: zero inputs
        const int64_t row = in ? r0 + r : 0;
        cp16(tile + kNodeH + (uint32_t)r * kRowH + 16u * c, a.hb_in + row * kH + 8 * c, in);
        cp16(tile + kNodeM + (uint32_t)r * kRowH + 16u * c, a.Mb + row * kH + 8 * c, in);
      }
    }
    cp_commit();
    cp_wait<0>();
    group_sync(grp);
    bool ones[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) ones[i][h] = r0 + wm * 32 + 16 * i + 8 * h + g < a.n;
    float acc[2][4][4];
    zero(acc);
    const uint32_t la = a_lane(lane, kRowH) + (uint32_t)(wm * 32) * kRowH;
    const uint32_t lb = b_lane(lane, kRowW) + (uint32_t)(wn * 32) * kRowW;
    if (Encode) {
      mma_chain<1>(acc, tile + kNodeH + a_lane(lane, kRow16) + (uint32_t)(wm * 32) * kRow16,
                   kRow16, base + kNodeW + lb, kRowW);
    } else {
      mma_chain<8>(acc, tile + kNodeH + la, kRowH, base + kNodeW + lb, kRowW);
      mma_chain<8>(acc, tile + kNodeM + la, kRowH, base + kNodeW + lb + 256u, kRowW);
      mma_const(acc, ones, base + kNodeW + lb + 512u, kRowW, lane);
    }
    group_sync(grp);  // all inputs read: the new states go over them
    uint32_t bits[2][2] = {{0u, 0u}, {0u, 0u}};
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int row = wm * 32 + 16 * i + 8 * h + g, c = wn * 32 + 8 * j + 2 * t4;
          float2 v = make_float2(relu0(acc[i][j][2 * h]), relu0(acc[i][j][2 * h + 1]));
          float2* hp = reinterpret_cast<float2*>(a.h + (r0 + row) * kH + c);
          if (!Encode) {
            bits[i][h] |= ((v.x > 0.f ? 1u : 0u) | (v.y > 0.f ? 2u : 0u)) << (8 * j + 2 * t4);
            const float2 old = *hp;
            v.x = old.x + v.x;
            v.y = old.y + v.y;
          }
          *hp = v;
          const uint32_t b = pack_bf16(v.x, v.y);
          *reinterpret_cast<uint32_t*>(smem + kNodeH + (uint32_t)row * kRowH + 2u * c) = b;
          *reinterpret_cast<uint32_t*>(a.hb + (r0 + row) * kH + c) = b;
        }
    if (!Encode && a.mask) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t w = bits[i][h];
          w |= __shfl_xor_sync(0xffffffffu, w, 1);
          w |= __shfl_xor_sync(0xffffffffu, w, 2);
          if (t4 == 0) a.mask[(r0 + wm * 32 + 16 * i + 8 * h + g) * 4 + wn] = w;
        }
    }
    group_sync(grp);
    zero(acc);
    if (Decode) {
      // 64 columns: the warps of the first two column groups
      if (wn < 2) {
        const uint32_t ld = b_lane(lane, kRowDec) + (uint32_t)(wn * 32) * kRowDec;
        mma_chain<8>(acc, tile + kNodeH + la, kRowH, base + kNodeW2 + ld, kRowDec);
        mma_const(acc, ones, base + kNodeW2 + ld + 256u, kRowDec, lane);
      }
    } else {
      mma_chain<8>(acc, tile + kNodeH + la, kRowH,
                   base + kNodeW2 + b_lane(lane, kRowH) + (uint32_t)(wn * 32) * kRowH, kRowH);
    }
    constexpr int kOut = Decode ? 64 : kH;
    if (!Decode || wn < 2) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int row = wm * 32 + 16 * i + 8 * h + g, c = wn * 32 + 8 * j + 2 * t4;
            float2 v = make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
            if (Decode && failed) v = make_float2(NAN, NAN);
            *reinterpret_cast<float2*>(a.out + (r0 + row) * kOut + c) = v;
          }
    }
  }
}

template <bool Encode, bool Decode>
int launch_node(const NodeArgs& a, cudaStream_t st) {
  auto* k = &k_node<Encode, Decode>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNodeBytes) !=
      cudaSuccess) {
    cudaGetLastError();
    return DEM_ERR_CUDA;
  }
  // few tiles: one a block
  const int64_t tiles = a.npad / kTileN;
  k<<<(unsigned)std::min<int64_t>(tiles, kSms), kNodeGroups * kGroupThreads, kNodeBytes, st>>>(a);
  return launch_status();
}

}  // namespace

extern "C" {

int mpnn_encode_nodes(int64_t n, int64_t npad, const uint16_t* nf, const uint16_t* Wn,
                      const uint16_t* Wm_next, float* h, uint16_t* hb, float* p1, void* stream) {
  return mpnn_encode_nodes_checked(n, npad, nf, Wn, Wm_next, h, hb, p1, nullptr, stream);
}

int mpnn_encode_nodes_checked(int64_t n, int64_t npad, const uint16_t* nf, const uint16_t* Wn,
                              const uint16_t* Wm_next, float* h, uint16_t* hb, float* p1,
                              int32_t* status, void* stream) {
  if (n <= 0 || npad < n || npad % kTileN || !nf || !Wn || !Wm_next || !h || !hb || !p1 ||
      !aligned16(nf, Wn, Wm_next, h, hb, p1))
    return DEM_ERR_INVALID;
  NodeArgs a{};
  a.n = n;
  a.npad = npad;
  a.nf = nf;
  a.W = Wn;
  a.W2 = Wm_next;
  a.h = h;
  a.hb = hb;
  a.out = p1;
  a.status = status;
  return launch_node<true, false>(a, static_cast<cudaStream_t>(stream));
}

int mpnn_encode_edges(int64_t E, const uint16_t* ef, const uint16_t* We, uint16_t* eb,
                      void* stream) {
  if (E < 0 || E > ((int64_t)1 << 37) || (E > 0 && (!ef || !We || !eb)) ||
      !aligned16(ef, We, eb))
    return DEM_ERR_INVALID;
  if (E == 0) return DEM_OK;
  const int64_t blocks = std::min<int64_t>((E + 127) / 128, 3 * kSms);  // 3 fit an SM
  k_edges<<<(unsigned)blocks, kEdgeThreads, 0, static_cast<cudaStream_t>(stream)>>>(E, ef, We,
                                                                                    eb);
  return launch_status();
}

int mpnn_message_sums(int64_t n, int64_t E, const int64_t* off, const int32_t* nbr,
                      const int32_t* dst, const uint16_t* hb, const uint16_t* eb,
                      const uint16_t* Wm, const float* p1, uint16_t* Mb, uint32_t* mask,
                      void* stream) {
  return mpnn_message_sums_checked(n, E, off, nbr, dst, hb, eb, Wm, p1, Mb, mask, -1, nullptr,
                                   stream);
}

int mpnn_message_sums_checked(int64_t n, int64_t E, const int64_t* off, const int32_t* nbr,
                              const int32_t* dst, const uint16_t* hb, const uint16_t* eb,
                              const uint16_t* Wm, const float* p1, uint16_t* Mb, uint32_t* mask,
                              int32_t tries, int32_t* status, void* stream) {
  if (n <= 0 || n > 0x7fffffff || E < 0 || !off || (E > 0 && (!nbr || !dst || !eb)) || !hb ||
      !Wm || !p1 || !Mb || !aligned16(hb, eb, Wm, p1, Mb, mask))
    return DEM_ERR_INVALID;
  const MessageArgs a{n,  E,  off, nbr,  dst,  hb, eb,
                      Wm, p1, Mb,  mask, tries < 0 ? kMbarTries : tries, status};
  auto* k = mask ? &k_message<true> : &k_message<false>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMsgBytes) !=
      cudaSuccess) {
    cudaGetLastError();
    return DEM_ERR_CUDA;
  }
  const int64_t blocks = std::min<int64_t>(kSms, std::max<int64_t>(1, (E + n + 127) / 128));
  k<<<(unsigned)blocks, kMsgThreads, kMsgBytes, static_cast<cudaStream_t>(stream)>>>(a);
  return launch_status();
}

int mpnn_update_nodes(int64_t n, int64_t npad, const uint16_t* hb_in, const uint16_t* Mb,
                      const uint16_t* Wu, const uint16_t* W_next, int32_t decode, float* h,
                      uint16_t* hb, float* out, uint32_t* mask, void* stream) {
  return mpnn_update_nodes_checked(n, npad, hb_in, Mb, Wu, W_next, decode, h, hb, out, mask,
                                   nullptr, stream);
}

int mpnn_update_nodes_checked(int64_t n, int64_t npad, const uint16_t* hb_in, const uint16_t* Mb,
                              const uint16_t* Wu, const uint16_t* W_next, int32_t decode,
                              float* h, uint16_t* hb, float* out, uint32_t* mask,
                              const int32_t* status, void* stream) {
  if (n <= 0 || npad < n || npad % kTileN || !hb_in || !Mb || !Wu || !W_next || !h || !hb ||
      !out || !aligned16(hb_in, Mb, Wu, W_next, h, hb, out, mask))
    return DEM_ERR_INVALID;
  NodeArgs a{};
  a.n = n;
  a.npad = npad;
  a.hb_in = hb_in;
  a.Mb = Mb;
  a.W = Wu;
  a.W2 = W_next;
  a.h = h;
  a.hb = hb;
  a.out = out;
  a.mask = mask;
  a.status = const_cast<int32_t*>(status);  // (read only)
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return decode ? launch_node<false, true>(a, st) : launch_node<false, false>(a, st);
}

}  // extern "C"
