// List rebuild: cell binning by counting sort, permutation of the particle
// state into cell order, per-cell triangle lists, and the Verlet list build
// with the pair-key history remap.
//
// The paper rebuilds a linked-cell list every step (Sec. 3.3); here cells are
// only used to rebuild a Verlet list with skin (the extension of Sec. 7), and
// the whole rebuild runs only in steps where the control block asks for it.
// Every kernel returns at once otherwise, so a step is a fixed launch
// sequence that a CUDA graph can replay.
//
// Determinism: particles are ordered by cell and, within a cell, by caller
// index; lists are ordered by partner caller index; triangle lists by triangle
// index.  Atomics are used only on integers (counts and arrival slots) whose
// final values do not depend on thread order, and the within-cell sort removes
// the arrival order.  The result depends only on positions.
#include <algorithm>
#include <cfloat>

#include "dem_geom.cuh"
#include "dem_internal.cuh"
#include "dem_math.cuh"

namespace dem {

namespace {

constexpr int kThreads = 256;
constexpr int kTotalSlots = 128;  // slots per entry of the list totals

__device__ __forceinline__ bool rebuilding(const Ctl* ctl) {
  return ctl->rebuild != 0 && ctl->status == 0;
}

__device__ __forceinline__ void set_status(Ctl* ctl, uint32_t code) {
  atomicCAS(&ctl->status, 0u, code);
}

// Shifted float position of slot s in the current dynamic state.
__device__ __forceinline__ float4 posf_of(const Params& p, const void* state, uint32_t s) {
  if (p.mixed) {
    const F8 P = static_cast<const F8*>(state)[s];
    return make_float4(P.hi.x + P.lo.x, P.hi.y + P.lo.y, P.hi.z + P.lo.z, P.hi.w + P.lo.w);
  }
  const D4 P = static_cast<const D4*>(state)[s];
  return make_float4((float)(P.x - p.origin[0]), (float)(P.y - p.origin[1]),
                     (float)(P.z - p.origin[2]), (float)P.w);
}

// Vertex slot j of element k at the reference pose, shifted and rounded like
// the pose arrays (unused slots repeat vertex 0); w = the vertex count in slot 0.
__device__ __forceinline__ float4 ref_vertex(const Params& p, const MeshDev& mesh, int4 tv,
                                             int nvk, int j) {
  const int vi = j < nvk ? (j == 0 ? tv.x : (j == 1 ? tv.y : (j == 2 ? tv.z : tv.w))) : tv.x;
  const D4 r = mesh.ref[vi];
  return make_float4((float)(r.x - p.origin[0]), (float)(r.y - p.origin[1]),
                     (float)(r.z - p.origin[2]), j == 0 ? (float)nvk : 0.f);
}

// A shifted position turned back into the mesh's reference frame: the
// rotation by -theta (cos c, sin s) about the axis through the mesh centre.
__device__ __forceinline__ V3<float> to_mesh_frame(const Params& p, V3<float> q, float c,
                                                   float s) {
  const float wn = (float)p.omega_norm;
  const V3<float> ax = mk(p.f_omega[0] / wn, p.f_omega[1] / wn, p.f_omega[2] / wn);
  const V3<float> cen = mk(p.center_hi[0], p.center_hi[1], p.center_hi[2]);
  const V3<float> r = q - cen;
  return cen + (c * r - s * cross(ax, r) + ((1.f - c) * dot(ax, r)) * ax);
}

// key = cell of each particle; local = its arrival index in the cell.
// Inactive particles (radius 0, awaiting spawning) go to an extra cell after
// the grid that no search visits, in caller order: they are caller indices
// n_active .. n-1, so each one's slot is its caller index.  The last block
// prepares the control block for the kernels that follow.
__global__ void __launch_bounds__(kThreads)
k_bin_count(Ctl* ctl, Params p, StateBufs sb, BinBuf bb, Lists L) {
  if (!rebuilding(ctl)) return;
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x == 0) {
      if (p.omega_norm > 0.0) {  // the rotation of this step, for the mesh-frame lookups
        const double th = p.omega_norm * ((double)ctl->step * p.dt);
        ctl->rot_c = cos(th);
        ctl->rot_s = sin(th);
      }
      ctl->mesh_candidates = 0;
      ctl->max_list_len = 0;
      if (p.n_tri > 0 && *bb.tcell_overflow) set_status(ctl, DEM_ERR_CAPACITY);
    }
    return;
  }
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= p.n) return;
  const float4 X = posf_of(p, buf_of(sb.P, ctl->phase & 1u), s);
  if (X.w == 0.f) {
    const uint32_t c = (uint32_t)p.ncells;
    bb.key[s] = c;
    bb.local[s] = list_of(L, ctl->lphase & 1u).gid[s] - ctl->n_active;
    atomicAdd(&bb.cell_count[c], 1u);
    return;
  }
  const uint32_t c = cell_index(p, cell_coords(p, X.x, X.y, X.z));
  bb.key[s] = c;
  bb.local[s] = atomicAdd(&bb.cell_count[c], 1u);
}

__global__ void __launch_bounds__(kThreads)
k_scatter(const Ctl* ctl, Params p, BinBuf bb) {
  if (!rebuilding(ctl)) return;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= p.n) return;
  bb.order[bb.cell_start[bb.key[s]] + bb.local[s]] = (uint32_t)s;
}

// Move the dynamic state and the per-slot identity into cell order, within a
// cell by caller index: a particle's rank among its cell's (a handful, in
// arrival order in bb.order) gives its slot.
template <typename Rec>
__global__ void __launch_bounds__(kThreads)
k_permute(const Ctl* ctl, Params p, BinBuf bb, StateBufs sb, Lists L) {
  if (!rebuilding(ctl)) return;
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= p.n) return;
  const uint32_t ph = ctl->phase & 1u, lph = ctl->lphase & 1u;
  const Rec* P0 = static_cast<const Rec*>(buf_of(sb.P, ph));
  const Rec* V0 = static_cast<const Rec*>(buf_of(sb.V, ph));
  const Rec* W0 = static_cast<const Rec*>(buf_of(sb.W, ph));
  const Rec* Q0 = static_cast<const Rec*>(buf_of(sb.Q, ph));
  Rec* P1 = static_cast<Rec*>(buf_of(sb.P, ph ^ 1u));
  Rec* V1 = static_cast<Rec*>(buf_of(sb.V, ph ^ 1u));
  Rec* W1 = static_cast<Rec*>(buf_of(sb.W, ph ^ 1u));
  Rec* Q1 = static_cast<Rec*>(buf_of(sb.Q, ph ^ 1u));
  const uint32_t* gid_old = list_of(L, lph).gid;
  uint32_t* gid_new = list_of(L, lph ^ 1u).gid;
  float4* posf_new = list_of(L, lph ^ 1u).posf;
  if (a % kTotalSlots == 0) bb.block_sums[a / kTotalSlots] = 0u;  // for the list build
  const uint32_t s = bb.order[a];
  const uint32_t c = bb.key[s], g = gid_old[s];
  uint32_t t = (uint32_t)a;  // inactive particles arrived in caller order
  if (c < (uint32_t)p.ncells) {
    const uint32_t e = bb.cell_start[c + 1];
    t = bb.cell_start[c];
    for (uint32_t i = t; i < e; ++i)
      if (gid_old[bb.order[i]] < g) ++t;
  }
  const Rec P = P0[s], V = V0[s];
  P1[t] = P;
  V1[t] = V;
  W1[t] = W0[s];
  Q1[t] = Q0[s];
  gid_new[t] = g;
  posf_new[t] = posf_of(p, P0, s);
  bb.src[t] = s;
  D4* inv_new = list_of(L, lph ^ 1u).inv;
  if (inv_new) inv_new[t] = inverses(p, P, V);
}

// ---- triangle cell lists -----------------------------------------------------

// The element cell lists are built once, when the scene is created, in the
// mesh's own frame (the elements at the reference pose), and kept: the mesh is
// rigid and the grid fixed.  A particle looks up the list of the cell that
// holds its position turned back by the mesh's current rotation (distances to
// the elements are the same in both frames).

__global__ void k_clear(uint32_t* a, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    a[i] = 0u;
}

// Cells within reach of element k at the reference pose: its bounding box
// grown by the reach R_k + R_max + skin (+ margin), then a conservative
// per-cell test: the cell centre within reach + half the cell diagonal of the
// element.  pass 0 counts, pass 1 fills.  blockIdx.x is the element; its cells are shared by
// the gridDim.y blocks of that element.
__global__ void k_tri_cells(Params p, MeshDev mesh, BinBuf bb, int pass) {
  const int k = blockIdx.x;
  if (k >= mesh.nt) return;
  // the reference pose (the lists are in the mesh's frame)
  const int4 tv = mesh.tri[k];
  const int nvk = tv.w >= 0 ? 4 : (tv.z >= 0 ? 3 : (tv.y >= 0 ? 2 : 1));
  const float4 A = ref_vertex(p, mesh, tv, nvk, 0), B = ref_vertex(p, mesh, tv, nvk, 1),
               C = ref_vertex(p, mesh, tv, nvk, 2), D = ref_vertex(p, mesh, tv, nvk, 3);
  const float reach = (float)mesh.rad[k] + p.rmax + p.skin + p.list_margin;
  // unused vertex slots repeat vertex 0, so the box of all four is the element's
  const float3 lo = make_float3(fminf(fminf(A.x, B.x), fminf(C.x, D.x)) - reach,
                                fminf(fminf(A.y, B.y), fminf(C.y, D.y)) - reach,
                                fminf(fminf(A.z, B.z), fminf(C.z, D.z)) - reach);
  const float3 hi = make_float3(fmaxf(fmaxf(A.x, B.x), fmaxf(C.x, D.x)) + reach,
                                fmaxf(fmaxf(A.y, B.y), fmaxf(C.y, D.y)) + reach,
                                fmaxf(fmaxf(A.z, B.z), fmaxf(C.z, D.z)) + reach);
  const int3 c0 = cell_coords(p, lo.x, lo.y, lo.z);
  const int3 c1 = cell_coords(p, hi.x, hi.y, hi.z);
  const int nx = c1.x - c0.x + 1, ny = c1.y - c0.y + 1, nz = c1.z - c0.z + 1;
  const int64_t total = (int64_t)nx * ny * nz;
  const float halfdiag = 0.5f * p.h * 1.7320508f * 1.0001f;
  const float lim = reach + halfdiag;
  const V3<float> a = mk(A.x, A.y, A.z), b = mk(B.x, B.y, B.z), c = mk(C.x, C.y, C.z),
                  dd = mk(D.x, D.y, D.z);
  for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.y * blockDim.x) {
    const int cx = c0.x + (int)(i % nx);
    const int cy = c0.y + (int)((i / nx) % ny);
    const int cz = c0.z + (int)(i / ((int64_t)nx * ny));
    const V3<float> q = mk((float)p.base[0] + (cx + 0.5f) * p.h,
                           (float)p.base[1] + (cy + 0.5f) * p.h,
                           (float)p.base[2] + (cz + 0.5f) * p.h);
    // boundary cells also hold clamped particles from outside the box:
    // accept them whenever the triangle is within reach of the clamped region
    const bool edge = cx == 0 || cy == 0 || cz == 0 || cx == p.nc[0] - 1 ||
                      cy == p.nc[1] - 1 || cz == p.nc[2] - 1;
    bool hit = edge;
    if (!hit) {
      const V3<float> y = closest_point_element(q, a, b, c, dd, nvk);
      const V3<float> d = q - y;
      hit = dot(d, d) <= lim * lim;
    }
    if (!hit) continue;
    const uint32_t cell = cell_index(p, make_int3(cx, cy, cz));
    if (pass == 0) {
      atomicAdd(&bb.tcell_count[cell], 1u);
    } else {
      const uint32_t pos = bb.tcell_start[cell] + atomicAdd(&bb.tcell_count[cell], 1u);
      if (pos < bb.tcap) bb.tcell_tri[pos] = (uint32_t)k;
    }
  }
}

// Lists beyond their capacity are reported by the first rebuild.
__global__ void k_tri_cells_check(Params p, BinBuf bb) {
  *bb.tcell_overflow = bb.tcell_start[p.ncells] > bb.tcap ? bb.tcell_start[p.ncells] : 0u;
}

// Order each cell's element list by element index.  One warp per cell: every
// lane ranks its elements against the whole list (indices in a cell are
// distinct, so ranks are a permutation) and writes them to their ranks; a few
// cells (around fan centres) hold a hundred elements or more, which a serial
// insertion sort per cell would make the slowest step of the rebuild.
constexpr int kSortWarps = 8;
constexpr int kSortMax = 512;  // longer lists (not met in practice) sort serially

__global__ void __launch_bounds__(32 * kSortWarps)
k_tri_cell_sort(Params p, BinBuf bb) {
  __shared__ uint32_t buf_s[kSortWarps][kSortMax];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint32_t* buf = buf_s[wib];
  const int64_t nw = (int64_t)gridDim.x * kSortWarps;
  for (int64_t c = (int64_t)blockIdx.x * kSortWarps + wib; c < p.ncells; c += nw) {
    const uint32_t a = bb.tcell_start[c], b = min(bb.tcell_start[c + 1], bb.tcap);
    if (b <= a + 1) continue;
    const uint32_t m = b - a;
    if (m > (uint32_t)kSortMax) {
      if (lane == 0)
        for (uint32_t i = a + 1; i < b; ++i) {
          const uint32_t v = bb.tcell_tri[i];
          uint32_t j = i;
          while (j > a && bb.tcell_tri[j - 1] > v) {
            bb.tcell_tri[j] = bb.tcell_tri[j - 1];
            --j;
          }
          bb.tcell_tri[j] = v;
        }
      __syncwarp();
      continue;
    }
    for (uint32_t i = lane; i < m; i += 32) buf[i] = bb.tcell_tri[a + i];
    __syncwarp();
    for (uint32_t i = lane; i < m; i += 32) {
      const uint32_t v = buf[i];
      uint32_t r = 0;
      for (uint32_t j = 0; j < m; ++j) r += buf[j] < v ? 1u : 0u;
      bb.tcell_tri[a + r] = v;
    }
    __syncwarp();
  }
}

// ---- Verlet list build + history remap -----------------------------------------

// History records are never cleared: a record counts only if its stamp is
// the current step, and a record left in a list buffer from an earlier list
// generation carries a stamp of at most the step that generation ended in,
// which is before the current one.  The buffers start filled with kStampNone
// (at creation and at a load).

// For one new slot t: collect the partners within R_t + R_u + skin (float test
// with a conservative margin) from the 27 surrounding cells, as they come, into
// the temporary fixed-capacity list, and the triangle candidates of the
// particle's cell into its triangle list, carrying each triangle contact's
// history over from the particle's previous list.  k_list_compact sorts the
// pair list and carries the pairs' history over.
//
// G lanes share a particle and take a row's candidates G at a time; the first
// candidates of three rows are loaded together.  Small scenes are bound by a
// particle's chain of ~76 tests, so more lanes share it; large ones by the
// instructions, of which groups need more (lanes idle at the ends of rows).
// Measured (GB300, us, G = 1 / 2 / 4 / 8): box n = 1,000 12.5 / 9.3 / 7.4 / 7.1
// (15.7 with one lane a particle and no loads ahead), drum n = 20,000 30 / 19 /
// 13.4 / 15.9 (32), 200,000 51 / 48 / 56 / -, 1,000,000 181 / 207 / 257 / -.
constexpr int kBuildThreads = 256;

template <typename Hist, int G>
__global__ void __launch_bounds__(kBuildThreads)
k_list_build(Ctl* ctl, Params p, BinBuf bb, Lists L, MeshDev mesh) {
  if (!rebuilding(ctl)) return;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int sub = lane & (G - 1), g0 = lane & ~(G - 1);
  const unsigned below = (1u << sub) - 1u, group = (1u << G) - 1u;
  const int t = (int)(blockIdx.x * (kBuildThreads / G) + threadIdx.x / G);
  const int n = p.n;
  const ListBuf lo = list_of(L, ctl->lphase & 1u);
  const ListBuf ln = list_of(L, (ctl->lphase & 1u) ^ 1u);
  const float4 X = t < n ? ln.posf[t] : make_float4(0.f, 0.f, 0.f, 0.f);
  const bool on = X.w != 0.f;  // (inactive: no list, no mesh candidates)
  const int3 c = cell_coords(p, X.x, X.y, X.z);
  int cnt = 0, ntc = 0;
  bool overflow = false;
  // the cells of a row along x are consecutive in the grid, so the three
  // cells x-1 .. x+1 of a neighbour row are one range of slots: 9 ranges, three
  // (one z) at a time
  const int x0 = max(c.x - 1, 0), x1 = min(c.x + 1, p.nc[0] - 1);
#pragma unroll 1
  for (int dz = -1; dz <= 1; ++dz) {
    const int cz = c.z + dz;
    uint32_t ua[3], ub[3];
    float4 Y[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int cy = c.y + r - 1;
      const bool in = on && cz >= 0 && cz < p.nc[2] && cy >= 0 && cy < p.nc[1];
      ua[r] = in ? bb.cell_start[cell_index(p, make_int3(x0, cy, cz))] + sub : 0u;
      ub[r] = in ? bb.cell_start[cell_index(p, make_int3(x1, cy, cz)) + 1] : 0u;
    }
#pragma unroll
    for (int r = 0; r < 3; ++r)
      if (ua[r] < ub[r]) Y[r] = ln.posf[ua[r]];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      bool more = __any_sync(full, ua[r] < ub[r]);
      while (more) {
        const uint32_t u = ua[r];
        bool hit = false;
        if (u < ub[r]) {
          const float ddx = X.x - Y[r].x, ddy = X.y - Y[r].y, ddz = X.z - Y[r].z;
          const float cut = X.w + Y[r].w + p.skin + p.list_margin;
          hit = ddx * ddx + ddy * ddy + ddz * ddz < cut * cut && u != (uint32_t)t;
        }
        ua[r] = u + G;
        if (ua[r] < ub[r]) Y[r] = ln.posf[ua[r]];
        more = __any_sync(full, ua[r] < ub[r]);
        const unsigned m = (__ballot_sync(full, hit) >> g0) & group;
        if (hit) {
          const int at = cnt + __popc(m & below);
          if (at < p.cap)
            bb.tmp_nbr[(size_t)at * n + t] = u;
          else
            overflow = true;
        }
        cnt += __popc(m);
      }
    }
  }
  // triangle candidates (fixed capacity per particle), history carried over:
  // the group takes the elements of the cell's list G at a time, in order
  if (mesh.nt > 0) {
    // the element list of the particle's cell in the mesh's frame
    int3 cm = c;
    if (p.omega_norm > 0.0) {
      const V3<float> qm = to_mesh_frame(p, mk(X.x, X.y, X.z), (float)ctl->rot_c,
                                         (float)ctl->rot_s);
      cm = cell_coords(p, qm.x, qm.y, qm.z);
    }
    const uint32_t cell = cell_index(p, cm);
    uint32_t i = on ? bb.tcell_start[cell] + sub : 0u;
    const uint32_t b = on ? min(bb.tcell_start[cell + 1], bb.tcap) : 0u;
    const uint32_t stamp_now = (uint32_t)ctl->step;  // records written in the previous step
    const uint32_t pose = pose_at(mesh, ctl->step);
    const Hist* hpm_o = static_cast<const Hist*>(lo.hpm);
    Hist* hpm_n = static_cast<Hist*>(ln.hpm);
    for (; __any_sync(full, i < b); i += G) {
      bool hit = false;
      uint32_t k = 0;
      if (i < b) {
        k = bb.tcell_tri[i];
        const float4* v4 = mesh.curf + 4 * (size_t)(pose + k);
        const float4 A = v4[0], B = v4[1], C = v4[2], D = v4[3];
        const V3<float> q = mk(X.x, X.y, X.z);
        const V3<float> y = closest_point_element(q, mk(A.x, A.y, A.z), mk(B.x, B.y, B.z),
                                                  mk(C.x, C.y, C.z), mk(D.x, D.y, D.z), (int)A.w);
        const V3<float> d = q - y;
        const float cut = X.w + (float)mesh.rad[k] + p.skin + p.list_margin;
        hit = dot(d, d) < cut * cut;
      }
      const unsigned m = (__ballot_sync(full, hit) >> g0) & group;
      if (hit) {
        const int at = ntc + __popc(m & below);
        if (at < p.capm) {
          ln.tric[(size_t)at * n + t] = k;
          // the particle's previous list (ascending, a few elements)
          const uint32_t s = bb.src[t];
          const int nt_o = (int)((lo.meta[s] >> 16) & 0xffu);
          int j = 0;
          while (j < nt_o && lo.tric[(size_t)j * n + s] < k) ++j;
          if (j < nt_o && lo.tric[(size_t)j * n + s] == k) {
            const Hist h = hpm_o[(size_t)j * n + s];
            if (h.stamp == stamp_now) hpm_n[(size_t)at * n + t] = h;
          }
        } else {
          overflow = true;
        }
      }
      ntc += __popc(m);
    }
  }
  if (overflow) set_status(ctl, DEM_ERR_CAPACITY);
  cnt = min(cnt, p.cap);
  if (sub == 0 && t < n) bb.tmp_cnt[t] = (uint32_t)cnt | ((uint32_t)min(ntc, p.capm) << 16);
  // the warp's entries into the total of its kTotalSlots slots
  const uint32_t sum = __reduce_add_sync(full, sub == 0 ? (uint32_t)cnt : 0u);
  if (lane == 0 && sum) atomicAdd(&bb.block_sums[t / kTotalSlots], sum);
}

// Exclusive scan of the list build's totals (one block, ascending); the sum of
// all to offs[n] and the control block.
constexpr int kOffsetThreads = 1024;

__device__ __forceinline__ uint32_t warp_scan_incl(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

__global__ void __launch_bounds__(kOffsetThreads)
k_list_offsets(Ctl* ctl, Params p, BinBuf bb, Lists L, int nblocks) {
  __shared__ uint32_t warp_s[kOffsetThreads / 32];
  if (!rebuilding(ctl)) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int kItems = 8;
  uint32_t carry = 0;
  for (int b0 = 0; b0 < nblocks; b0 += kOffsetThreads * kItems) {
    const int i0 = b0 + (int)threadIdx.x * kItems;
    uint32_t v[kItems], mine = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      v[k] = i0 + k < nblocks ? bb.block_sums[i0 + k] : 0u;
      mine += v[k];
    }
    const uint32_t incl = warp_scan_incl(mine);
    if (lane == 31) warp_s[wid] = incl;
    __syncthreads();
    const uint32_t wtot = warp_scan_incl(warp_s[lane]);  // every warp: all the totals
    const uint32_t before = __shfl_sync(0xffffffffu, wtot, wid > 0 ? wid - 1 : 0);
    uint32_t ex = carry + (wid > 0 ? before : 0u) + incl - mine;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      if (i0 + k < nblocks) bb.block_sums[i0 + k] = ex;
      ex += v[k];
    }
    carry += __shfl_sync(0xffffffffu, wtot, 31);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    list_of(L, (ctl->lphase & 1u) ^ 1u).offs[p.n] = carry;
    ctl->list_entries = carry;
  }
}

// Sort the new pair lists by partner caller index into CSR form and copy each
// pair's friction history record from the previous list where that list has
// the pair and the contact touched in the previous step (with one evaluation
// per pair only the entries of partners with a higher caller index hold
// records).  A warp takes the entries of its slots, kStage at a time: staged
// in shared memory with their caller indices, each entry's place is its rank
// among its particle's entries, and a binary search of the particle's previous
// list (sorted the same way, a cache line or two) finds the old record.
// Sorting here, all lanes busy, instead of by insertion in the list build, one
// thread a particle in local memory, with the kernels of a rebuild down from 24
// to 9, took a rebuild (with its launches) from 635 to 480 us on the
// 1,000,000-sphere drum, from 315 to 170 us on the 200,000-sphere column and
// from 128 to 66 us on the 1,000-sphere box.
// Slots: 32 a warp, 8 in small scenes (fewer batches in a warp's chain: 23.4
// -> 11.2 us at 20,000 spheres, 9.2 -> 6.4 us at 1,000).
template <typename Hist, int Slots>
__global__ void __launch_bounds__(32 * (kTotalSlots / Slots))
k_list_compact(Ctl* ctl, Params p, BinBuf bb, Lists L) {
  constexpr int kWarps = kTotalSlots / Slots;  // a block takes one of the list totals
  constexpr uint32_t kStage = 16 * Slots;      // >= 64, the longest list
  __shared__ uint32_t seg_s[kWarps][33];
  __shared__ uint32_t off_s[kWarps][32];   // previous list: first entry
  __shared__ uint32_t nold_s[kWarps][32];  // and length
  __shared__ uint32_t gid_s[kWarps][32];
  __shared__ uint32_t slot_s[kWarps][kStage];
  __shared__ uint32_t pgid_s[kWarps][kStage];
  __shared__ uint32_t total_s[kWarps];
  if (!rebuilding(ctl)) return;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int n = p.n;
  const int t = (blockIdx.x * kWarps + wib) * Slots + lane;
  const bool own = lane < Slots && t < n;
  const ListBuf lo = list_of(L, ctl->lphase & 1u);
  const ListBuf ln = list_of(L, (ctl->lphase & 1u) ^ 1u);
  uint32_t* seg = seg_s[wib];
  uint32_t* slot = slot_s[wib];
  uint32_t* pgid = pgid_s[wib];
  const uint32_t packed = own ? bb.tmp_cnt[t] : 0u;
  const uint32_t cnt = packed & 0xffffu;
  const uint32_t incl = warp_scan_incl(cnt);
  seg[lane + 1] = incl;
  if (lane == 0) seg[0] = 0;
  if (lane == 31) total_s[wib] = incl;
  uint32_t g_own = 0, off_o = 0, nn_o = 0;
  if (cnt) {
    const uint32_t s = bb.src[t];
    g_own = ln.gid[t];
    off_o = lo.offs[s];
    nn_o = lo.meta[s] & 0xffu;
  }
  off_s[wib][lane] = off_o;
  nold_s[wib][lane] = nn_o;
  gid_s[wib][lane] = g_own;
  __syncthreads();
  uint32_t base = bb.block_sums[blockIdx.x];  // first entry of the warp's first slot
  for (int w = 0; w < wib; ++w) base += total_s[w];
  if (own) ln.offs[t] = base + incl - cnt;
  const bool one_eval = p.pair_res != nullptr;
  const Hist* hpp_o = static_cast<const Hist*>(lo.hpp);
  Hist* hpp_n = static_cast<Hist*>(ln.hpp);
  const uint32_t stamp_now = (uint32_t)ctl->step;  // records written in the previous step
  uint32_t nlow = 0;
  for (int a = 0; a < Slots;) {
    // slots a .. b-1: as many as the stage holds (at least one)
    const uint32_t first = seg[a];
    const unsigned fit =
        __ballot_sync(full, lane >= a && lane < Slots && seg[lane + 1] - first <= kStage);
    const int b = 32 - __clz((int)fit);
    if (lane >= a && lane < b) {
      const uint32_t at = seg[lane] - first;
      for (uint32_t k = 0; k < cnt; ++k) {
        const uint32_t u = bb.tmp_nbr[(size_t)k * n + t];
        const uint32_t g = ln.gid[u];
        slot[at + k] = u;
        pgid[at + k] = g;
        nlow += g < g_own ? 1u : 0u;
      }
    }
    __syncwarp();
    const uint32_t m = seg[b] - first;
    for (uint32_t e = lane; e < m; e += 32) {
      // the slot owning the entry: largest tl with seg[tl] <= first + e
      int tl = 0;
#pragma unroll
      for (int step = Slots / 2; step > 0; step >>= 1)
        if (seg[tl + step] <= first + e) tl += step;
      const uint32_t j0 = seg[tl] - first, j1 = seg[tl + 1] - first;
      const uint32_t g = pgid[e];
      uint32_t pos = base + seg[tl];
      for (uint32_t j = j0; j < j1; ++j) pos += pgid[j] < g ? 1u : 0u;
      ln.nbr[pos] = slot[e];
      ln.ngid[pos] = g;
      if (one_eval && g < gid_s[wib][tl]) continue;
      uint32_t x = off_s[wib][tl], y = x + nold_s[wib][tl];
      const uint32_t end = y;
      while (x < y) {
        const uint32_t mid = (x + y) >> 1;
        if (lo.ngid[mid] < g) x = mid + 1;
        else y = mid;
      }
      if (x < end && lo.ngid[x] == g) {
        const Hist h = hpp_o[x];
        if (h.stamp == stamp_now) hpp_n[pos] = h;
      }
    }
    __syncwarp();
    a = b;
  }
  if (own) ln.meta[t] = cnt | (nlow << 8) | (packed & 0xffff0000u);
  // counters, one atomic a warp
  const uint32_t ntc = __reduce_add_sync(full, packed >> 16);
  const uint32_t most = __reduce_max_sync(full, cnt);
  if (lane == 0) {
    if (ntc) atomicAdd(&ctl->mesh_candidates, ntc);
    if (most > ctl->max_list_len) atomicMax(&ctl->max_list_len, most);
  }
}

__global__ void k_rebuild_end(Ctl* ctl, Params p) {
  if (!rebuilding(ctl)) return;
  ctl->rebuild = 0u;
  ctl->phase ^= 1u;
  ctl->lphase ^= 1u;
  ctl->rebuilds += 1;
  ctl->mesh_angle_ref = p.omega_norm * ((double)ctl->step * p.dt);
}

inline unsigned blocks_for(int64_t n, int threads) {
  return (unsigned)((n + threads - 1) / threads);
}

}  // namespace

// For every entry whose partner u has the lower caller index, the index of
// u's entry for the same pair: u's list is sorted by partner caller index, so
// a binary search over its upper entries finds this particle.  That entry of
// u gets, in return, this entry's index k in this particle's list.
__global__ void __launch_bounds__(128)
k_mirror(Ctl* ctl, Params p, Lists L) {
  if (!rebuilding(ctl)) return;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= p.n) return;
  const ListBuf ln = list_of(L, (ctl->lphase & 1u) ^ 1u);
  const uint32_t meta = ln.meta[t];
  const uint32_t nlow = (meta >> 8) & 0xffu;
  const uint32_t off = ln.offs[t];
  const uint32_t gt = ln.gid[t];
  for (uint32_t k = 0; k < nlow; ++k) {
    const uint32_t u = ln.nbr[off + k];
    const uint32_t mu = ln.meta[u];
    uint32_t lo = ln.offs[u] + ((mu >> 8) & 0xffu), hi = ln.offs[u] + (mu & 0xffu);
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (ln.gid[ln.nbr[mid]] < gt) lo = mid + 1;
      else hi = mid;
    }
    ln.mir[off + k] = lo;
    ln.back[lo] = (uint8_t)k;
  }
}

int64_t list_block_sums_size(int64_t n) { return blocks_for(n, kTotalSlots) + 1; }

void launch_mesh_cells(cudaStream_t st, Ctl* ctl, const Params& p, BinBuf bb, MeshDev mesh) {
  const unsigned gcells = (unsigned)std::min<int64_t>(blocks_for(p.ncells, kThreads), 152 * 16);
  const dim3 elements((unsigned)mesh.nt, (unsigned)p.tri_chunks);
  k_clear<<<gcells, kThreads, 0, st>>>(bb.tcell_count, p.ncells);
  k_tri_cells<<<elements, 128, 0, st>>>(p, mesh, bb, 0);
  // (the scan leaves the counts cleared for the second pass)
  launch_scan(st, ctl, bb.tcell_count, bb.tcell_start, p.ncells, bb.block_sums, bb.scan_done,
              true);
  k_tri_cells_check<<<1, 1, 0, st>>>(p, bb);
  k_tri_cells<<<elements, 128, 0, st>>>(p, mesh, bb, 1);
  k_tri_cell_sort<<<152 * 8, 32 * kSortWarps, 0, st>>>(p, bb);
}

namespace {

template <typename Hist, int G>
void launch_list_build(cudaStream_t st, Ctl* ctl, const Params& p, Lists L, BinBuf bb,
                       MeshDev mesh) {
  k_list_build<Hist, G><<<blocks_for((int64_t)p.n * G, kBuildThreads), kBuildThreads, 0, st>>>(
      ctl, p, bb, L, mesh);
}

template <typename Hist>
void launch_lists(cudaStream_t st, Ctl* ctl, const Params& p, Lists L, BinBuf bb, MeshDev mesh) {
  if (p.n <= 100000)
    launch_list_build<Hist, 4>(st, ctl, p, L, bb, mesh);
  else if (p.n <= 400000)
    launch_list_build<Hist, 2>(st, ctl, p, L, bb, mesh);
  else
    launch_list_build<Hist, 1>(st, ctl, p, L, bb, mesh);
  const unsigned nbl = blocks_for(p.n, kTotalSlots);
  k_list_offsets<<<1, kOffsetThreads, 0, st>>>(ctl, p, bb, L, (int)nbl);
  if (p.n <= 100000)
    k_list_compact<Hist, 8><<<nbl, 4 * kTotalSlots, 0, st>>>(ctl, p, bb, L);
  else
    k_list_compact<Hist, 32><<<nbl, kTotalSlots, 0, st>>>(ctl, p, bb, L);
}

}  // namespace

void launch_rebuild(cudaStream_t st, Ctl* ctl, const Params& p, StateBufs sb, Lists L,
                    BinBuf bb, MeshDev mesh) {
  const unsigned nb = blocks_for(p.n, kThreads);
  k_bin_count<<<nb + 1, kThreads, 0, st>>>(ctl, p, sb, bb, L);
  launch_scan(st, ctl, bb.cell_count, bb.cell_start, p.ncells + 1, bb.block_sums, bb.scan_done,
              true);
  k_scatter<<<nb, kThreads, 0, st>>>(ctl, p, bb);
  if (p.mixed)
    k_permute<F8><<<nb, kThreads, 0, st>>>(ctl, p, bb, sb, L);
  else
    k_permute<D4><<<nb, kThreads, 0, st>>>(ctl, p, bb, sb, L);
  if (p.hist32)
    launch_lists<HistM>(st, ctl, p, L, bb, mesh);
  else
    launch_lists<HistD>(st, ctl, p, L, bb, mesh);
  if (p.pair_res) k_mirror<<<blocks_for(p.n, 128), 128, 0, st>>>(ctl, p, L);
  k_rebuild_end<<<1, 1, 0, st>>>(ctl, p);
}

}  // namespace dem
