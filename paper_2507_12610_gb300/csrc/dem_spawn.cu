// Particle spawning (arXiv 2507.12610, Sec. 3.1, "Particle generation").
//
// One block per spawn event.  The attempts of an event depend on each other (a
// kept sphere blocks later ones, a failed attempt hands its radius to the next),
// but until an attempt succeeds all that the next ones need is known: the radius
// carried over and, from the number of draws so far, their centres.  So the
// warps test the next kSpawnWarps attempts at once, as if each before them
// failed; the first that succeeds is kept, and those after it are taken again.
// An event then costs one test per kSpawnWarps attempts and one per kept sphere
// instead of one per attempt: 64 attempts above the 20,000-row heap took 225 us
// an event with one warp, about 45 us now.  The lanes of a warp share its
// test: the particles of the 27 cells around the centre (binned at the last list
// rebuild; they have moved less than the skin since, and a cell is wider than
// two radii plus the skin), the spheres kept earlier in the event, and the mesh
// elements listed for the centre's cell; spheres clearly apart in single precision,
// and elements whose box is, are left out of the double-precision test.  Kept particles
// take the next inactive caller index, whose slot is its caller index (inactive
// particles sit at the end of the slot order in caller order, see the binning),
// and the control block asks for a list rebuild at the next step.  A new
// particle cannot touch anything at the positions of this step, so it needs no
// list entries before that rebuild; what the step reads of it beside its state
// (DEM_FP64: ListBuf::inv, whose c_i is the drag of that first step) is written here.
//
// Compiled without FMA contraction: the centre and radius of a kept sphere
// are the same bits as those of the plain evaluation of the same formulas.
#include "dem_geom.cuh"
#include "dem_internal.cuh"
#include "dem_math.cuh"
#include "dem_step_common.cuh"

namespace dem {

namespace {

// k-th uniform in [0, 1) of the spawn stream: SplitMix64 (Steele, Lea & Flood,
// "Fast splittable pseudorandom number generators", OOPSLA 2014) evaluated at
// seed + (k + 1) * 0x9E3779B97F4A7C15, top 53 bits.
__device__ __forceinline__ double spawn_uniform(uint64_t seed, uint64_t k) {
  uint64_t z = seed + (k + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

__device__ __forceinline__ double lerp_box(double lo, double hi, double u) {
  return lo + u * (hi - lo);
}

__device__ __forceinline__ void split_ff(double a, float& hi, float& lo) {
  hi = (float)a;
  lo = (float)(a - (double)hi);
}

struct Sphere {
  double x, y, z, r;
};

__device__ __forceinline__ Sphere sphere_of(const Params&, const D4& P) {
  return Sphere{P.x, P.y, P.z, P.w};
}
__device__ __forceinline__ Sphere sphere_of(const Params& p, const F8& P) {
  return Sphere{p.origin[0] + ((double)P.hi.x + (double)P.lo.x),
                p.origin[1] + ((double)P.hi.y + (double)P.lo.y),
                p.origin[2] + ((double)P.hi.z + (double)P.lo.z),
                (double)P.hi.w + (double)P.lo.w};
}

// |c - x_j| < r + R_j, written as the plain squared comparison
__device__ __forceinline__ bool overlaps(double cx, double cy, double cz, double r,
                                         const Sphere& o) {
  const double dx = cx - o.x, dy = cy - o.y, dz = cz - o.z;
  const double s = r + o.r;
  return dx * dx + dy * dy + dz * dz < s * s;
}

__device__ __forceinline__ void put_new(const Params& p, D4* P, D4* V, D4* W, D4* Q, uint32_t i,
                                        double cx, double cy, double cz, double r) {
  const double m = 4.0 / 3.0 * M_PI * p.rho * r * r * r;
  P[i] = make_D4(cx, cy, cz, r);
  V[i] = make_D4(p.sp_v0[0], p.sp_v0[1], p.sp_v0[2], m);
  W[i] = make_D4(p.sp_w0[0], p.sp_w0[1], p.sp_w0[2], 0.0);
  Q[i] = make_D4(1.0, 0.0, 0.0, 0.0);
}

__device__ __forceinline__ void put_new(const Params& p, F8* P, F8* V, F8* W, F8* Q, uint32_t i,
                                        double cx, double cy, double cz, double r) {
  const double m = 4.0 / 3.0 * M_PI * p.rho * r * r * r;
  F8 a, b, c, d;
  split_ff(cx - p.origin[0], a.hi.x, a.lo.x);
  split_ff(cy - p.origin[1], a.hi.y, a.lo.y);
  split_ff(cz - p.origin[2], a.hi.z, a.lo.z);
  split_ff(r, a.hi.w, a.lo.w);
  split_ff(p.sp_v0[0], b.hi.x, b.lo.x);
  split_ff(p.sp_v0[1], b.hi.y, b.lo.y);
  split_ff(p.sp_v0[2], b.hi.z, b.lo.z);
  b.hi.w = (float)m;
  b.lo.w = (float)(1.0 / m);
  split_ff(p.sp_w0[0], c.hi.x, c.lo.x);
  split_ff(p.sp_w0[1], c.hi.y, c.lo.y);
  split_ff(p.sp_w0[2], c.hi.z, c.lo.z);
  c.hi.w = (float)(1.0 / r);
  c.lo.w = 0.f;
  d.hi = make_float4(1.f, 0.f, 0.f, 0.f);
  d.lo = make_float4(0.f, 0.f, 0.f, 0.f);
  P[i] = a;
  V[i] = b;
  W[i] = c;
  Q[i] = d;
}

// Whether the sphere at shifted float centre C with radius r is clearly apart
// from particle record P: the centres' distance in single precision exceeds the
// sum of the radii by more than its rounding (list_margin covers several units
// in the last place of the coordinates).  DEM_FP64 records go straight to the
// double-precision test (rounding them costs as much).
__device__ __forceinline__ bool clearly_apart(const Params& p, const float4& C, const F8& P) {
  const float dx = C.x - (P.hi.x + P.lo.x), dy = C.y - (P.hi.y + P.lo.y),
              dz = C.z - (P.hi.z + P.lo.z);
  const float s = C.w + (P.hi.w + P.lo.w) + p.list_margin;
  return dx * dx + dy * dy + dz * dz > s * s * 1.0001f;
}
__device__ __forceinline__ bool clearly_apart(const Params&, const float4&, const D4&) {
  return false;
}

// Whether point C is farther than reach from the box around an element's vertices
// v[0 .. 3], in single precision.  No element is nearer than its box, and the box's
// distance is off by the coordinates' rounding alone; a single-precision closest
// point is off by more on thin triangles (0.4 mm on one of 16 mm x 10 um: the
// sphere would be kept inside the wall).
__device__ __forceinline__ bool outside_box(const float4& C, const float4* v, float reach) {
  const float4 a = v[0], b = v[1], c = v[2], d = v[3];  // (unused slots repeat vertex 0)
  const auto out = [](float x, float p, float q, float r, float s) {
    const float lo = fminf(fminf(p, q), fminf(r, s)), hi = fmaxf(fmaxf(p, q), fmaxf(r, s));
    return fmaxf(fmaxf(lo - x, x - hi), 0.f);
  };
  const float dx = out(C.x, a.x, b.x, c.x, d.x), dy = out(C.y, a.y, b.y, c.y, d.y),
              dz = out(C.z, a.z, b.z, c.z, d.z);
  return dx * dx + dy * dy + dz * dz > reach * reach;
}

constexpr int kSpawnWarps = 16;

template <typename Rec>
__global__ void __launch_bounds__(32 * kSpawnWarps)
k_spawn(Ctl* ctl, Params p, StateBufs sb, Lists L, BinBuf bb, MeshDev mesh) {
  __shared__ double kx[kSpawnMaxAttempts], ky[kSpawnMaxAttempts], kz[kSpawnMaxAttempts],
      kr[kSpawnMaxAttempts];
  __shared__ uint32_t free_s[kSpawnWarps];  // the warp's attempt overlaps nothing
  if (step_idle(ctl)) return;
  if (ctl->step % p.sp_every != 0) return;
  const uint32_t A = ctl->n_active;
  if (A >= (uint32_t)p.n) return;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t ph = ctl->phase & 1u;
  Rec* P = static_cast<Rec*>(buf_of(sb.P, ph));
  const uint32_t pose = pose_at(mesh, ctl->step);
  double co = 1.0, si = 0.0;
  if (mesh.nt > 0 && p.omega_norm > 0.0) {
    const double th = p.omega_norm * ((double)ctl->step * p.dt);
    co = cos(th);
    si = sin(th);
  }
  uint64_t draws = ctl->spawn_draws;
  double carry = ctl->spawn_carry;
  uint32_t kept = 0;
  for (int a = 0; a < p.sp_attempts && A + kept < (uint32_t)p.n;) {
    // attempts a .. a + nb - 1, warp w takes a + w: its draws follow those of
    // w failed attempts (three coordinates each, the radius carried over)
    const int nb = min(kSpawnWarps, p.sp_attempts - a);
    double r = carry;
    if (r < 0.0) r = lerp_box(p.sp_rmin, p.sp_rmax, spawn_uniform(p.sp_seed, draws++));
    double cx = 0.0, cy = 0.0, cz = 0.0;
    if (wid < nb) {
      const uint64_t d = draws + 3ull * (uint64_t)wid;
      cx = lerp_box(p.sp_lo[0], p.sp_hi[0], spawn_uniform(p.sp_seed, d));
      cy = lerp_box(p.sp_lo[1], p.sp_hi[1], spawn_uniform(p.sp_seed, d + 1));
      cz = lerp_box(p.sp_lo[2], p.sp_hi[2], spawn_uniform(p.sp_seed, d + 2));
      bool ov = false;
      const float4 C = make_float4((float)(cx - p.origin[0]), (float)(cy - p.origin[1]),
                                   (float)(cz - p.origin[2]), (float)r);
      const int3 cc = cell_coords(p, C.x, C.y, C.z);
      if (lane < 27) {
        const int x = cc.x + lane % 3 - 1, y = cc.y + (lane / 3) % 3 - 1,
                  z = cc.z + lane / 9 - 1;
        if (x >= 0 && x < p.nc[0] && y >= 0 && y < p.nc[1] && z >= 0 && z < p.nc[2]) {
          const uint32_t cell = cell_index(p, make_int3(x, y, z));
          const uint32_t e = bb.cell_start[cell + 1];
          for (uint32_t u = bb.cell_start[cell]; u < e && !ov; ++u) {
            const Rec Pu = P[u];
            if (!clearly_apart(p, C, Pu)) ov = overlaps(cx, cy, cz, r, sphere_of(p, Pu));
          }
        }
      }
      for (uint32_t k = lane; k < kept && !ov; k += 32)
        ov = overlaps(cx, cy, cz, r, Sphere{kx[k], ky[k], kz[k], kr[k]});
      if (mesh.nt > 0) {
        // the element lists are in the mesh's frame: the centre turned back by
        // the rotation of this step selects the list (the test itself is made
        // against the elements at their current pose)
        int3 cm = cc;
        if (p.omega_norm > 0.0) {
          const V3<double> ax = (1.0 / p.omega_norm) *
                                mk(p.mesh_omega[0], p.mesh_omega[1], p.mesh_omega[2]);
          const V3<double> cen = mk(p.mesh_center[0], p.mesh_center[1], p.mesh_center[2]);
          const V3<double> rr = mk(cx, cy, cz) - cen;
          const V3<double> qm =
              cen + (co * rr - si * cross(ax, rr) + (dot(ax, rr) * (1.0 - co)) * ax);
          cm = cell_coords(p, (float)(qm.x - p.origin[0]), (float)(qm.y - p.origin[1]),
                           (float)(qm.z - p.origin[2]));
        }
        const uint32_t cell = cell_index(p, cm);
        const uint32_t e = min(bb.tcell_start[cell + 1], bb.tcap);
        for (uint32_t i = bb.tcell_start[cell] + lane; i < e && !ov; i += 32) {
          const uint32_t k = bb.tcell_tri[i];
          const uint32_t kp = pose + k;
          const float4* vf = mesh.curf + 4 * (size_t)kp;
          if (outside_box(C, vf, C.w + (float)mesh.rad[k] + 4.f * p.mesh_prefilter)) continue;
          const int nvk = (int)vf[0].w;
          const V3<double> y = closest_point_element(
              mk(cx, cy, cz), xyz(mesh.cur[4 * kp]), xyz(mesh.cur[4 * kp + 1]),
              xyz(mesh.cur[4 * kp + 2]), xyz(mesh.cur[4 * kp + 3]), nvk);
          ov = overlaps(cx, cy, cz, r, Sphere{y.x, y.y, y.z, mesh.rad[k]});
        }
      }
      ov = __any_sync(full, ov);
      if (lane == 0) free_s[wid] = ov ? 0u : 1u;
    }
    __syncthreads();
    const unsigned ok = __ballot_sync(full, lane < nb && free_s[lane < nb ? lane : 0] != 0u);
    const int first = __ffs((int)ok) - 1;  // -1: all failed
    if (first == wid && lane == 0) {
      Rec* V = static_cast<Rec*>(buf_of(sb.V, ph));
      put_new(p, P, V, static_cast<Rec*>(buf_of(sb.W, ph)), static_cast<Rec*>(buf_of(sb.Q, ph)),
              A + kept, cx, cy, cz, r);
      D4* inv = list_of(L, ctl->lphase & 1u).inv;
      if (inv) inv[A + kept] = inverses(p, P[A + kept], V[A + kept]);
      kx[kept] = cx;
      ky[kept] = cy;
      kz[kept] = cz;
      kr[kept] = r;
    }
    __syncthreads();
    const int taken = first >= 0 ? first + 1 : nb;
    a += taken;
    draws += 3ull * (uint64_t)taken;
    carry = first >= 0 ? -1.0 : r;
    kept += first >= 0 ? 1u : 0u;
  }
  if (threadIdx.x == 0) {
    ctl->n_active = A + kept;
    ctl->spawn_carry = carry;
    ctl->spawn_draws = draws;
    if (kept) ctl->force_rebuild = 1u;
  }
}

}  // namespace

void launch_spawn(cudaStream_t st, Ctl* ctl, const Params& p, StateBufs sb, Lists L, BinBuf bb,
                  MeshDev mesh) {
  if (p.sp_attempts <= 0) return;
  if (p.mixed)
    k_spawn<F8><<<1, 32 * kSpawnWarps, 0, st>>>(ctl, p, sb, L, bb, mesh);
  else
    k_spawn<D4><<<1, 32 * kSpawnWarps, 0, st>>>(ctl, p, sb, L, bb, mesh);
}

}  // namespace dem
