// Static ray-patch intersection (Sec. 5, Eq. ray, Eq. ineqray): nearest hit of each ray with the
// bicubic Hermite shell by subdivision of the patches' Bezier forms.
//
//   k_ray_nets   one thread per patch: Bezier control net (Hermite data b0 = a, b1 = a + a'/3,
//                b2 = b - b'/3, b3 = b per direction, tensor product) and its box.
//   k_ray_groups the box of every kGroup consecutive patches, to skip groups a ray misses.
//   k_trace_rays one ray per thread, FP64: all patch boxes are tested in patch order (staged
//                through shared memory, one chunk at a time for the whole CTA), hits go into a
//                binary min-heap in local memory keyed by the box's entry time tau_min; the top
//                candidate is refined (box at most kEpsTau on every side: an intersection at the
//                midpoint of its tau interval), or split into four sub-patches, at the parameter
//                midpoint (Fig. submid) or, in the Newton variant, around a Newton root of
//                x(u, v) = o + tau d that is abandoned together with its neighbourhood
//                (Fig. subany). The search ends when the heap's top cannot beat the best tau.
//                The children's boxes (4 children x 3 coordinates per split, most of a split's
//                FP64 work) are pooled over the warp: lanes whose rays are done or need no split
//                take jobs of the lanes that do, so a long search left alone in its warp runs
//                its 12 box jobs side by side instead of one after another.
//                A ray whose local heap fills moves it into one of kRedoThreads larger heaps
//                in global memory and continues.
//                Without statistics, children (and popped patch roots) that an FP32 test proves to
//                lead to no hit are left out before their FP64 boxes (bezier.cuh), and group and patch
//                boxes are tested in FP32 first. FP64 issue bounds this kernel (one warp instruction per
//                64 cycles and sub-partition), so an FP32 test costs a few percent of the box it saves,
//                and its tilted lines prune where axis-aligned boxes overlap the ray at every level
//                (near-tangent rays). Rays whose result could depend on the order of equal keys are
//                searched again in full (bezier.cuh, Ties; no more than two of 786,432 camera rays; watching
//                for them costs 3%: drape, Newton split 29.6 -> 30.5 ms). Newton iterations run one at a time beside the other lanes' splits,
//                few of them on four lanes each, and every box job on four lanes. Measured, 1024 x 768 rays:
//                drape, Newton split 240 -> 12.8 ms (another drape, with more tangent rays, 373 -> 35 ms),
//                midpoint split 217 -> 142 ms; 512 x 384: cylinder, Newton split 61 -> 3.3 ms, midpoint
//                58 -> 51 ms, plane 1.5 -> 0.38 ms. What is left of the midpoint split are the levels
//                below the test's margin, boxed as before.
//   k_trace_rays_redo  the rays that found no free global heap, traced again from the start
//                with one (the search is deterministic, so the result is the one an unbounded
//                heap gives).
//
// Sub-patches are cut from the patch's net by blossoming (each restricted curve's points are
// f(a,a,a), f(a,a,b), f(a,b,b), f(b,b,b), De Casteljau with one parameter per level) and only
// their box is kept: per coordinate the 4 theta1-curves are restricted, then the 4 theta2-curves,
// folded straight into the slab test. This file is compiled without mul-add contraction: each
// product and sum is rounded separately, in the order written, so every decision of the search
// (slab intervals, heap order, refinement, Newton convergence) is that of the same sequence of
// IEEE FP64 operations in any plain sequential program.
#include <cmath>
#include <type_traits>

#include "bezier.cuh"
#include "common.cuh"

namespace bhem {
namespace {

using namespace bz;

constexpr double kEpsTau = 1e-9;     // refinement size (positions' units; unit directions)
constexpr int kNetBlock = 128;
constexpr int kRayBlock = 128;
constexpr int kRootChunk = 32;       // group boxes staged in shared memory per pass
constexpr int kGroup = 32;           // consecutive patches per group box

// FP32 net of a patch for the culling test, relative to its centre
struct CullNet {
  double c[3];
  float radius;
  float box[6];   // the patch's box, rounded outwards: min xyz, max xyz
  float pad;
  float n[48];
};

// Min and max of coordinate c of the sub-patch [u0, u1] x [v0, v1] of the net P ([c][i][j]).
__device__ __forceinline__ void sub_range(const double* __restrict__ P, int c, double u0, double u1, double v0,
                                          double v1, double& mn, double& mx) {
  const double* Pc = P + 16 * c;
  double T[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const double in[4] = {__ldg(Pc + j), __ldg(Pc + 4 + j), __ldg(Pc + 8 + j), __ldg(Pc + 12 + j)};
    double o[4];
    curve_restrict(in, u0, u1, o);
#pragma unroll
    for (int i = 0; i < 4; ++i) T[i][j] = o[i];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    double o[4];
    curve_restrict(T[i], v0, v1, o);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double s = o[j];
      if (i == 0 && j == 0) {
        mn = s;
        mx = s;
      }
      if (s < mn) mn = s;
      if (s > mx) mx = s;
    }
  }
}

// One axis of the slab test (Eq. ineqray): narrows [lo, hi]; false when the ray misses.
__device__ __forceinline__ bool slab(double mn, double mx, double o, double d, double inv, double& lo,
                                     double& hi) {
  if (d == 0.0) return !(o < mn || o > mx);
  double a = (mn - o) * inv, b = (mx - o) * inv;
  if (a > b) {
    const double t = a;
    a = b;
    b = t;
  }
  if (a > lo) lo = a;
  if (b < hi) hi = b;
  return true;
}

// Box of each group of kGroup consecutive patches (min xyz, max xyz of its patches' boxes). A ray
// that misses a group's box misses every member's: FP64 subtraction and multiplication by the
// same 1/d are monotone, so the group's slab interval contains each member's.
__global__ void k_ray_groups(int np, const double* __restrict__ boxes, double* __restrict__ gboxes) {
  const int gi = blockIdx.x * blockDim.x + threadIdx.x;
  const int p0 = gi * kGroup;
  if (p0 >= np) return;
  const int p1 = min(np, p0 + kGroup);
  double mn[3], mx[3];
  for (int c = 0; c < 3; ++c) {
    mn[c] = boxes[(size_t)p0 * 8 + c];
    mx[c] = boxes[(size_t)p0 * 8 + 3 + c];
  }
  for (int p = p0 + 1; p < p1; ++p)
    for (int c = 0; c < 3; ++c) {
      const double a = boxes[(size_t)p * 8 + c], b = boxes[(size_t)p * 8 + 3 + c];
      if (a < mn[c]) mn[c] = a;
      if (b > mx[c]) mx[c] = b;
    }
  double* G = gboxes + (size_t)gi * 8;
  for (int c = 0; c < 3; ++c) {
    G[c] = mn[c];
    G[3 + c] = mx[c];
  }
  G[6] = 0.0;
  G[7] = 0.0;
}

__global__ void __launch_bounds__(kNetBlock) k_ray_nets(int np, const int4* __restrict__ pnodes,
                                                        const double* __restrict__ q, double dxi1, double dxi2,
                                                        double* __restrict__ nets, double* __restrict__ boxes,
                                                        CullNet* __restrict__ culls) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  const int4 n4 = pnodes[p];
  const int nd[4] = {n4.x, n4.y, n4.z, n4.w};
  double* P = nets + (size_t)p * 48;
  patch_net(q, nd, dxi1, dxi2, P);
  if (culls) center_net32(P, culls[p].n, culls[p].c, culls[p].radius);   // its box below
  // the root box is the box of the net cut to [0, 1]^2, as for every other candidate
  double e = 0.0;
  double* B = boxes + (size_t)p * 8;
  for (int c = 0; c < 3; ++c) {
    double mn, mx;
    sub_range(P, c, 0.0, 1.0, 0.0, 1.0, mn, mx);
    B[c] = mn;
    B[3 + c] = mx;
    if (culls) {
      culls[p].box[c] = __double2float_rd(mn);
      culls[p].box[3 + c] = __double2float_ru(mx);
    }
    if (mx - mn > e) e = mx - mn;
  }
  B[6] = e;
  B[7] = 0.0;
}

// Newton's method on F(u, v, tau) = x(u, v) - o - tau d, Jacobian [x_u | x_v | -d] by Cramer's
// rule, at most kNewtonIters iterations; it gives up when an iterate leaves the window win (the
// candidate's rectangle widened by its extent on each side). The lanes of a warp take one iteration
// at a time, beside the splits of the lanes that need none: the number of iterations varies from one
// to twelve, and a lane that ran them all at once would hold the others up.
// One iteration from (u, v, tau) of every lane with `want`; state 1: converged (at the point given),
// 2: it gives up, 0: the next point. Few lanes are served by four lanes each (a coordinate of the
// surface point and a component of the step per lane: about 200 FP64 operations for eight iterations,
// against 370 for one to 32), more by themselves. All 32 lanes of the warp call it.
constexpr int kSharedNewton = 8;

__device__ void newton_step(bool want, const double* __restrict__ nets, int patch, const double o[3], const double d[3],
                            double on, const double win[4], double& u, double& v, double& tau, int& state) {
  const unsigned mask = __ballot_sync(0xffffffffu, want);
  const int count = __popc(mask), lane = threadIdx.x & 31;
  if (count == 0) return;
  double delta[3] = {0.0, 0.0, 0.0};
  if (count <= kSharedNewton) {
    const int own = nth_lane(mask, lane >> 2), c = min(lane & 3, 2), g = lane & 28;
    const int p = __shfl_sync(0xffffffffu, patch, own);
    const double uu = __shfl_sync(0xffffffffu, u, own), vv = __shfl_sync(0xffffffffu, v, own);
    const double tt = __shfl_sync(0xffffffffu, tau, own), oon = __shfl_sync(0xffffffffu, on, own);
    const double o0 = __shfl_sync(0xffffffffu, o[0], own), o1 = __shfl_sync(0xffffffffu, o[1], own),
                 o2 = __shfl_sync(0xffffffffu, o[2], own);
    const double d0 = __shfl_sync(0xffffffffu, d[0], own), d1 = __shfl_sync(0xffffffffu, d[1], own),
                 d2 = __shfl_sync(0xffffffffu, d[2], own);
    const double oc = c == 0 ? o0 : c == 1 ? o1 : o2, dc = c == 0 ? d0 : c == 1 ? d1 : d2;
    double Bu[4], dBu[4], Bv[4], dBv[4], x, xu, xv;
    bernstein(uu, Bu, dBu);
    bernstein(vv, Bv, dBv);
    bezier_eval_coord(nets + (size_t)p * 48 + 16 * c, Bu, dBu, Bv, dBv, x, xu, xv);
    const double f = (x - oc) - tt * dc;
    double F[3], J[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      F[r] = __shfl_sync(0xffffffffu, f, g + r);
      J[r][0] = __shfl_sync(0xffffffffu, xu, g + r);
      J[r][1] = __shfl_sync(0xffffffffu, xv, g + r);
      J[r][2] = -__shfl_sync(0xffffffffu, dc, g + r);
    }
    const double fn = sqrt((F[0] * F[0] + F[1] * F[1]) + F[2] * F[2]);
    bool regular;
    const double step = cramer_component(J, F, c, &regular);
    const int st = fn <= 1e-12 * ((1.0 + oon) + fabs(tt)) ? 1 : !regular ? 2 : 0;
    const int src = 4 * __popc(mask & ((1u << lane) - 1u));   // the lanes that served this one
    const int got = __shfl_sync(0xffffffffu, st, src & 31);
#pragma unroll
    for (int k = 0; k < 3; ++k) delta[k] = __shfl_sync(0xffffffffu, step, (src + k) & 31);
    if (!want) return;
    state = got;
  } else {
    if (!want) return;
    const double* P = nets + (size_t)patch * 48;
    double x[3], xu[3], xv[3], F[3];
    bezier_eval(P, u, v, x, xu, xv);
#pragma unroll
    for (int c = 0; c < 3; ++c) F[c] = (x[c] - o[c]) - tau * d[c];
    const double fn = sqrt((F[0] * F[0] + F[1] * F[1]) + F[2] * F[2]);
    const double J[3][3] = {{xu[0], xv[0], -d[0]}, {xu[1], xv[1], -d[1]}, {xu[2], xv[2], -d[2]}};
    bool regular = true;
    state = fn <= 1e-12 * ((1.0 + on) + fabs(tau)) ? 1 : 0;
    if (state == 0)
#pragma unroll
      for (int k = 0; k < 3; ++k) delta[k] = cramer_component(J, F, k, &regular);
    if (!regular) state = 2;
  }
  if (state) return;
  u += delta[0];
  v += delta[1];
  tau += delta[2];
  if (!isfinite(u) || !isfinite(v) || !isfinite(tau) || u < win[0] || u > win[1] || v < win[2] || v > win[3])
    state = 2;   // left the window
}

struct Ray {
  double o[3], d[3], inv[3];
  // culling: |d| (0: nothing is culled), d / |d| and two unit directions about perpendicular to it and to each
  // other; o and 1 / d in FP32 (infinite for a zero component, NaN for one too small or too large for
  // FP32: that axis then never rules a box out)
  float len, dir[3], e1[3], e2[3], o32[3], inv32[3];
};

__device__ __forceinline__ void load_ray(const double* __restrict__ origins, const double* __restrict__ dirs,
                                         long long k, Ray& r) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    r.o[c] = origins[3 * k + c];
    r.d[c] = dirs[3 * k + c];
    r.inv[c] = r.d[c] != 0.0 ? 1.0 / r.d[c] : 0.0;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    r.o32[c] = (float)r.o[c];
    r.inv32[c] = r.d[c] == 0.0 ? INFINITY : !(fabs(r.d[c]) >= 1e-30 && fabs(r.d[c]) <= 1e30) ? NAN : (float)r.inv[c];
  }
  // directions are unit vectors by contract, but the search takes any: the culling works in distances along
  // the ray, |d| times the differences of tau
  const double len = sqrt((r.d[0] * r.d[0] + r.d[1] * r.d[1]) + r.d[2] * r.d[2]);
  r.len = len >= 1e-15 && len <= 1e15 ? (float)len : 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) r.dir[c] = (float)(r.d[c] / len);
  // e1 = dir x (the axis it is least along), normalised; e2 = dir x e1
  const float dx = r.dir[0], dy = r.dir[1], dz = r.dir[2];
  const float ax = fabsf(dx), ay = fabsf(dy), az = fabsf(dz);
  float e[3] = {0.f, dz, -dy};
  if (ay < ax && ay <= az) { e[0] = -dz; e[1] = 0.f; e[2] = dx; }
  else if (az < ax && az < ay) { e[0] = dy; e[1] = -dx; e[2] = 0.f; }
  const float s = rsqrtf(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]);
  for (int c = 0; c < 3; ++c) r.e1[c] = e[c] * s;
  r.e2[0] = dy * r.e1[2] - dz * r.e1[1];
  r.e2[1] = dz * r.e1[0] - dx * r.e1[2];
  r.e2[2] = dx * r.e1[1] - dy * r.e1[0];
}

// Root candidate: the whole patch p with box B = (min xyz, max xyz, largest side).
__device__ __forceinline__ void root_push(Heap& h, const double* B, int p, const Ray& r) {
  double lo = 0.0, hi = INFINITY;
  bool in = true;
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (in) in = slab(B[c], B[3 + c], r.o[c], r.d[c], r.inv[c], lo, hi);
  if (in && !(lo > hi)) h.push(Cand{lo, hi, B[6], 0.0, 1.0, 0.0, 1.0, p});
}

// Whether the ray surely misses an outward-rounded FP32 box: the slab test with the box widened by the
// rounding of o and of the differences (2^-24 of their terms, against 1e-6) and the interval's ends
// taken apart by 1e-6 (their relative error is under 2^-21). A NaN (0 times infinity, or an axis not
// used) leaves an axis out, since fminf and fmaxf drop it.
__device__ __forceinline__ bool surely_missed(const float* B, const Ray& r) {
  float lo = 0.f, hi = 1e30f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float mn = B[c], mx = B[3 + c], w = 1e-6f * (fabsf(r.o32[c]) + fmaxf(fabsf(mn), fabsf(mx)));
    const float a = ((mn - w) - r.o32[c]) * r.inv32[c], b = ((mx + w) - r.o32[c]) * r.inv32[c];
    if (a == a && b == b) {
      lo = fmaxf(lo, fminf(a, b));
      hi = fminf(hi, fmaxf(a, b));
    }
  }
  lo = fminf(lo, 1e30f);
  hi = fmaxf(hi, -1e30f);
  return lo - 1e-6f * lo > hi + 1e-6f * fabsf(hi);
}

// Per-lane state of one ray's search.
struct Search {
  double best = INFINITY, bu = 0.0, bv = 0.0, on = 0.0;
  int bp = -1, nexp = 0, flags = 0, newton_iters = 0;
  bool live = false;
  bool cull = true;   // (kCull) false when the ray is searched again because of ties
  Ties ties;
};

// Shared-memory exchange of one warp: the children each lane produced in the current split and
// the coordinate ranges computed for them by whichever lanes took those jobs.
struct PlainSmem {
  double rect[32][4][4];        // child rectangles u0, u1, v0, v1 in push order
  double range[32][12][2];      // (child * 3 + coordinate): min, max
  int patch[32];
  unsigned short jobs[32 * 12]; // lane * 12 + child * 3 + coordinate
};
struct CullSmem : PlainSmem {
  float path[32][14];           // path point from the patch's centre, e1, e2, dir, distance to the best hit, margin
  unsigned char cull[32][4];    // child proven not to lead to a hit
};
template <bool kCull> using WarpSmem = std::conditional_t<kCull, CullSmem, PlainSmem>;

__device__ __forceinline__ float cull_margin(const CullNet* __restrict__ N, const float* path) {
  return fmaxf(path[13], kCullRel * (N->radius + fabsf(path[0]) + fabsf(path[1]) + fabsf(path[2])));
}

// Culling test of one child of a ray's candidate: the control points, seen along the ray (projected
// on e1 and e2, the path point at the origin), lie on one side of a line through the origin, or all
// of them lie beyond the best hit along d. Lines tried: along e1, along e2, along the net's two
// chords (a smooth sub-patch is nearly a parallelogram with those sides).
__device__ __forceinline__ bool child_is_culled(const CullNet* __restrict__ N, const float* path, const double* R) {
  const float r[4] = {(float)R[0], (float)R[1], (float)R[2], (float)R[3]};
  float a[16], b[16], t[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float x = __ldg(N->n + k) - path[0], y = __ldg(N->n + 16 + k) - path[1], z = __ldg(N->n + 32 + k) - path[2];
    a[k] = __fmaf_rn(x, path[3], __fmaf_rn(y, path[4], z * path[5]));
    b[k] = __fmaf_rn(x, path[6], __fmaf_rn(y, path[7], z * path[8]));
    t[k] = __fmaf_rn(x, path[9], __fmaf_rn(y, path[10], z * path[11]));
  }
  const float eps = cull_margin(N, path);
  restrict_net32(a, r);
  if (one_side32(a, eps)) return true;
  restrict_net32(b, r);
  if (one_side32(b, eps)) return true;
  // the chords of the u and of the v direction; a line along (p, q) has the normal (-q, p)
  const float up = (a[12] - a[0]) + (a[15] - a[3]), uq = (b[12] - b[0]) + (b[15] - b[3]);
  if (one_side32(a, b, -uq, up, eps)) return true;
  const float vp = (a[3] - a[0]) + (a[15] - a[12]), vq = (b[3] - b[0]) + (b[15] - b[12]);
  if (one_side32(a, b, -vq, vp, eps)) return true;
  restrict_net32(t, r);
  float mn = t[0];
#pragma unroll
  for (int k = 1; k < 16; ++k) mn = fminf(mn, t[k]);
  return mn > path[12] + eps;   // path[12]: distance_to_best; +infinity without a hit
}

__device__ __forceinline__ void put_rect(PlainSmem& sm, int lane, int& nch, double u0, double u1, double v0,
                                         double v1) {
  if (!(u1 > u0) || !(v1 > v0)) return;   // degenerate pieces of a pinwheel split
  double* R = sm.rect[lane][nch++];
  R[0] = u0;
  R[1] = u1;
  R[2] = v0;
  R[3] = v1;
}

// From the path point at t0 to the best hit, along the ray, rounded up.
__device__ __forceinline__ float distance_to_best(const Ray& r, double best, double t0) {
  const float beyond = (float)(best - t0) * r.len;
  return beyond + 1e-6f * fabsf(beyond);
}

// Prepares the culling of candidate c's children: the ray from c's entry point on, relative to the
// patch's centre. True when c is a whole patch that is itself culled (it is not split then).
template <bool kCull>
__device__ __forceinline__ bool starts_culled(WarpSmem<kCull>& sm, int lane, const Cand& c, const Ray& r,
                                              const CullNet* __restrict__ culls, double best, double on, bool cull,
                                              bool& cullable) {
  if constexpr (kCull) {
    float* path = sm.path[lane];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      path[k] = (float)((r.o[k] + c.t0 * r.d[k]) - culls[c.patch].c[k]);
      path[3 + k] = r.e1[k];
      path[6 + k] = r.e2[k];
      path[9 + k] = r.dir[k];
    }
    const float far = (float)on + fabsf((float)c.t0) * fmaxf(1.f, r.len);
    path[13] = fmaxf(kCullAbs, 4e-12f * (1.f + far));   // 4 x Newton's tolerance
    // nothing is culled among children of the margin's size: their tests are left out. Far from the
    // origin (FP64 distances above 1e4 are 1e-12 apart) equal keys near the hit are common, and such rays are
    // searched again in full, so nothing is culled there either.
    cullable = cull && r.len > 0.f && (float)c.ext > 8.f * cull_margin(culls + c.patch, path) && far < kCullFar;
    if (!cullable) return false;
    path[12] = distance_to_best(r, best, c.t0);
    if (c.u1 - c.u0 == 1.0 && c.v1 - c.v0 == 1.0) {
      const double R[4] = {0.0, 1.0, 0.0, 1.0};
      return child_is_culled(culls + c.patch, path, R);
    }
  }
  return false;
}

// Lists the warp's jobs, `per` for each child in a lane's mask `keep` (lane * 12 + child * per + 0 ..
// per - 1), in lane order; returns their number. All 32 lanes call it; ends with a warp barrier.
__device__ __forceinline__ int list_jobs(PlainSmem& sm, int lane, unsigned keep, int per) {
  const int nj = per * __popc(keep);
  int pre = nj;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, pre, off);
    if (lane >= off) pre += y;
  }
  const int total = __shfl_sync(0xffffffffu, pre, 31);
  pre -= nj;
  for (unsigned m = keep; m; m &= m - 1) {
    const int ch = __ffs(m) - 1;
    for (int k = 0; k < per; ++k) sm.jobs[pre++] = (unsigned short)(lane * 12 + ch * per + k);
  }
  __syncwarp();
  return total;
}

// The search over the candidates already in each lane's heap, all 32 lanes of the warp together
// (lanes without a ray pass live = false). Every iteration each live lane takes its top
// candidate and, when it splits it, lists its children; the 3 coordinate ranges of every child
// of every lane are then computed as one pool of jobs spread over the warp's lanes, and each
// lane finishes its own children (slab test, push) in order. A ray stops early once its heap
// overflows.
// kCull: children (and patch roots) that provably lead to no hit are left out; without it every child
// is boxed, and the search statistics are those of the plain algorithm.
template <bool kCull, bool kNewton>
__device__ void search(Heap& h, const Ray& r, const double* __restrict__ nets, const CullNet* __restrict__ culls,
                       Search& S, WarpSmem<kCull>& sm, int lane) {
  S.on = sqrt((r.o[0] * r.o[0] + r.o[1] * r.o[1]) + r.o[2] * r.o[2]);
  Cand c{};                // the candidate being split
  int newton = -1;         // its Newton iterations so far; -1: none in progress
  double u = 0.0, v = 0.0, t = 0.0;
  bool cullable = false;
  while (__any_sync(0xffffffffu, S.live)) {
    int nch = 0;
    bool split = false, root = false;   // split c now; around the root (u, v, t)
    if (S.live && newton < 0) {
      if (h.n == 0 || h.overflow) {
        S.live = false;
      } else {
        c = h.pop();
        if constexpr (kCull) S.ties.popped(c, h.n > 0, h.a[0].t0, S.best, kEpsTau);
        if ((kCull && S.cull && S.ties.again) || c.t0 >= S.best - kEpsTau) {   // nothing left can be closer
          S.live = false;
        } else if (c.ext <= kEpsTau || (c.u1 - c.u0 < 1e-13 && c.v1 - c.v0 < 1e-13)) {   // refined
          const double tm = 0.5 * (c.t0 + c.t1);
          if (tm < S.best - kEpsTau) {
            S.best = tm;
            if constexpr (kCull) S.ties.hit(S.best, kEpsTau);
            S.bp = c.patch;
            S.bu = 0.5 * (c.u0 + c.u1);
            S.bv = 0.5 * (c.v0 + c.v1);
          }
        } else if (S.nexp == kMaxExpansions) {
          S.flags |= SHELL_RAY_LIMIT;
          S.live = false;
        } else if (!starts_culled<kCull>(sm, lane, c, r, culls, S.best, S.on, S.cull, cullable)) {
          ++S.nexp;
          u = 0.5 * (c.u0 + c.u1);
          v = 0.5 * (c.v0 + c.v1);
          if constexpr (kNewton) {
            double x[3], xu[3], xv[3];
            bezier_eval(nets + (size_t)c.patch * 48, u, v, x, xu, xv);
            t = ((x[0] - r.o[0]) * r.d[0] + (x[1] - r.o[1]) * r.d[1]) + (x[2] - r.o[2]) * r.d[2];
            newton = 0;
          } else {
            split = true;
          }
        }
      }
    }
    if constexpr (kNewton) {
      const bool want = newton >= 0;
      const double wu = c.u1 - c.u0, wv = c.v1 - c.v0;
      const double win[4] = {c.u0 - wu, c.u1 + wu, c.v0 - wv, c.v1 + wv};
      int state = 0;
      newton_step(want, nets, c.patch, r.o, r.d, S.on, win, u, v, t, state);
      if (want) {
        ++newton;
        ++S.newton_iters;
        if (state || newton == kNewtonIters) {
          newton = -1;
          split = true;
          root = state == 1 && u >= c.u0 && u <= c.u1 && v >= c.v0 && v <= c.v1 && t >= 0.0;
        }
      }
    }
    if (split) {
      if (root) {
        if constexpr (kCull) S.ties.root(t, S.best);
        if (t < S.best) {
          S.best = t;
          if constexpr (kCull) S.ties.hit(S.best, kEpsTau);
          S.bp = c.patch;
          S.bu = u;
          S.bv = v;
        }
        // Fig. subany: drop [a1, a2] x [b1, b2] around the root, four rectangles remain
        const double hu = kNbhd * (c.u1 - c.u0), hv = kNbhd * (c.v1 - c.v0);
        const double a1 = fmax(c.u0, u - hu), a2 = fmin(c.u1, u + hu);
        const double b1 = fmax(c.v0, v - hv), b2 = fmin(c.v1, v + hv);
        put_rect(sm, lane, nch, c.u0, a1, b1, c.v1);
        put_rect(sm, lane, nch, a1, c.u1, b2, c.v1);
        put_rect(sm, lane, nch, c.u0, a2, c.v0, b1);
        put_rect(sm, lane, nch, a2, c.u1, c.v0, b2);
      } else {   // Fig. submid: four quarters at the parameter midpoint
        const double um = 0.5 * (c.u0 + c.u1), vm = 0.5 * (c.v0 + c.v1);
        put_rect(sm, lane, nch, c.u0, um, vm, c.v1);
        put_rect(sm, lane, nch, um, c.u1, vm, c.v1);
        put_rect(sm, lane, nch, c.u0, um, c.v0, vm);
        put_rect(sm, lane, nch, um, c.u1, c.v0, vm);
      }
      sm.patch[lane] = c.patch;
      h.boxes += nch;
      if constexpr (kCull) {   // a root found above may have brought the best hit nearer
        sm.path[lane][12] = distance_to_best(r, S.best, c.t0);
      }
    }
    unsigned keep = (1u << nch) - 1u;   // children to box
    if constexpr (kCull) {
      const int total = list_jobs(sm, lane, cullable ? keep : 0u, 1);
      for (int j = lane; j < total; j += 32) {
        const int code = sm.jobs[j], owner = code / 12, ch = code - 12 * owner;
        sm.cull[owner][ch] = child_is_culled(culls + sm.patch[owner], sm.path[owner], sm.rect[owner][ch]);
      }
      __syncwarp();
      for (int ch = 0; ch < nch; ++ch)
        if (cullable && sm.cull[lane][ch]) keep &= ~(1u << ch);
      __syncwarp();
    }
    // the warp's pool of (lane, child, coordinate) range jobs
    const int total = list_jobs(sm, lane, keep, 3);
    // four lanes per job: eight jobs a round, 110 FP64 operations long (one lane per job: 450)
    for (int base = 0; base < total; base += 8) {
      const int j = base + (lane >> 2), code = sm.jobs[min(j, total - 1)], owner = code / 12, k = code - 12 * owner;
      double o[4];
      cut_row(nets + (size_t)sm.patch[owner] * 48 + 16 * (k % 3), lane & 3, sm.rect[owner][k / 3], o);
      double mn = o[0], mx = o[0];
#pragma unroll
      for (int i = 1; i < 4; ++i) {
        if (o[i] < mn) mn = o[i];
        if (o[i] > mx) mx = o[i];
      }
#pragma unroll
      for (int off = 1; off < 4; off <<= 1) {
        const double a = __shfl_xor_sync(0xffffffffu, mn, off), b = __shfl_xor_sync(0xffffffffu, mx, off);
        if (a < mn) mn = a;
        if (b > mx) mx = b;
      }
      if ((lane & 3) == 0 && j < total) {
        sm.range[owner][k][0] = mn;
        sm.range[owner][k][1] = mx;
      }
    }
    __syncwarp();
    for (int ch = 0; ch < nch; ++ch) {
      if (!(keep >> ch & 1)) continue;
      double lo = 0.0, hi = INFINITY, e = 0.0;
      bool in = true;
      for (int cc = 0; cc < 3 && in; ++cc) {
        const double mn = sm.range[lane][3 * ch + cc][0], mx = sm.range[lane][3 * ch + cc][1];
        if (mx - mn > e) e = mx - mn;
        in = slab(mn, mx, r.o[cc], r.d[cc], r.inv[cc], lo, hi);
      }
      if (in && !(lo > hi) && !(lo >= S.best)) {
        const double* R = sm.rect[lane][ch];
        h.push(Cand{lo, hi, e, R[0], R[1], R[2], R[3], sm.patch[lane]});
      }
    }
    __syncwarp();
  }
  if (h.overflow) {
    S.flags |= SHELL_RAY_OVERFLOW;   // void: reported as a miss
  } else if (S.bp >= 0) {
    S.flags |= SHELL_RAY_HIT;
  }
}

// Patch roots in patch order, by one lane; a box that the FP32 test rules out would not be pushed.
template <bool kCull>
__device__ void push_roots(Heap& h, const Ray& r, const double* __restrict__ boxes, const CullNet* __restrict__ culls,
                           int np) {
  for (int p = 0; p < np; ++p) {
    if constexpr (kCull)
      if (surely_missed(culls[p].box, r)) continue;
    root_push(h, boxes + 8 * (size_t)p, p, r);
  }
  h.boxes = np;
}

// The search, and again without culling for the rays whose ties can matter. All 32 lanes call it.
template <bool kCull, bool kNewton>
__device__ void search_all(Heap& h, const Ray& r, const double* __restrict__ nets, const double* __restrict__ boxes,
                           const CullNet* __restrict__ culls, int np, Search& S, WarpSmem<kCull>& sm, int lane) {
  for (;;) {
    search<kCull, kNewton>(h, r, nets, culls, S, sm, lane);
    if constexpr (!kCull) return;
    const bool again = S.cull && S.ties.again && !h.overflow;
    if (!__any_sync(0xffffffffu, again)) return;
    if (again) {   // the other lanes' searches have ended
      S = Search();
      S.cull = false;
      S.live = true;
      h.n = 0;
      push_roots<kCull>(h, r, boxes, culls, np);
    }
  }
}

struct RayOut {
  double* tau;
  int* patch;
  double* uv;
  int* flags;
  int* stats;
};

__device__ __forceinline__ void write_hit(const RayOut& out, long long k, const Search& S, const Heap& h) {
  const bool hit = (S.flags & SHELL_RAY_HIT) != 0;
  out.tau[k] = hit ? S.best : INFINITY;
  out.patch[k] = hit ? S.bp : -1;
  out.uv[2 * k] = hit ? S.bu : 0.0;
  out.uv[2 * k + 1] = hit ? S.bv : 0.0;
  out.flags[k] = S.flags;
  if (out.stats) {
    out.stats[4 * k] = S.nexp;
    out.stats[4 * k + 1] = h.peak;
    out.stats[4 * k + 2] = h.boxes;
    out.stats[4 * k + 3] = S.newton_iters;
  }
}

// First pass: one ray per thread, a kHeapCap-entry heap in local memory, the search shared by the
// warp. A ray whose heap overflows stops and is appended to redo_list for the second pass (or,
// when the list is full, reported with SHELL_RAY_OVERFLOW).
template <bool kCull, bool kNewton>
__global__ void __launch_bounds__(kRayBlock, 4) k_trace_rays(long long n, const double* __restrict__ origins,
                                                          const double* __restrict__ dirs, int np,
                                                          const double* __restrict__ nets,
                                                          const double* __restrict__ boxes,
                                                          const double* __restrict__ gboxes,
                                                          const CullNet* __restrict__ culls,
                                                          RayOut out, int* __restrict__ redo_count,
                                                          int* __restrict__ redo_list, Cand* __restrict__ heaps) {
  using Box = std::conditional_t<kCull, float, double>;
  __shared__ Box sbox[kRootChunk * 8];
  __shared__ WarpSmem<kCull> wsm[kRayBlock / 32];
  const int lane = threadIdx.x & 31;
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool active = k < n;
  Ray r;
  Cand storage[kHeapCap];
  Heap h(storage, kHeapCap);
  h.spill = heaps;
  h.spill_count = redo_count + 1;
  if (active) load_ray(origins, dirs, k, r);
  // every patch's box in patch order, skipping the groups whose box the ray misses (their members
  // would all be missed); the whole CTA stages one chunk of group boxes at a time
  const int ngroups = (np + kGroup - 1) / kGroup;
  for (int base = 0; base < ngroups; base += kRootChunk) {
    const int m = min(kRootChunk, ngroups - base);
    __syncthreads();
    for (int i = threadIdx.x; i < m * 8; i += blockDim.x) {
      const double v = gboxes[(size_t)base * 8 + i];
      if constexpr (kCull) sbox[i] = i % 8 < 3 ? __double2float_rd(v) : __double2float_ru(v);
      else sbox[i] = v;
    }
    __syncthreads();
    if (!active) continue;
    for (int j = 0; j < m; ++j) {
      const Box* G = sbox + 8 * j;
      const int p0 = (base + j) * kGroup, p1 = min(np, p0 + kGroup);
      if constexpr (kCull) {
        if (surely_missed(G, r)) continue;
        for (int p = p0; p < p1; ++p)
          if (!surely_missed(culls[p].box, r)) root_push(h, boxes + 8 * (size_t)p, p, r);
      } else {
        double lo = 0.0, hi = INFINITY;
        bool in = true;
#pragma unroll
        for (int c = 0; c < 3; ++c)
          if (in) in = slab(G[c], G[3 + c], r.o[c], r.d[c], r.inv[c], lo, hi);
        if (!in || lo > hi) continue;
        for (int p = p0; p < p1; ++p) root_push(h, boxes + 8 * (size_t)p, p, r);
      }
    }
  }
  h.boxes = np;
  Search S;
  S.live = active;
  search_all<kCull, kNewton>(h, r, nets, boxes, culls, np, S, wsm[threadIdx.x >> 5], lane);
  if (!active) return;
  if (h.overflow) {
    const int slot = atomicAdd(redo_count, 1);
    if (slot < kRedoList) {
      redo_list[slot] = (int)k;
      return;                                                         // written by the second pass
    }
  }
  write_hit(out, k, S, h);
}

// Second pass over the rays whose first-pass heap overflowed: the same search from the start
// with a kRedoHeap-entry heap per thread in global memory (heaps: kRedoThreads x kRedoHeap).
template <bool kCull, bool kNewton>
__global__ void __launch_bounds__(kRedoThreads) k_trace_rays_redo(const double* __restrict__ origins,
                                                                  const double* __restrict__ dirs, int np,
                                                                  const double* __restrict__ nets,
                                                                  const double* __restrict__ boxes,
                                                                  const CullNet* __restrict__ culls,
                                                                  RayOut out, const int* __restrict__ redo_count,
                                                                  const int* __restrict__ redo_list,
                                                                  Cand* __restrict__ heaps) {
  __shared__ WarpSmem<kCull> wsm[kRedoThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  const int count = min(*redo_count, kRedoList);
  for (int base = 0; base < count; base += kRedoThreads) {   // uniform trip count: the warp stays whole
    const int i = base + tid;
    const bool active = i < count;
    const long long k = active ? redo_list[i] : 0;
    Ray r;
    Heap h(heaps + (size_t)tid * kRedoHeap, kRedoHeap);
    if (active) {
      load_ray(origins, dirs, k, r);
      push_roots<kCull>(h, r, boxes, culls, np);
    }
    Search S;
    S.live = active;
    search_all<kCull, kNewton>(h, r, nets, boxes, culls, np, S, wsm[tid >> 5], lane);
    if (active) write_hit(out, k, S, h);
  }
}

}  // namespace

// One allocation per shell: kRedoThreads x kRedoHeap candidates (at the 256-byte aligned base),
// then two counters (queries sent to the second pass, global heaps claimed) and the redo list.
shell_status search_scratch(Shell& s, void** heaps, int** counters, int** redo_list) {
  if (!s.d_search) {
    const size_t bytes = sizeof(bz::Cand) * (size_t)bz::kRedoThreads * bz::kRedoHeap + sizeof(int) * (4 + bz::kRedoList);
    const cudaError_t e = cudaMalloc(&s.d_search, bytes);
    if (e != cudaSuccess) {
      cudaGetLastError();
      s.d_search = nullptr;
      return fail(SHELL_ERR_OOM, std::string("search scratch: ") + cudaGetErrorString(e));
    }
  }
  *heaps = s.d_search;
  *counters = (int*)((bz::Cand*)s.d_search + (size_t)bz::kRedoThreads * bz::kRedoHeap);
  *redo_list = *counters + 4;   // counters: redo count, spill count, query counter, pad
  return SHELL_OK;
}

}  // namespace bhem

using namespace bhem;

extern "C" shell_status shell_trace_rays(shell_t* shell, const double* q, long long n_rays, const double* origins,
                                         const double* dirs, int variant, double* tau, int* patch, double* uv,
                                         int* flags, int* stats) {
  if (!shell) return fail(SHELL_ERR_ARG, "NULL shell");
  if (variant != SHELL_RAY_MIDPOINT && variant != SHELL_RAY_NEWTON) return fail(SHELL_ERR_ARG, "ray variant");
  if (n_rays < 0 || n_rays > INT32_MAX) return fail(SHELL_ERR_ARG, "n_rays outside [0, 2^31 - 1]");
  if (n_rays == 0) return SHELL_OK;
  if (!q || !origins || !dirs || !tau || !patch || !uv || !flags) return fail(SHELL_ERR_ARG, "NULL argument");
  Shell& s = *shell;
  const int np = s.n_patches;
  void* heaps_v = nullptr;
  int *redo_count = nullptr, *redo_list = nullptr;
  BHEM_TRY(search_scratch(s, &heaps_v, &redo_count, &redo_list));
  if (!s.d_ray_nets) {
    const size_t ngroups = ((size_t)np + kGroup - 1) / kGroup;
    const cudaError_t e = cudaMalloc((void**)&s.d_ray_nets, sizeof(double) * (56 * (size_t)np + 8 * ngroups) + sizeof(CullNet) * np);
    if (e != cudaSuccess) {
      cudaGetLastError();
      s.d_ray_nets = nullptr;
      return fail(SHELL_ERR_OOM, std::string("ray nets: ") + cudaGetErrorString(e));
    }
  }
  Cand* heaps = (Cand*)heaps_v;
  double* nets = s.d_ray_nets;
  double* boxes = nets + 48 * (size_t)np;
  double* gboxes = boxes + 8 * (size_t)np;
  const int ngroups = (np + kGroup - 1) / kGroup;
  // with statistics, which are those of the plain search, nothing is culled
  CullNet* culls = stats ? nullptr : reinterpret_cast<CullNet*>(gboxes + 8 * (size_t)ngroups);
  RayOut out{tau, patch, uv, flags, stats};
  BHEM_CUDA(cudaMemsetAsync(redo_count, 0, 2 * sizeof(int), s.stream));
  k_ray_nets<<<grid_for(np, kNetBlock), kNetBlock, 0, s.stream>>>(np, s.d_patch_nodes, q, s.grid.dxi1,
                                                                  s.grid.dxi2, nets, boxes, culls);
  k_ray_groups<<<grid_for(ngroups, kNetBlock), kNetBlock, 0, s.stream>>>(np, boxes, gboxes);
  const unsigned ctas = (unsigned)((n_rays + kRayBlock - 1) / kRayBlock);
  const bool newton = variant == SHELL_RAY_NEWTON;
  auto trace = culls ? (newton ? k_trace_rays<true, true> : k_trace_rays<true, false>)
                     : (newton ? k_trace_rays<false, true> : k_trace_rays<false, false>);
  auto redo = culls ? (newton ? k_trace_rays_redo<true, true> : k_trace_rays_redo<true, false>)
                    : (newton ? k_trace_rays_redo<false, true> : k_trace_rays_redo<false, false>);
  trace<<<ctas, kRayBlock, 0, s.stream>>>(n_rays, origins, dirs, np, nets, boxes, gboxes, culls, out, redo_count,
                                          redo_list, heaps);
  redo<<<1, kRedoThreads, 0, s.stream>>>(origins, dirs, np, nets, boxes, culls, out, redo_count, redo_list, heaps);
  s.launches += 4;
  BHEM_CUDA(cudaGetLastError());
  return SHELL_OK;
}
