// Point-patch continuous collision detection (Sec. 5, "Dynamic Ray-Patch Intersection",
// Eq. ineqccd): the earliest time in a step at which each moving point meets the moving shell.
//
// Over the step the control points move linearly, p_ij + s dp_ij (s = t / dt in [0, 1]; dp is
// the Bezier net of the nodal displacement over the step), and a point moves as x0 + s dx.
//
//   k_ccd_nets   one thread per patch: start net P, displacement net dP and the swept box (the
//                box of p_ij and p_ij + dp_ij).
//   k_ccd_groups the swept box of every kGroup consecutive patches, to skip groups whole.
//   k_ccd_points one point per thread, FP64. Patches whose swept box misses the point's segment
//                box are skipped; the others enter a binary min-heap keyed by their earliest
//                feasible time s_min. Feasible times of a (sub)net: for each axis and each face
//                of its box, the union over control points of the half-lines a + b s <= 0 is
//                the real line minus one open interval (L, R); [0, 1] minus those six intervals
//                is a sorted list of closed intervals. A candidate whose start-box side plus
//                displacement-box side is at most kEpsX on every axis is refined (contact at
//                s_min); otherwise it is split at its parameter midpoint (Fig. submid) or, in the
//                Newton variant, around a root of x(u, v, s) = x0 + s dx found by Newton's
//                method in (u, v, s), whose neighbourhood is abandoned (Fig. subany). The search
//                ends when the heap's top cannot beat the best s. Feasibility tests, of the
//                patch roots (up to four per lane per round, in patch order) and of the children
//                of every split, are pooled over the warp, one job per (sub)patch and axis; the
//                owner lane then removes the intervals in order. Full local heaps move into
//                global ones as in the ray search.
//                Without statistics, roots and children that an FP32 test proves to lead to no contact
//                are left out before their FP64 feasibility tests (bezier.cuh), most patches fall to an
//                FP32 box comparison, points whose contact could depend on the order of equal keys are searched
//                again in full (bezier.cuh, Ties), and in every form Newton iterations run one at a time beside the
//                other lanes' splits, few of them or few axis jobs on eight lanes each. FP64 issue bounds
//                this kernel (a warp instruction per 64 cycles and sub-partition, whether for one lane
//                or 32): in bulk the operations count, in a long search left alone their chain.
//                Measured, Newton split: drape 262,144 points 119 -> 47 ms, 4,000 points 17.3 -> 5.8 ms;
//                cylinder 33 -> 16.5 ms, plane 6.2 -> 2.8 ms. Midpoint split (half of whose levels are
//                below the test's margin): drape 112 -> 86 ms, plane 58 -> 48 ms.
//   k_ccd_points_redo  points that found no free global heap, searched again from the start.
//
// Compiled without mul-add contraction, like rays.cu: every decision is that of the same IEEE FP64
// operations in the same order as a plain sequential program of these steps.
#include <cmath>

#include "bezier.cuh"
#include "common.cuh"

namespace bhem {
namespace {

using namespace bz;

constexpr double kEpsX = 1e-9;       // refinement size (positions' units)
constexpr double kEpsS = 1e-9;       // stopping test on the normalised time
constexpr int kNetBlock = 128;
constexpr int kCcdBlock = 64;         // 2 warps: the per-warp exchange is 22.7 KB
constexpr int kMaxPieces = 8;        // [0, 1] minus six open intervals has at most 7 pieces
constexpr int kNetStride = 104;      // doubles per patch: P (48), dP (48), swept box (6), unused (2)
constexpr int kGroup = 32;           // consecutive patches per group swept box
// Axis jobs that a warp runs with eight lanes each: four jobs a round of about 220 FP64 operations,
// against 32 jobs a round of about 1,000 with one lane each.
constexpr int kFineJobs = 16;

// FP32 nets of a patch for the culling test: start net relative to its centre, displacement net
struct CullNet {
  double c[3];
  float radius, dradius;   // largest 1-norms of a control point and of a displacement
  float box[6];            // swept box, rounded outwards: min xyz, max xyz
  float n[48], dn[48];
};

__global__ void __launch_bounds__(kNetBlock) k_ccd_nets(int np, const int4* __restrict__ pnodes,
                                                        const double* __restrict__ q, const double* __restrict__ dq,
                                                        double dxi1, double dxi2, double* __restrict__ nets,
                                                        CullNet* __restrict__ culls) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= np) return;
  const int4 n4 = pnodes[p];
  const int nd[4] = {n4.x, n4.y, n4.z, n4.w};
  double* P = nets + (size_t)p * kNetStride;
  double* dP = P + 48;
  double* box = P + 96;
  patch_net(q, nd, dxi1, dxi2, P);
  patch_net(dq, nd, dxi1, dxi2, dP);
  for (int k = 0; k < 3; ++k) {
    double mn = P[16 * k], mx = P[16 * k];
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j) {
        const double a = P[16 * k + 4 * i + j], b = P[16 * k + 4 * i + j] + dP[16 * k + 4 * i + j];
        if (a < mn) mn = a;
        if (a > mx) mx = a;
        if (b < mn) mn = b;
        if (b > mx) mx = b;
      }
    box[k] = mn;
    box[3 + k] = mx;
    if (culls) {
      culls[p].box[k] = __double2float_rd(mn);
      culls[p].box[3 + k] = __double2float_ru(mx);
    }
  }
  box[6] = 0.0;
  box[7] = 0.0;
  if (culls) {
    center_net32(P, culls[p].n, culls[p].c, culls[p].radius);
    float r = 0.f;
    for (int k = 0; k < 16; ++k) {
      float n = 0.f;
      for (int c = 0; c < 3; ++c) {
        const float v = (float)dP[16 * c + k];
        culls[p].dn[16 * c + k] = v;
        n += fabsf(v);
      }
      r = fmaxf(r, n);
    }
    culls[p].dradius = r;
  }
}

// Swept box of every kGroup consecutive patches (min xyz, max xyz of its members' swept boxes,
// 8 doubles per group after the per-patch data). A segment box that misses it misses every
// member's (comparisons only).
__global__ void k_ccd_groups(int np, const double* __restrict__ nets, double* __restrict__ gboxes) {
  const int gi = blockIdx.x * blockDim.x + threadIdx.x;
  const int p0 = gi * kGroup;
  if (p0 >= np) return;
  const int p1 = min(np, p0 + kGroup);
  double mn[3], mx[3];
  for (int c = 0; c < 3; ++c) {
    mn[c] = nets[(size_t)p0 * kNetStride + 96 + c];
    mx[c] = nets[(size_t)p0 * kNetStride + 99 + c];
  }
  for (int p = p0 + 1; p < p1; ++p)
    for (int c = 0; c < 3; ++c) {
      const double a = nets[(size_t)p * kNetStride + 96 + c], b = nets[(size_t)p * kNetStride + 99 + c];
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

// Coordinate k of the sub-net [u0, u1] x [v0, v1] of P ([c][i][j]): S[i][j], theta1-curves cut
// first, then theta2-curves.
__device__ __forceinline__ void cut_coord(const double* __restrict__ P, int k, double u0, double u1, double v0,
                                          double v1, double S[4][4]) {
  const double* Pc = P + 16 * k;
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
  for (int i = 0; i < 4; ++i) curve_restrict(T[i], v0, v1, S[i]);
}

// One axis k of the feasibility test (Eq. ineqccd) of the sub-net [u0, u1] x [v0, v1] of the
// moving net (P, dP) for the point x0 + s dx (x0k = x0[k], dxk = dx[k]): the open intervals
// (L, R) that the lower and upper faces remove from the times (res[0..3] = L_lower, R_lower,
// L_upper, R_upper; *all bit 0 / bit 1 when a face removes nothing because some control point
// has b = 0 on the right side), and the axis's start-box side plus displacement-box side (res[4]).
__device__ void axis_job(const double* __restrict__ P, const double* __restrict__ dP, double u0, double u1,
                         double v0, double v1, int k, double x0k, double dxk, double res[5], int* all) {
  double S[4][4], dS[4][4];
  cut_coord(P, k, u0, u1, v0, v1, S);
  cut_coord(dP, k, u0, u1, v0, v1, dS);
  double Ll = -INFINITY, Rl = INFINITY, Lu = -INFINITY, Ru = INFINITY;   // lower face, upper face
  bool all_l = false, all_u = false;
  double mn = S[0][0], mx = S[0][0], dmn = dS[0][0], dmx = dS[0][0];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // the same updates as a three-way branch on the sign of b, as selects, so that the lanes
      // of a warp do not diverge (r is only used when b != 0)
      const double a = S[i][j] - x0k, b = dS[i][j] - dxk;
      const double r = -a / b;
      const bool pos = b > 0.0, neg = b < 0.0;
      Ll = (pos && r > Ll) ? r : Ll;
      Ru = (pos && r < Ru) ? r : Ru;
      Rl = (neg && r < Rl) ? r : Rl;
      Lu = (neg && r > Lu) ? r : Lu;
      all_l = all_l || (!pos && !neg && a <= 0.0);
      all_u = all_u || (!pos && !neg && a >= 0.0);
      const double sv = S[i][j], dv = dS[i][j];
      if (sv < mn) mn = sv;
      if (sv > mx) mx = sv;
      if (dv < dmn) dmn = dv;
      if (dv > dmx) dmx = dv;
    }
  res[0] = Ll;
  res[1] = Rl;
  res[2] = Lu;
  res[3] = Ru;
  res[4] = (mx - mn) + (dmx - dmn);
  *all = (all_l ? 1 : 0) | (all_u ? 2 : 0);
}

// axis_job by eight neighbouring lanes (lanes 0-3 cut the start net, 4-7 the displacement net, then
// each lane classifies two control points); lane 0 of the eight has the result. The same operations
// in the same places; minima and maxima over the control points in another order. All 32 lanes call it.
__device__ __forceinline__ void axis_job8(const double* __restrict__ P, const double* R, int k, double x0k, double dxk,
                                          double res[5], int* all) {
  const int lane = threadIdx.x & 31, c = lane & 3;
  const bool disp = lane & 4;
  double o[4];
  cut_row(P + (disp ? 48 : 0) + 16 * k, c, R, o);
  // lane c keeps S[c][0..1] and gets dS[c][0..1]; lane 4 + c keeps dS[c][2..3] and gets S[c][2..3]
  const double g0 = __shfl_xor_sync(0xffffffffu, disp ? o[0] : o[2], 4);
  const double g1 = __shfl_xor_sync(0xffffffffu, disp ? o[1] : o[3], 4);
  const double Sv[2] = {disp ? g0 : o[0], disp ? g1 : o[1]}, dS[2] = {disp ? o[2] : g0, disp ? o[3] : g1};
  double Ll = -INFINITY, Rl = INFINITY, Lu = -INFINITY, Ru = INFINITY;
  bool all_l = false, all_u = false;
  double mn = Sv[0], mx = Sv[0], dmn = dS[0], dmx = dS[0];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const double a = Sv[j] - x0k, b = dS[j] - dxk;
    const double r = -a / b;
    const bool pos = b > 0.0, neg = b < 0.0;
    Ll = (pos && r > Ll) ? r : Ll;
    Ru = (pos && r < Ru) ? r : Ru;
    Rl = (neg && r < Rl) ? r : Rl;
    Lu = (neg && r > Lu) ? r : Lu;
    all_l = all_l || (!pos && !neg && a <= 0.0);
    all_u = all_u || (!pos && !neg && a >= 0.0);
    if (Sv[j] < mn) mn = Sv[j];
    if (Sv[j] > mx) mx = Sv[j];
    if (dS[j] < dmn) dmn = dS[j];
    if (dS[j] > dmx) dmx = dS[j];
  }
  auto up = [](double& m, int off) {
    const double y = __shfl_xor_sync(0xffffffffu, m, off);
    if (y > m) m = y;
  };
  auto down = [](double& m, int off) {
    const double y = __shfl_xor_sync(0xffffffffu, m, off);
    if (y < m) m = y;
  };
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) {
    up(Ll, off);
    down(Rl, off);
    up(Lu, off);
    down(Ru, off);
    down(mn, off);
    up(mx, off);
    down(dmn, off);
    up(dmx, off);
  }
  const unsigned group = 0xffu << (lane & 24);
  const unsigned vl = __ballot_sync(0xffffffffu, all_l) & group, vu = __ballot_sync(0xffffffffu, all_u) & group;
  res[0] = Ll;
  res[1] = Rl;
  res[2] = Lu;
  res[3] = Ru;
  res[4] = (mx - mn) + (dmx - dmn);
  *all = (vl ? 1 : 0) | (vu ? 2 : 0);
}

// The feasible times of one (sub)net from its three axis results (ax[k][0..4], all[k]): [0, 1]
// minus the removed intervals, axes in order and the lower face first. False when none is left;
// else the first piece [t0, t1] and the largest per-axis extent (ext).
__device__ bool combine_axes(const double (*ax)[5], const unsigned char* all, double& t0, double& t1,
                             double& ext) {
  double lo[kMaxPieces], hi[kMaxPieces];
  int n = 1;
  lo[0] = 0.0;
  hi[0] = 1.0;
  double e = 0.0;
  for (int k = 0; k < 3; ++k) {
    const double w = ax[k][4];
    if (w > e) e = w;
    for (int side = 0; side < 2; ++side) {
      const double L = ax[k][2 * side], R = ax[k][2 * side + 1];
      if ((all[k] >> side & 1) || !(L < R)) continue;
      // remove the open interval (L, R) from every piece (pieces stay sorted)
      double nlo[kMaxPieces], nhi[kMaxPieces];
      int m = 0;
      for (int p = 0; p < n; ++p) {
        const double a1 = lo[p], b1 = hi[p] < L ? hi[p] : L;
        if (a1 <= b1 && m < kMaxPieces) {
          nlo[m] = a1;
          nhi[m] = b1;
          ++m;
        }
        const double a2 = lo[p] > R ? lo[p] : R, b2 = hi[p];
        if (a2 <= b2 && m < kMaxPieces) {
          nlo[m] = a2;
          nhi[m] = b2;
          ++m;
        }
      }
      n = m;
      for (int p = 0; p < m; ++p) {
        lo[p] = nlo[p];
        hi[p] = nhi[p];
      }
      if (n == 0) return false;
    }
  }
  t0 = lo[0];
  t1 = hi[0];
  ext = e;
  return true;
}

// Newton on F(u, v, s) = X(u, v) + s D(u, v) - x0 - s dx, Jacobian [X_u + s D_u | X_v + s D_v |
// D - dx] by Cramer's rule, at most kNewtonIters iterations; gives up when (u, v) leaves the window
// win (the candidate's rectangle widened by its extent on each side). The lanes of a warp take one
// iteration at a time, beside the other lanes' splits: the iterations vary from one to twelve, and a
// lane that ran them all at once would hold the others up.
struct Query {
  double x0[3], dx[3], seg_lo[3], seg_hi[3], scale;
  float lo32[3], hi32[3];   // the segment's box, rounded outwards
};

__device__ __forceinline__ void load_query(const double* __restrict__ x0s, const double* __restrict__ dxs,
                                           long long k, Query& Q) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Q.x0[c] = x0s[3 * k + c];
    Q.dx[c] = dxs[3 * k + c];
    const double x1 = Q.x0[c] + Q.dx[c];
    Q.seg_lo[c] = Q.x0[c] < x1 ? Q.x0[c] : x1;
    Q.seg_hi[c] = Q.x0[c] < x1 ? x1 : Q.x0[c];
    Q.lo32[c] = __double2float_rd(Q.seg_lo[c]);
    Q.hi32[c] = __double2float_ru(Q.seg_hi[c]);
  }
  Q.scale = (1.0 + sqrt((Q.x0[0] * Q.x0[0] + Q.x0[1] * Q.x0[1]) + Q.x0[2] * Q.x0[2])) +
            sqrt((Q.dx[0] * Q.dx[0] + Q.dx[1] * Q.dx[1]) + Q.dx[2] * Q.dx[2]);
}

struct Search {
  double best = INFINITY, bu = 0.0, bv = 0.0;
  int bp = -1, nexp = 0, flags = 0, newton_iters = 0;
  bool live = false;
  // the candidate being split, its Newton iterations so far (-1: none in progress) and iterate, and
  // whether its children may be culled
  Cand c{};
  int newton = -1;
  double u = 0.0, v = 0.0, s = 0.0;
  bool cullable = false;
  bool cull = true;   // (kCull) false when the point is searched again because of ties
  Ties ties;
};

// Shared-memory exchange of one warp: children listed by each lane in the current split, and
// the axis results computed for them by whichever lanes took the (child, axis) jobs.
struct WarpSmem {
  double rect[32][4][4];
  double ax[32][4][3][5];       // child, axis: L_lower, R_lower, L_upper, R_upper, extent
  double pt[32][6];             // the owner's x0, dx
  int patch[32][4];
  unsigned char all[32][4][3];  // bit 0 / 1: lower / upper face removes nothing
  unsigned short jobs[32 * 12]; // lane * 12 + child * 3 + axis
};

// One iteration from (u, v, s) of every lane with `want`; state 1: converged (at the point given), 2: it
// gives up, 0: the next point. Few lanes are served by eight lanes each (a coordinate of one net and a
// component of the step per lane: about 220 FP64 operations for four iterations, against 850 for one to
// 32), more by themselves. All 32 lanes of the warp call it.
constexpr int kSharedNewton = 12;

__device__ void newton_step(bool want, const double* __restrict__ nets, int patch, WarpSmem& sm, double scale,
                            const double win[4], double& u, double& v, double& s, int& state) {
  const unsigned mask = __ballot_sync(0xffffffffu, want);
  const int count = __popc(mask), lane = threadIdx.x & 31;
  if (count == 0) return;
  double delta[3] = {0.0, 0.0, 0.0};
  if (count <= kSharedNewton) {
    const int rank = __popc(mask & ((1u << lane) - 1u)), g = lane & 24, q = lane & 7;
    const int c = q % 3, net = q / 3 % 2;   // lanes 6, 7 repeat coordinates of the start net
    for (int base = 0; base < count; base += 4) {
      const int own = nth_lane(mask, base + (lane >> 3));
      const int p = __shfl_sync(0xffffffffu, patch, own);
      const double uu = __shfl_sync(0xffffffffu, u, own), vv = __shfl_sync(0xffffffffu, v, own);
      const double ss = __shfl_sync(0xffffffffu, s, own), sc = __shfl_sync(0xffffffffu, scale, own);
      double Bu[4], dBu[4], Bv[4], dBv[4], x, xu, xv;
      bernstein(uu, Bu, dBu);
      bernstein(vv, Bv, dBv);
      bezier_eval_coord(nets + (size_t)p * kNetStride + 48 * net + 16 * c, Bu, dBu, Bv, dBv, x, xu, xv);
      const double D = __shfl_sync(0xffffffffu, x, g + 3 + c), Du = __shfl_sync(0xffffffffu, xu, g + 3 + c),
                   Dv = __shfl_sync(0xffffffffu, xv, g + 3 + c);
      const double dxc = sm.pt[own][3 + c];
      const double f = (x + ss * D) - (sm.pt[own][c] + ss * dxc);
      const double j0 = xu + ss * Du, j1 = xv + ss * Dv, j2 = D - dxc;
      double F[3], J[3][3];
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        F[r] = __shfl_sync(0xffffffffu, f, g + r);
        J[r][0] = __shfl_sync(0xffffffffu, j0, g + r);
        J[r][1] = __shfl_sync(0xffffffffu, j1, g + r);
        J[r][2] = __shfl_sync(0xffffffffu, j2, g + r);
      }
      const double fn = sqrt((F[0] * F[0] + F[1] * F[1]) + F[2] * F[2]);
      bool regular;
      const double step = cramer_component(J, F, c, &regular);
      const int st = fn <= 1e-12 * sc ? 1 : !regular ? 2 : 0;
      const int src = 8 * (rank - base);   // the lanes that serve this one in this round
      const bool mine = want && src >= 0 && src < 32;
      const int got = __shfl_sync(0xffffffffu, st, src & 31);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double y = __shfl_sync(0xffffffffu, step, (src + k) & 31);
        if (mine) delta[k] = y;
      }
      if (mine) state = got;
    }
    if (!want) return;
  } else {
    if (!want) return;
    const double* P = nets + (size_t)patch * kNetStride;
    double X[3], Xu[3], Xv[3], D[3], Du[3], Dv[3], F[3], J[3][3];
    bezier_eval(P, u, v, X, Xu, Xv);
    bezier_eval(P + 48, u, v, D, Du, Dv);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double dxc = sm.pt[lane][3 + c];
      F[c] = (X[c] + s * D[c]) - (sm.pt[lane][c] + s * dxc);
      J[c][0] = Xu[c] + s * Du[c];
      J[c][1] = Xv[c] + s * Dv[c];
      J[c][2] = D[c] - dxc;
    }
    const double fn = sqrt((F[0] * F[0] + F[1] * F[1]) + F[2] * F[2]);
    bool regular = true;
    state = fn <= 1e-12 * scale ? 1 : 0;
    if (state == 0)
#pragma unroll
      for (int k = 0; k < 3; ++k) delta[k] = cramer_component(J, F, k, &regular);
    if (!regular) state = 2;
  }
  if (state) return;
  u += delta[0];
  v += delta[1];
  s += delta[2];
  if (!isfinite(u) || !isfinite(v) || !isfinite(s) || u < win[0] || u > win[1] || v < win[2] || v > win[3])
    state = 2;   // left the window
}

__device__ __forceinline__ void put_rect(WarpSmem& sm, int lane, int& nch, int patch, double u0, double u1,
                                         double v0, double v1) {
  if (!(u1 > u0) || !(v1 > v0)) return;
  sm.patch[lane][nch] = patch;
  double* R = sm.rect[lane][nch++];
  R[0] = u0;
  R[1] = u1;
  R[2] = v0;
  R[3] = v1;
}

// Culling data of one lane, in the memory of its axis results (written only after the culling):
// the times between which a contact of its children matters and the margin's least value.
struct CullTimes { float s0, s1, margin; };
__device__ __forceinline__ CullTimes& cull_times(WarpSmem& sm, int lane) {
  return *reinterpret_cast<CullTimes*>(&sm.ax[lane][0][0][0]);
}

__device__ __forceinline__ float cull_margin(const CullNet* __restrict__ N, const float X[3], const float dX[3],
                                             float least) {
  const float r = ((fabsf(X[0]) + fabsf(X[1])) + fabsf(X[2])) + ((fabsf(dX[0]) + fabsf(dX[1])) + fabsf(dX[2]));
  return fmaxf(least, kCullRel * (N->radius + N->dradius + r));
}

// Culling test of one child: at both ends of the times that matter (the motion is linear, so all
// through them) the control points lie on one side of a plane through the moving point. Planes tried:
// the child's tangent plane at the start of those times and the planes along its two chords normal to it.
__device__ bool child_is_culled(const CullNet* __restrict__ N, const double* pt, const CullTimes T, const double* R) {
  const float r[4] = {(float)R[0], (float)R[1], (float)R[2], (float)R[3]};
  float X[3], dX[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    X[c] = (float)(pt[c] - N->c[c]);
    dX[c] = (float)pt[3 + c];
  }
  const float eps = cull_margin(N, X, dX, T.margin);
  // corners of the child at time s0 (any directions would do: they only choose the planes)
  float Bu[2][4], Bv[2][4];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float u = r[k], v = r[2 + k], p = 1.f - u, q = 1.f - v;
    Bu[k][0] = p * p * p;
    Bu[k][1] = 3.f * u * p * p;
    Bu[k][2] = 3.f * u * u * p;
    Bu[k][3] = u * u * u;
    Bv[k][0] = q * q * q;
    Bv[k][1] = 3.f * v * q * q;
    Bv[k][2] = 3.f * v * v * q;
    Bv[k][3] = v * v * v;
  }
  float cu[3], cv[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float f[2][2] = {};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float g0 = 0.f, g1 = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float x = __fmaf_rn(T.s0, __ldg(N->dn + 16 * c + 4 * i + j), __ldg(N->n + 16 * c + 4 * i + j));
        g0 = __fmaf_rn(Bv[0][j], x, g0);
        g1 = __fmaf_rn(Bv[1][j], x, g1);
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        f[k][0] = __fmaf_rn(Bu[k][i], g0, f[k][0]);
        f[k][1] = __fmaf_rn(Bu[k][i], g1, f[k][1]);
      }
    }
    cu[c] = (f[1][0] - f[0][0]) + (f[1][1] - f[0][1]);
    cv[c] = (f[0][1] - f[0][0]) + (f[1][1] - f[1][0]);
  }
  const float n[3] = {cu[1] * cv[2] - cu[2] * cv[1], cu[2] * cv[0] - cu[0] * cv[2], cu[0] * cv[1] - cu[1] * cv[0]};
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    float m[3];
    if (k == 0) {
      m[0] = n[0]; m[1] = n[1]; m[2] = n[2];
    } else {
      const float* e = k == 1 ? cv : cu;
      m[0] = n[1] * e[2] - n[2] * e[1];
      m[1] = n[2] * e[0] - n[0] * e[2];
      m[2] = n[0] * e[1] - n[1] * e[0];
    }
    // scaled to a 1-norm of 1 (tiny sub-patches' products would underflow); no plane from a degenerate net
    const float l = fabsf(m[0]) + fabsf(m[1]) + fabsf(m[2]);
    if (!(l > 1e-30f)) continue;
    const float il = 1.f / l;
    float a[16], b[16];
#pragma unroll
    for (int c = 0; c < 3; ++c) m[c] *= il;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      float x = 0.f, d = 0.f;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        x = __fmaf_rn(m[c], __ldg(N->n + 16 * c + i) - X[c], x);
        d = __fmaf_rn(m[c], __ldg(N->dn + 16 * c + i) - dX[c], d);
      }
      a[i] = __fmaf_rn(T.s0, d, x);
      b[i] = __fmaf_rn(T.s1, d, x);
    }
    restrict_net32(a, r);
    restrict_net32(b, r);
    float mn = fminf(a[0], b[0]), mx = fmaxf(a[0], b[0]);
#pragma unroll
    for (int i = 1; i < 16; ++i) {
      mn = fminf(mn, fminf(a[i], b[i]));
      mx = fmaxf(mx, fmaxf(a[i], b[i]));
    }
    if (mn > eps || mx < -eps) return true;
  }
  return false;
}

// Lists the warp's jobs, `per` for each child in a lane's mask `keep` (lane * 12 + child * per + 0 ..
// per - 1), in lane order; returns their number. All 32 lanes call it; ends with a warp barrier.
__device__ __forceinline__ int list_jobs(WarpSmem& sm, int lane, unsigned keep, int per) {
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

// The warp's pool of (lane, child, axis) jobs: every lane lists nch children in sm.rect /
// sm.patch; with kCull those that an FP32 test proves to lead to no contact are left out (lanes with
// cullable set; s0: no contact of its children is earlier); the 3 axes of every child are spread over
// the 32 lanes, then each lane combines its own children's axes and pushes the feasible ones in order.
// All 32 lanes call it together.
template <bool kCull>
__device__ void pool_and_push(Heap& h, const Query& Q, const double* __restrict__ nets,
                              const CullNet* __restrict__ culls, const Search& S, WarpSmem& sm, int lane, int nch,
                              bool cullable, double s0) {
  unsigned keep = (1u << nch) - 1u;
  if constexpr (kCull) {
    CullTimes& T = cull_times(sm, lane);
    T.s0 = (float)s0 - 1e-6f;
    T.s1 = (S.best < 1.0 ? (float)S.best : 1.f) + 1e-6f;
    T.margin = fmaxf(kCullAbs, 4e-12f * (float)Q.scale);   // 4 x Newton's tolerance
    const int total = list_jobs(sm, lane, cullable ? keep : 0u, 1);
    for (int j = lane; j < total; j += 32) {
      const int code = sm.jobs[j], owner = code / 12, ch = code - 12 * owner;
      sm.all[owner][ch][0] =
          child_is_culled(culls + sm.patch[owner][ch], sm.pt[owner], cull_times(sm, owner), sm.rect[owner][ch]);
    }
    __syncwarp();
    if (cullable)
      for (int ch = 0; ch < nch; ++ch)
        if (sm.all[lane][ch][0]) keep &= ~(1u << ch);
    __syncwarp();
  }
  const int total = list_jobs(sm, lane, keep, 3);
  if (total <= kFineJobs) {   // few jobs (a long search left alone): eight lanes each
    for (int base = 0; base < total; base += 4) {
      const int j = base + (lane >> 3), code = sm.jobs[min(j, total - 1)], owner = code / 12, q = code - 12 * owner;
      const int ch = q / 3, k = q % 3;
      double res[5];
      int all = 0;
      axis_job8(nets + (size_t)sm.patch[owner][ch] * kNetStride, sm.rect[owner][ch], k, sm.pt[owner][k],
                sm.pt[owner][3 + k], res, &all);
      if ((lane & 7) == 0 && j < total) {
#pragma unroll
        for (int i = 0; i < 5; ++i) sm.ax[owner][ch][k][i] = res[i];
        sm.all[owner][ch][k] = (unsigned char)all;
      }
    }
  }
  for (int j = lane; total > kFineJobs && j < total; j += 32) {
    const int code = sm.jobs[j], owner = code / 12, q = code - 12 * owner, ch = q / 3, k = q % 3;
    const double* R = sm.rect[owner][ch];
    const double* P = nets + (size_t)sm.patch[owner][ch] * kNetStride;
    int all = 0;
    axis_job(P, P + 48, R[0], R[1], R[2], R[3], k, sm.pt[owner][k], sm.pt[owner][3 + k], sm.ax[owner][ch][k], &all);
    sm.all[owner][ch][k] = (unsigned char)all;
  }
  __syncwarp();
  for (int ch = 0; ch < nch; ++ch) {
    if (!(keep >> ch & 1)) continue;
    double t0, t1, e;
    if (combine_axes(sm.ax[lane][ch], sm.all[lane][ch], t0, t1, e) && !(t0 >= S.best)) {
      const double* R = sm.rect[lane][ch];
      h.push(Cand{t0, t1, e, R[0], R[1], R[2], R[3], sm.patch[lane][ch]});
    }
  }
  __syncwarp();
}

// Whether the FP32 box B surely misses the query's segment box (both rounded outwards).
__device__ __forceinline__ bool surely_missed(const float* B, const Query& Q) {
  return Q.hi32[0] < B[0] || Q.hi32[1] < B[1] || Q.hi32[2] < B[2] || Q.lo32[0] > B[3] || Q.lo32[1] > B[4] ||
         Q.lo32[2] > B[5];
}

// One round of a lane's root scan: the patches from `next` on, in order, whose swept box
// (nets[p * kNetStride + 96 ..]: min xyz, max xyz) meets the query's segment box, up to four;
// true when the scan has passed the last patch.
template <bool kCull>
__device__ __forceinline__ bool root_round(Heap& h, const Query& Q, const double* __restrict__ nets,
                                           const CullNet* __restrict__ culls, int np, WarpSmem& sm, int lane,
                                           int& next, int& nch) {
  while (next < np && nch < 4) {
    if constexpr (kCull) {   // most patches fall to an FP32 comparison
      if (next % kGroup != 0 && surely_missed(culls[next].box, Q)) {
        ++next;
        continue;
      }
    }
    if (next % kGroup == 0) {   // a group that the segment box misses is skipped whole
      const double* G = nets + (size_t)np * kNetStride + (size_t)(next / kGroup) * 8;
      bool gmiss = false;
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if (Q.seg_hi[c] < G[c] || Q.seg_lo[c] > G[3 + c]) gmiss = true;
      if (gmiss) {
        next += kGroup;
        continue;
      }
    }
    const double* sw = nets + (size_t)next * kNetStride + 96;
    bool miss = false;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (Q.seg_hi[c] < sw[c] || Q.seg_lo[c] > sw[3 + c]) miss = true;
    if (!miss) put_rect(sm, lane, nch, next, 0.0, 1.0, 0.0, 1.0);
    ++next;
  }
  h.boxes += nch;
  return next >= np;
}

// Root phase, all 32 lanes together: the pooled feasibility tests push each lane's roots in
// patch order.
template <bool kCull>
__device__ void push_roots(Heap& h, const Query& Q, const double* __restrict__ nets,
                           const CullNet* __restrict__ culls, int np, Search& S, WarpSmem& sm, int lane) {
  int next = 0;
  bool more = S.live;
  while (__any_sync(0xffffffffu, more)) {
    int nch = 0;
    if (more && root_round<kCull>(h, Q, nets, culls, np, sm, lane, next, nch)) more = false;
    pool_and_push<kCull>(h, Q, nets, culls, S, sm, lane, nch, S.cull && Q.scale < kCullFar, 0.0);
  }
}

// One step of a lane's search (lanes with `searching`; all 32 call it): pop the earliest candidate and either finish (nothing earlier can
// remain), record a refined contact, or start to split it; one iteration of its Newton solve; and when
// that is over (or there is none), list its 4 children (Newton pinwheel or midpoint split) for the
// warp's pooled feasibility tests.
template <bool kCull, bool kNewton>
__device__ __forceinline__ void split_step(Heap& h, const Query& Q, const double* __restrict__ nets,
                                           const CullNet* __restrict__ culls, Search& S, WarpSmem& sm,
                                           int lane, int& nch, bool searching) {
  bool split = false, root = false;   // split c now; around the root (u, v, s)
  Cand& c = S.c;
  if (searching && S.newton < 0) {
    if (h.n == 0 || h.overflow) {
      S.live = false;
    } else {
      c = h.pop();
      if constexpr (kCull) S.ties.popped(c, h.n > 0, h.a[0].t0, S.best, kEpsS);
      if ((kCull && S.cull && S.ties.again) || c.t0 >= S.best - kEpsS) {   // nothing left can be earlier
        S.live = false;
      } else if (c.ext <= kEpsX || (c.u1 - c.u0 < 1e-13 && c.v1 - c.v0 < 1e-13)) {   // refined
        if (c.t0 < S.best - kEpsS) {
          S.best = c.t0;
          if constexpr (kCull) S.ties.hit(S.best, kEpsS);
          S.bp = c.patch;
          S.bu = 0.5 * (c.u0 + c.u1);
          S.bv = 0.5 * (c.v0 + c.v1);
        }
      } else if (S.nexp == kMaxExpansions) {
        S.flags |= SHELL_RAY_LIMIT;
        S.live = false;
      } else {
        ++S.nexp;
        if constexpr (kCull) {
          // nothing is culled among children of the margin's size, nor far from the origin (bezier.cuh)
          const CullNet* N = culls + c.patch;
          const float X[3] = {(float)(Q.x0[0] - N->c[0]), (float)(Q.x0[1] - N->c[1]), (float)(Q.x0[2] - N->c[2])};
          const float dX[3] = {(float)Q.dx[0], (float)Q.dx[1], (float)Q.dx[2]};
          S.cullable = S.cull && Q.scale < kCullFar && (float)c.ext > 8.f * cull_margin(N, X, dX, kCullAbs);
        }
        S.u = 0.5 * (c.u0 + c.u1);
        S.v = 0.5 * (c.v0 + c.v1);
        S.s = c.t0;
        if constexpr (kNewton) S.newton = 0;
        else split = true;
      }
    }
  }
  if constexpr (kNewton) {
    const bool want = searching && S.newton >= 0;
    const double wu = c.u1 - c.u0, wv = c.v1 - c.v0;
    const double win[4] = {c.u0 - wu, c.u1 + wu, c.v0 - wv, c.v1 + wv};
    int state = 0;
    newton_step(want, nets, c.patch, sm, Q.scale, win, S.u, S.v, S.s, state);
    if (want) {
      ++S.newton;
      ++S.newton_iters;
      if (state || S.newton == kNewtonIters) {
        S.newton = -1;
        split = true;
        root = state == 1 && S.u >= c.u0 && S.u <= c.u1 && S.v >= c.v0 && S.v <= c.v1 && S.s >= 0.0 && S.s <= 1.0;
      }
    }
  }
  if (!split) return;
  if (root) {
    if constexpr (kCull) S.ties.root(S.s, S.best);
    if (S.s < S.best) {
      S.best = S.s;
      if constexpr (kCull) S.ties.hit(S.best, kEpsS);
      S.bp = c.patch;
      S.bu = S.u;
      S.bv = S.v;
    }
    const double hu = kNbhd * (c.u1 - c.u0), hv = kNbhd * (c.v1 - c.v0);
    const double a1 = fmax(c.u0, S.u - hu), a2 = fmin(c.u1, S.u + hu);
    const double b1 = fmax(c.v0, S.v - hv), b2 = fmin(c.v1, S.v + hv);
    put_rect(sm, lane, nch, c.patch, c.u0, a1, b1, c.v1);
    put_rect(sm, lane, nch, c.patch, a1, c.u1, b2, c.v1);
    put_rect(sm, lane, nch, c.patch, c.u0, a2, c.v0, b1);
    put_rect(sm, lane, nch, c.patch, a2, c.u1, c.v0, b2);
  } else {
    const double um = 0.5 * (c.u0 + c.u1), vm = 0.5 * (c.v0 + c.v1);
    put_rect(sm, lane, nch, c.patch, c.u0, um, vm, c.v1);
    put_rect(sm, lane, nch, c.patch, um, c.u1, vm, c.v1);
    put_rect(sm, lane, nch, c.patch, c.u0, um, c.v0, vm);
    put_rect(sm, lane, nch, c.patch, um, c.u1, c.v0, vm);
  }
  h.boxes += nch;
}

__device__ __forceinline__ void finish_flags(const Heap& h, Search& S) {
  if (h.overflow) {
    S.flags |= SHELL_RAY_OVERFLOW;
  } else if (S.bp >= 0) {
    S.flags |= SHELL_RAY_HIT;
  }
}

// The search over the candidates in each lane's heap, all 32 lanes of the warp together (lanes
// without a query pass live = false).
template <bool kCull, bool kNewton>
__device__ void search(Heap& h, const Query& Q, const double* __restrict__ nets, const CullNet* __restrict__ culls,
                       int np, Search& S, WarpSmem& sm, int lane) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    sm.pt[lane][c] = Q.x0[c];
    sm.pt[lane][3 + c] = Q.dx[c];
  }
  push_roots<kCull>(h, Q, nets, culls, np, S, sm, lane);
  while (__any_sync(0xffffffffu, S.live)) {
    int nch = 0;
    split_step<kCull, kNewton>(h, Q, nets, culls, S, sm, lane, nch, S.live);
    pool_and_push<kCull>(h, Q, nets, culls, S, sm, lane, nch, S.cullable, S.c.t0);
  }
  finish_flags(h, S);
}

// Whether the point has to be searched again without culling.
template <bool kCull>
__device__ __forceinline__ bool ties_matter(const Heap& h, const Search& S) {
  return kCull && S.cull && S.ties.again && !h.overflow;
}

struct CcdOut {
  double* s;
  int* patch;
  double* uv;
  int* flags;
  int* stats;
};

__device__ __forceinline__ void write_result(const CcdOut& out, long long k, const Search& S, const Heap& h) {
  const bool hit = (S.flags & SHELL_RAY_HIT) != 0;
  out.s[k] = hit ? S.best : INFINITY;
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

// Persistent over the queries: every lane starts on query (global lane index) and, when its
// search ends, writes the result and takes the next query from counters[2], while the other lanes
// of its warp go on. A lane's root scan and splits feed the same pooled feasibility tests, so a
// warp keeps all its lanes busy until the queue is empty; each query's heap receives the same
// pushes in the same order as in a one-query-per-lane search.
template <bool kCull, bool kNewton>
__global__ void __launch_bounds__(kCcdBlock, 8) k_ccd_points(long long n, const double* __restrict__ x0s,
                                                             const double* __restrict__ dxs, int np,
                                                             const double* __restrict__ nets,
                                                             const CullNet* __restrict__ culls,
                                                             CcdOut out, int* __restrict__ counters,
                                                             int* __restrict__ redo_list, Cand* __restrict__ heaps) {
  __shared__ WarpSmem wsm[kCcdBlock / 32];
  WarpSmem& sm = wsm[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const long long lanes = (long long)gridDim.x * blockDim.x;
  Cand storage[kHeapCap];
  Heap h(storage, kHeapCap);
  Query Q{};
  Search S;
  long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int phase = 0, next = 0;   // phase 0: no query left, 1: root scan, 2: search
  auto begin = [&]() {
    h.a = storage;
    h.cap = kHeapCap;
    h.n = 0;
    h.peak = 0;
    h.boxes = 0;
    h.overflow = false;
    h.spill = heaps;
    h.spill_count = counters + 1;
    S = Search();
    phase = 0;
    if (k < n) {
      load_query(x0s, dxs, k, Q);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        sm.pt[lane][c] = Q.x0[c];
        sm.pt[lane][3 + c] = Q.dx[c];
      }
      S.live = true;
      phase = 1;
      next = 0;
    }
  };
  begin();
  while (__any_sync(0xffffffffu, phase != 0)) {
    int nch = 0;
    const bool scan = phase == 1, searching = phase == 2;
    if (scan && root_round<kCull>(h, Q, nets, culls, np, sm, lane, next, nch)) phase = 2;
    split_step<kCull, kNewton>(h, Q, nets, culls, S, sm, lane, nch, searching);
    pool_and_push<kCull>(h, Q, nets, culls, S, sm, lane, nch, scan ? S.cull && Q.scale < kCullFar : S.cullable,
                         scan ? 0.0 : S.c.t0);   // ends with a warp barrier: sm.pt may change below
    if (searching && !S.live) {
      finish_flags(h, S);
      if (ties_matter<kCull>(h, S)) {
        h.n = 0;
        h.boxes = 0;
        S = Search();
        S.cull = false;
        S.live = true;
        phase = 1;
        next = 0;
        continue;
      }
      bool deferred = false;
      if (h.overflow) {
        const int slot = atomicAdd(counters, 1);
        if (slot < kRedoList) {
          redo_list[slot] = (int)k;   // written by the second pass
          deferred = true;
        }
      }
      if (!deferred) write_result(out, k, S, h);
      k = lanes + atomicAdd(counters + 2, 1);
      begin();
    }
  }
}

template <bool kCull, bool kNewton>
__global__ void __launch_bounds__(kCcdBlock) k_ccd_points_redo(const double* __restrict__ x0s,
                                                                  const double* __restrict__ dxs, int np,
                                                                  const double* __restrict__ nets,
                                                                  const CullNet* __restrict__ culls,
                                                                  CcdOut out, const int* __restrict__ counters,
                                                                  const int* __restrict__ redo_list,
                                                                  Cand* __restrict__ heaps) {
  __shared__ WarpSmem wsm[kCcdBlock / 32];
  const int tid = blockIdx.x * kCcdBlock + threadIdx.x, lane = threadIdx.x & 31;
  const int count = min(counters[0], kRedoList);
  for (int base = 0; base < count; base += kRedoThreads) {   // uniform trip count: the warp stays whole
    const int i = base + tid;
    const bool active = i < count;
    const long long k = active ? redo_list[i] : 0;
    Query Q;
    Heap h(heaps + (size_t)tid * kRedoHeap, kRedoHeap);
    if (active) load_query(x0s, dxs, k, Q);
    Search S;
    S.live = active;
    search<kCull, kNewton>(h, Q, nets, culls, np, S, wsm[threadIdx.x >> 5], lane);
    const bool again = ties_matter<kCull>(h, S);
    if (__any_sync(0xffffffffu, again)) {
      Search T;
      T.cull = false;
      T.live = again;
      if (again) h.n = 0;
      search<kCull, kNewton>(h, Q, nets, culls, np, T, wsm[threadIdx.x >> 5], lane);
      if (again) S = T;
    }
    if (active) write_result(out, k, S, h);
  }
}

}  // namespace
}  // namespace bhem

using namespace bhem;

extern "C" shell_status shell_ccd_points(shell_t* shell, const double* q, const double* dq, long long n_points,
                                         const double* x0, const double* dx, int variant, double* s, int* patch,
                                         double* uv, int* flags, int* stats) {
  if (!shell) return fail(SHELL_ERR_ARG, "NULL shell");
  if (variant != SHELL_RAY_MIDPOINT && variant != SHELL_RAY_NEWTON) return fail(SHELL_ERR_ARG, "split variant");
  if (n_points < 0 || n_points > INT32_MAX) return fail(SHELL_ERR_ARG, "n_points outside [0, 2^31 - 1]");
  if (n_points == 0) return SHELL_OK;
  if (!q || !dq || !x0 || !dx || !s || !patch || !uv || !flags) return fail(SHELL_ERR_ARG, "NULL argument");
  Shell& sh = *shell;
  const int np = sh.n_patches;
  void* heaps_v = nullptr;
  int *counters = nullptr, *redo_list = nullptr;
  BHEM_TRY(search_scratch(sh, &heaps_v, &counters, &redo_list));
  if (!sh.d_ccd_nets) {
    const size_t ngroups = ((size_t)np + kGroup - 1) / kGroup;
    const cudaError_t e = cudaMalloc((void**)&sh.d_ccd_nets, sizeof(double) * (kNetStride * (size_t)np + 8 * ngroups) + sizeof(CullNet) * np);
    if (e != cudaSuccess) {
      cudaGetLastError();
      sh.d_ccd_nets = nullptr;
      return fail(SHELL_ERR_OOM, std::string("collision nets: ") + cudaGetErrorString(e));
    }
  }
  Cand* heaps = (Cand*)heaps_v;
  // with statistics, which are those of the plain search, nothing is culled
  const int groups = (np + kGroup - 1) / kGroup;
  CullNet* culls =
      stats ? nullptr : reinterpret_cast<CullNet*>(sh.d_ccd_nets + (size_t)kNetStride * np + 8 * (size_t)groups);
  CcdOut out{s, patch, uv, flags, stats};
  BHEM_CUDA(cudaMemsetAsync(counters, 0, 4 * sizeof(int), sh.stream));
  k_ccd_nets<<<grid_for(np, kNetBlock), kNetBlock, 0, sh.stream>>>(np, sh.d_patch_nodes, q, dq, sh.grid.dxi1,
                                                                   sh.grid.dxi2, sh.d_ccd_nets, culls);
  k_ccd_groups<<<grid_for(groups, kNetBlock), kNetBlock, 0, sh.stream>>>(
      np, sh.d_ccd_nets, sh.d_ccd_nets + (size_t)kNetStride * np);
  const bool newton = variant == SHELL_RAY_NEWTON;
  // persistent: exactly the CTAs that can be resident at once (a CTA that waits for a free SM would
  // start only after the queue is empty), lanes refill from the query counter
  if (sh.num_sms <= 0) BHEM_CUDA(cudaDeviceGetAttribute(&sh.num_sms, cudaDevAttrMultiProcessorCount, sh.device));
  auto points = culls ? (newton ? k_ccd_points<true, true> : k_ccd_points<true, false>)
                      : (newton ? k_ccd_points<false, true> : k_ccd_points<false, false>);
  auto redo = culls ? (newton ? k_ccd_points_redo<true, true> : k_ccd_points_redo<true, false>)
                    : (newton ? k_ccd_points_redo<false, true> : k_ccd_points_redo<false, false>);
  int occ = 0;
  BHEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, points, kCcdBlock, 0));
  const long long ctas = std::min<long long>((n_points + kCcdBlock - 1) / kCcdBlock,
                                             (long long)std::max(1, occ) * sh.num_sms);
  points<<<(unsigned)ctas, kCcdBlock, 0, sh.stream>>>(n_points, x0, dx, np, sh.d_ccd_nets, culls, out,
                                                      counters, redo_list, heaps);
  redo<<<kRedoThreads / kCcdBlock, kCcdBlock, 0, sh.stream>>>(x0, dx, np, sh.d_ccd_nets, culls, out,
                                                              counters, redo_list, heaps);
  sh.launches += 4;
  BHEM_CUDA(cudaGetLastError());
  return SHELL_OK;
}
