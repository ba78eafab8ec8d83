// Device building blocks shared by the ray-patch intersection (rays.cu) and the point-patch
// continuous collision detection (ccd.cu) of Sec. 5: the Bezier net of a Hermite patch, cuts of
// a cubic to a parameter range by blossoming, Bezier evaluation, a 3x3 determinant, and the
// candidate heap. Files that include this header are compiled without mul-add contraction, so
// every product and sum here is rounded on its own, in the order written.
#pragma once

#include <cmath>

#include "bhem.h"

namespace bhem {
namespace bz {

constexpr double kNbhd = 1e-3;       // abandoned neighbourhood, fraction of the parameter extent
constexpr int kNewtonIters = 12;
constexpr int kMaxExpansions = 65536;
constexpr int kHeapCap = SHELL_RAY_HEAP;
constexpr int kRedoThreads = 128;    // global heaps: kRedoThreads of kRedoHeap candidates
constexpr int kRedoHeap = 8192;
constexpr int kRedoList = 65536;     // queries the second pass can take per call

// Bezier net P ([c][i][j], i along theta1) of the patch with corner nodes nd (00, 10, 01, 11):
// Hermite data b0 = a, b1 = a + a'/3, b2 = b - b'/3, b3 = b along theta1, then theta2;
// derivative DOFs scaled to the local parameters by dxi1, dxi2.
__device__ __forceinline__ void patch_net(const double* __restrict__ q, const int nd[4], double dxi1, double dxi2,
                                          double* __restrict__ P) {
  for (int c = 0; c < 3; ++c) {
    double H[4][4];   // H[2 pu + r][2 pv + s]: theta1 end pu, derivative order r; theta2 likewise
#pragma unroll
    for (int pv = 0; pv < 2; ++pv)
#pragma unroll
      for (int pu = 0; pu < 2; ++pu) {
        const double* X = q + 12 * (size_t)nd[pu + 2 * pv];
        H[2 * pu][2 * pv] = X[c];
        H[2 * pu + 1][2 * pv] = X[3 + c] * dxi1;
        H[2 * pu][2 * pv + 1] = X[6 + c] * dxi2;
        H[2 * pu + 1][2 * pv + 1] = X[9 + c] * dxi1 * dxi2;
      }
    double U[4][4];   // along theta1 first, then theta2
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      U[0][b] = H[0][b];
      U[1][b] = H[0][b] + H[1][b] / 3.0;
      U[2][b] = H[2][b] - H[3][b] / 3.0;
      U[3][b] = H[2][b];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      P[16 * c + 4 * i + 0] = U[i][0];
      P[16 * c + 4 * i + 1] = U[i][0] + U[i][1] / 3.0;
      P[16 * c + 4 * i + 2] = U[i][2] - U[i][3] / 3.0;
      P[16 * c + 4 * i + 3] = U[i][2];
    }
  }
}

__device__ __forceinline__ double lerp(double p, double q, double t) { return (1.0 - t) * p + t * q; }

// Bezier points of the cubic with points in[0..3] restricted to [a, b] (blossom values).
__device__ __forceinline__ void curve_restrict(const double in[4], double a, double b, double out[4]) {
  double A1[3], B1[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    A1[i] = lerp(in[i], in[i + 1], a);
    B1[i] = lerp(in[i], in[i + 1], b);
  }
  double AA[2], AB[2], BB[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    AA[i] = lerp(A1[i], A1[i + 1], a);
    AB[i] = lerp(A1[i], A1[i + 1], b);
    BB[i] = lerp(B1[i], B1[i + 1], b);
  }
  out[0] = lerp(AA[0], AA[1], a);
  out[1] = lerp(AA[0], AA[1], b);
  out[2] = lerp(AB[0], AB[1], b);
  out[3] = lerp(BB[0], BB[1], b);
}

// 4x4 transpose over four neighbouring lanes (c = lane % 4): lane c's o[j] becomes lane j's o[c].
// All 32 lanes of the warp call it.
__device__ __forceinline__ void transpose4(double o[4], int c) {
  {
    const bool h = c & 2;
    const double a = __shfl_xor_sync(0xffffffffu, h ? o[0] : o[2], 2);
    const double b = __shfl_xor_sync(0xffffffffu, h ? o[1] : o[3], 2);
    o[0] = h ? a : o[0];
    o[1] = h ? b : o[1];
    o[2] = h ? o[2] : a;
    o[3] = h ? o[3] : b;
  }
  {
    const bool h = c & 1;
    const double a = __shfl_xor_sync(0xffffffffu, h ? o[0] : o[1], 1);
    const double b = __shfl_xor_sync(0xffffffffu, h ? o[2] : o[3], 1);
    o[0] = h ? a : o[0];
    o[1] = h ? o[1] : a;
    o[2] = h ? b : o[2];
    o[3] = h ? o[3] : b;
  }
}

// A coordinate's net Pc ([i][j]) cut to [u0, u1] x [v0, v1] by four neighbouring lanes: lane c cuts
// the theta1-curve c, then the theta2-curve c, and returns row S[c][0..3] (the operations of one
// thread cutting all eight curves). All 32 lanes of the warp call it.
__device__ __forceinline__ void cut_row(const double* __restrict__ Pc, int c, const double* R, double S[4]) {
  const double in[4] = {__ldg(Pc + c), __ldg(Pc + 4 + c), __ldg(Pc + 8 + c), __ldg(Pc + 12 + c)};
  double T[4];
  curve_restrict(in, R[0], R[1], T);
  transpose4(T, c);
  curve_restrict(T, R[2], R[3], S);
}

// Cubic Bernstein polynomials and their derivatives at t.
__device__ __forceinline__ void bernstein(double t, double B[4], double dB[4]) {
  const double s = 1.0 - t;
  B[0] = s * s * s;
  B[1] = 3.0 * t * s * s;
  B[2] = 3.0 * t * t * s;
  B[3] = t * t * t;
  dB[0] = -3.0 * s * s;
  dB[1] = 3.0 * s * (s - 2.0 * t);
  dB[2] = 3.0 * t * (2.0 * s - t);
  dB[3] = 3.0 * t * t;
}

// x(u, v), x_u, x_v of one coordinate's net Pc ([i][j]) from the Bernstein values: sums over j first,
// then i.
__device__ __forceinline__ void bezier_eval_coord(const double* __restrict__ Pc, const double Bu[4], const double dBu[4],
                                                  const double Bv[4], const double dBv[4], double& x, double& xu,
                                                  double& xv) {
  double Q[4], R[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double* row = Pc + 4 * i;
    const double p0 = __ldg(row), p1 = __ldg(row + 1), p2 = __ldg(row + 2), p3 = __ldg(row + 3);
    Q[i] = ((Bv[0] * p0 + Bv[1] * p1) + Bv[2] * p2) + Bv[3] * p3;
    R[i] = ((dBv[0] * p0 + dBv[1] * p1) + dBv[2] * p2) + dBv[3] * p3;
  }
  x = ((Bu[0] * Q[0] + Bu[1] * Q[1]) + Bu[2] * Q[2]) + Bu[3] * Q[3];
  xu = ((dBu[0] * Q[0] + dBu[1] * Q[1]) + dBu[2] * Q[2]) + dBu[3] * Q[3];
  xv = ((Bu[0] * R[0] + Bu[1] * R[1]) + Bu[2] * R[2]) + Bu[3] * R[3];
}

// x(u, v), x_u, x_v of the net P ([c][i][j]).
static __device__ void bezier_eval(const double* __restrict__ P, double u, double v, double x[3], double xu[3],
                            double xv[3]) {
  double Bu[4], dBu[4], Bv[4], dBv[4];
  bernstein(u, Bu, dBu);
  bernstein(v, Bv, dBv);
#pragma unroll
  for (int c = 0; c < 3; ++c) bezier_eval_coord(P + 16 * c, Bu, dBu, Bv, dBv, x[c], xu[c], xv[c]);
}

__device__ __forceinline__ double det3(const double M[3][3]) {
  return (M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) -
          M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0])) +
         M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
}

// Component k of the Newton step -J^-1 F by Cramer's rule; *ok: |det J| is large enough.
__device__ __forceinline__ double cramer_component(const double J[3][3], const double F[3], int k, bool* ok) {
  const double det = det3(J);
  *ok = fabs(det) > 1e-300;
  double M[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int s = 0; s < 3; ++s) M[r][s] = s == k ? -F[r] : J[r][s];
  return det3(M) / det;
}

// Lane of the n-th set bit of a warp mask (n from 0; 0 when there is none).
__device__ __forceinline__ int nth_lane(unsigned mask, int n) {
  const unsigned l = __fns(mask, 0, n + 1);
  return l < 32 ? (int)l : 0;
}

// ------------------------------------------------------------------------------------------
// FP32 culling of sub-patches that a query provably cannot meet.
//
// The searches spend their time in FP64 boxes of children (GB300 issues an FP64 warp instruction in
// the time of about 64 FP32 ones), and most children are either off the query's path or stay in the
// heap without ever giving a hit, because an axis-aligned box of a tilted surface is loose. A child
// whose control points lie on one side of a plane through the query's path cannot hold the surface
// point of a hit, nor can any of its descendants (convex hull property), so leaving it out changes no
// hit: the candidates that do lead to hits keep their FP64 keys and, by them, their order. Candidates of
// equal keys are popped in an order that the heap's other entries decide; the culled search watches for
// those that can matter and then searches again without culling (Ties). The test is FP32
// with a margin kCullRel R (R: sum of the magnitudes that enter) that covers every rounding in it:
// net, path and parameters rounded to FP32 (1 + 12 units), 6 levels of blends (18), the projections
// (10): under 48 units of 2^-24 against 64; and at least kCullAbs, twelve times what a refined
// candidate (a box of 1e-9 that the path touches) or a converged Newton iterate (1e-12) may be off.
// ------------------------------------------------------------------------------------------
constexpr float kCullRel = 64.0f / 16777216.0f;
constexpr float kCullAbs = 2e-8f;
constexpr float kCullFar = 1e4f;   // no culling beyond this distance from the origin

__device__ __forceinline__ float lerp32(float p, float q, float t) { return __fmaf_rn(t, q - p, p); }

// in place: the cubic with points x[0], x[S], x[2S], x[3S] restricted to [a, b] (blossom values)
template <int S>
__device__ __forceinline__ void restrict32(float* x, float a, float b) {
  float A[3], B[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    A[i] = lerp32(x[S * i], x[S * (i + 1)], a);
    B[i] = lerp32(x[S * i], x[S * (i + 1)], b);
  }
  const float aa0 = lerp32(A[0], A[1], a), aa1 = lerp32(A[1], A[2], a);
  const float ab0 = lerp32(A[0], A[1], b), ab1 = lerp32(A[1], A[2], b);
  const float bb0 = lerp32(B[0], B[1], b), bb1 = lerp32(B[1], B[2], b);
  x[0] = lerp32(aa0, aa1, a);
  x[S] = lerp32(aa0, aa1, b);
  x[2 * S] = lerp32(ab0, ab1, b);
  x[3 * S] = lerp32(bb0, bb1, b);
}

// in place: the 4x4 net x[4 i + j] restricted to [u0, u1] x [v0, v1]
__device__ __forceinline__ void restrict_net32(float x[16], const float r[4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) restrict32<4>(x + j, r[0], r[1]);
#pragma unroll
  for (int i = 0; i < 4; ++i) restrict32<1>(x + 4 * i, r[2], r[3]);
}

// Whether all 16 values are above eps or all below -eps.
__device__ __forceinline__ bool one_side32(const float x[16], float eps) {
  float mn = x[0], mx = x[0];
#pragma unroll
  for (int k = 1; k < 16; ++k) {
    mn = fminf(mn, x[k]);
    mx = fmaxf(mx, x[k]);
  }
  return mn > eps || mx < -eps;
}

// The same for the combination p x + q y.
__device__ __forceinline__ bool one_side32(const float x[16], const float y[16], float p, float q, float eps) {
  float mn = INFINITY, mx = -INFINITY;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const float v = __fmaf_rn(p, x[k], q * y[k]);
    mn = fminf(mn, v);
    mx = fmaxf(mx, v);
  }
  const float e = (fabsf(p) + fabsf(q)) * eps;
  return mn > e || mx < -e;
}

// FP32 copy of a net relative to its centre point (the mean of its corners): N[c][i][j], centre C[3],
// and the largest 1-norm of a control point.
__device__ __forceinline__ void center_net32(const double* P, float* N, double* C, float& radius) {
  float r = 0.f;
  for (int c = 0; c < 3; ++c) C[c] = 0.25 * ((P[16 * c] + P[16 * c + 3]) + (P[16 * c + 12] + P[16 * c + 15]));
  for (int k = 0; k < 16; ++k) {
    float n = 0.f;
    for (int c = 0; c < 3; ++c) {
      const float v = (float)(P[16 * c + k] - C[c]);
      N[16 * c + k] = v;
      n += fabsf(v);
    }
    r = fmaxf(r, n);
  }
  radius = r;
}

struct Cand {
  double t0, t1, ext, u0, u1, v0, v1;
  int patch;
};

// Order-dependent results of a culled search. Of candidates with equal keys the heap pops first whichever its
// other entries have brought to the top, and those are not the same when some are left out. That changes the
// result in two ways only: two roots of exactly equal tau, of which the first found stays; and equal keys
// within eps of the best hit, since a candidate that near to it is not searched any more (candidates of
// an earlier key all are, in whichever order, and the least of their hits wins). Rays and points aimed at
// nodes and patch edges, or points that start on the surface, meet such ties. Keys are at least -0, so they
// compare as integers without the sign (an FP64 comparison costs as much as 64 of those).
struct Ties {
  long long last = -1;   // the largest key that another entry of the heap shared
  bool again = false;    // the search is void: it has to be repeated without culling

  // after a pop of c: top is the key of the heap's next entry, if it has one. Equal keys of candidates a
  // thousandth of a patch wide hardly ever end without mattering, so the search is not carried on (20,000
  // points that start on a drape, Newton split: 25 ms instead of 30; 20 without culling, the one kind of call
  // found that it slows down).
  __device__ __forceinline__ void popped(const Cand& c, bool more, const double& top, double best, double eps) {
    constexpr long long kAbs = 0x7fffffffffffffffLL;
    const long long k = __double_as_longlong(c.t0) & kAbs;
    if (!more || (__double_as_longlong(top) & kAbs) != k) return;
    if (k > last) last = k;
    if (c.u1 - c.u0 <= 0x1p-10 && c.v1 - c.v0 <= 0x1p-10) again = true;
    hit(best, eps);
  }
  __device__ __forceinline__ void root(double t, double best) { again = again || t == best; }
  // after best has changed
  __device__ __forceinline__ void hit(double best, double eps) {
    again = again || (last >= 0 && __longlong_as_double(last) >= best - 2.0 * eps);
  }
};

// Binary min-heap on t0 (sift rules of a textbook binary heap) over caller-given storage: a
// local array in the first pass, a slice of library-owned global memory in the second. A full
// first-pass heap moves itself into a free global slice (spill, kRedoThreads slices of kRedoHeap
// entries, claimed through *spill_count) and carries on; only when none is left does it report
// an overflow.
struct Heap {
  Cand* a;
  int cap;
  int n = 0, peak = 0;
  int boxes = 0;       // candidate boxes formed (patch roots included)
  bool overflow = false;
  Cand* spill = nullptr;
  int* spill_count = nullptr;

  __device__ Heap(Cand* storage, int capacity) : a(storage), cap(capacity) {}

  __device__ void push(const Cand& c) {
    if (n == cap) {
      if (spill) {
        const int slot = atomicAdd(spill_count, 1);
        if (slot < kRedoThreads) {
          Cand* g = spill + (size_t)slot * kRedoHeap;
          for (int i = 0; i < n; ++i) g[i] = a[i];
          a = g;
          cap = kRedoHeap;
        }
        spill = nullptr;
      }
      if (n == cap) {
        overflow = true;
        return;
      }
    }
    int i = n++;
    if (n > peak) peak = n;
    while (i > 0) {
      const int parent = (i - 1) / 2;
      if (a[parent].t0 <= c.t0) break;
      a[i] = a[parent];
      i = parent;
    }
    a[i] = c;
  }

  __device__ Cand pop() {
    const Cand top = a[0], last = a[--n];
    int i = 0;
    for (;;) {
      const int l = 2 * i + 1, r = l + 1;
      int m = i;
      double km = last.t0;
      if (l < n && a[l].t0 < km) {
        m = l;
        km = a[l].t0;
      }
      if (r < n && a[r].t0 < km) m = r;
      if (m == i) break;
      a[i] = a[m];
      i = m;
    }
    if (n > 0) a[i] = last;
    return top;
  }
};

}  // namespace bz
}  // namespace bhem
