// Elastic energy and gradient of a shell with no device allocation at all.
//
// Everything here is self-contained: the kernel derives the patch topology from the grid and the
// rest geometry from the rest DOFs, takes the 1D shape factors by value, and keeps its only scratch
// (per-CTA partial sums for the energy, a ticket counter) in one file-scope device array. The caller passes inputs and outputs; no shell object is needed.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"

namespace bhem {
namespace noalloc {

constexpr int kMaxCtas = 16384;
constexpr int kMaxPatches = 8 * kMaxCtas;   // 131072 patches (e.g. 362 x 362)
constexpr int kWarps = 4;                   // patches in flight per CTA (1 on small grids)
constexpr int kSpreadPatches = 608;         // grids up to this run one warp per CTA: one per sub-partition

struct Scratch {
  double partials[kMaxCtas];   // per-CTA energy sums (fully rewritten by every call)
  unsigned ticket;             // last-CTA counter: must be 0 when a call starts
};

// The only scratch memory of this entry point: about 131 KB, held by every GPU that loads the
// library until the process exits.
static __device__ __align__(256) unsigned char g_scratch[sizeof(Scratch)];

// ---- App. A.1 / A.2: 1D factors w[d][gauss][a] of the shape functions and Gauss weights, formed on the
// host (200 values) and passed by value, so that no kernel has to build them first
struct Tables {
  double w1[48], w2[48], wt[16];
};

inline double hermite(int p, int r, double t, int d) {
  const double s = p ? 1.0 - t : t;
  double v;
  if (r == 0) v = d == 0 ? (2 * s - 3) * s * s + 1 : d == 1 ? 6 * s * s - 6 * s : 12 * s - 6;
  else        v = d == 0 ? ((s - 2) * s + 1) * s : d == 1 ? (3 * s - 4) * s + 1 : 6 * s - 4;
  if (p == 1 && r == 1) v = -v;
  if (p == 1 && (d & 1)) v = -v;
  return v;
}

inline Tables make_tables(double d1, double d2) {
  const double xi = std::sqrt(3.0 / 7.0 - 2.0 / 7.0 * std::sqrt(6.0 / 5.0));
  const double xo = std::sqrt(3.0 / 7.0 + 2.0 / 7.0 * std::sqrt(6.0 / 5.0));
  const double th[4] = {0.5 * (1 - xo), 0.5 * (1 - xi), 0.5 * (1 + xi), 0.5 * (1 + xo)};
  const double wi = (18.0 + std::sqrt(30.0)) / 72.0, wo = (18.0 - std::sqrt(30.0)) / 72.0;
  const double wt[4] = {wo, wi, wi, wo};
  Tables T;
  for (int e = 0; e < 48; ++e) {
    const int d = e / 16, g = e / 4 % 4, p = e % 4 >> 1, r = e & 1;
    double v1 = hermite(p, r, th[g], d), v2 = v1;
    if (r) {
      v1 *= d1;
      v2 *= d2;
    }
    for (int i = 0; i < d; ++i) {
      v1 /= d1;
      v2 /= d2;
    }
    T.w1[e] = v1;
    T.w2[e] = v2;
  }
  for (int g = 0; g < 16; ++g) T.wt[g] = d1 * d2 * wt[g & 3] * wt[g >> 2];
  return T;
}

struct D3 { double x, y, z; };
__device__ __forceinline__ D3 operator+(D3 a, D3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ D3 operator-(D3 a, D3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ D3 operator*(double s, D3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ D3 cross(D3 a, D3 b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ __forceinline__ double from(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
__device__ __forceinline__ D3 from(D3 v, int lane) { return {from(v.x, lane), from(v.y, lane), from(v.z, lane)}; }

// DOF index (corner * 12 + kind * 3 + c) of the factor pair (a, b), component c
__device__ __forceinline__ int dof_of(int a, int b, int c) {
  return ((a >> 1) + 2 * (b >> 1)) * 12 + ((a & 1) + 2 * (b & 1)) * 3 + c;
}

struct WarpScratch {
  double q[2][48];        // rest and current DOFs; then the gradient's second contraction reads T
  double T[2][144];       // after the theta^1 contraction
  double G[16][15];       // gradient vectors per Gauss point
};

// St. Venant-Kirchhoff membrane + bending energy (thickness-integrated) and its gradient per
// generalised coordinate, one warp per patch. Bound by FP64 issue (a warp instruction per 64 cycles
// and sub-partition), so by the length of a warp's chain on small grids and by its operations on large
// ones: the interpolations and the gradient are sum-factorised over the tensor-product basis, lanes
// 0-15 form the geometry of the rest state at the 16 Gauss points while lanes 16-31 form the current
// one's with the same instructions, and each half then forms one of the two tangent directions'
// gradient vectors. About 350 FP64 instructions per patch and warp; with half a warp per patch, the
// shape table built by a kernel of its own and full 16 x 5 contractions it was 1,000 per two patches:
// 10 x 10 patches 74 us a call, now 24 us.
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
k_energy_grad(const __grid_constant__ Tables tab, int nu, int nv, int per_u, int per_v, const double* __restrict__ rest,
              const double* __restrict__ q, double lam, double mu, double h,
              double* __restrict__ grad, double* __restrict__ energy_out, Scratch* S) {
  __shared__ double w1[48], w2[48];
  __shared__ WarpScratch sw[WARPS];
  __shared__ double sred[WARPS];
  __shared__ int last;
  for (int e = threadIdx.x; e < 48; e += 32 * WARPS) {
    w1[e] = tab.w1[e];
    w2[e] = tab.w2[e];
  }
  __syncthreads();
  const int n1 = per_u ? nu : nu + 1, n2 = per_v ? nv : nv + 1;
  const int np = nu * nv;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, half = lane >> 4, g = lane & 15, g1 = g & 3, g2 = g >> 2;
  WarpScratch& W = sw[wid];
  const double wtg = tab.wt[g];
  double e_sum = 0.0;
  for (int p = blockIdx.x * WARPS + wid; p < np; p += gridDim.x * WARPS) {
    const int pu = p % nu, pv = p / nu;
    int nd[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) nd[c] = ((pv + (c >> 1)) % n2) * n1 + (pu + (c & 1)) % n1;
    for (int l = lane; l < 96; l += 32) {
      const int f = l / 48, k = l % 48, corner = k / 12;
      const int node = corner == 0 ? nd[0] : corner == 1 ? nd[1] : corner == 2 ? nd[2] : nd[3];
      // positions relative to corner 0: every shape-function derivative annihilates a translation, and
      // the sums then round at the patch's size instead of the sheet's
      const double* x = f ? q : rest;
      const double x0 = k % 12 < 3 ? x[(size_t)nd[0] * 12 + k % 12] : 0.0;
      W.q[f][k] = x[(size_t)node * 12 + k % 12] - x0;
    }
    __syncwarp();
    // theta^1: T[(d1 * 4 + gauss) * 12 + b * 3 + c] = sum_a w1[d1][gauss][a] Q[a][b][c]
    for (int e = lane; e < 288; e += 32) {
      const int f = e / 144, k = e % 144, c = k % 3, b = (k / 3) % 4, dg = k / 12;
      double t = 0.0;
#pragma unroll
      for (int a = 0; a < 4; ++a) t = __fma_rn(w1[dg * 4 + a], W.q[f][dof_of(a, b, c)], t);
      W.T[f][k] = t;
    }
    __syncwarp();
    // theta^2 at this lane's Gauss point and field: kinds (1,0), (0,1), (2,0), (0,2), (1,1)
    constexpr int kd1[5] = {1, 0, 2, 0, 1}, kd2[5] = {0, 1, 0, 2, 1};
    D3 v[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      D3 s{0.0, 0.0, 0.0};
      const double* T = W.T[half] + (kd1[k] * 4 + g1) * 12;
      const double* w = w2 + (kd2[k] * 4 + g2) * 4;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        s.x = __fma_rn(w[b], T[b * 3 + 0], s.x);
        s.y = __fma_rn(w[b], T[b * 3 + 1], s.y);
        s.z = __fma_rn(w[b], T[b * 3 + 2], s.z);
      }
      v[k] = s;
    }
    // fundamental forms of the lane's field
    D3 n = cross(v[0], v[1]);
    double nn = dot(n, n), isq = rsqrt(nn);
    D3 a3 = isq * n;
    double f1[3] = {dot(v[0], v[0]), dot(v[1], v[1]), dot(v[0], v[1])};
    double f2[3] = {dot(v[2], a3), dot(v[3], a3), dot(v[4], a3)};
    // rest forms from lane g, current geometry from lane 16 + g
    double ab[3], bb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ab[k] = from(f1[k], g);
      bb[k] = from(f2[k], g);
      f1[k] = from(f1[k], 16 + g);
      f2[k] = from(f2[k], 16 + g);
    }
    const double rn = from(nn, g), ri = from(isq, g);
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] = from(v[k], 16 + g);
    a3 = from(a3, 16 + g);
    isq = from(isq, 16 + g);
    // contravariant rest metric (det = |a_1 x a_2|^2), Voigt H
    const double idet = ri * ri, ai11 = ab[1] * idet, ai22 = ab[0] * idet, ai12 = -ab[2] * idet;
    const double lm = lam + 2 * mu;
    const double H00 = lm * ai11 * ai11, H01 = lam * ai11 * ai22 + 2 * mu * ai12 * ai12;
    const double H02 = lm * ai11 * ai12, H11 = lm * ai22 * ai22;
    const double H12 = lm * ai12 * ai22, H22 = (lam + mu) * ai12 * ai12 + mu * ai11 * ai22;
    const double wgt = wtg * (rn * ri);   // times sqrt(det)
    const double al[3] = {0.5 * (f1[0] - ab[0]), 0.5 * (f1[1] - ab[1]), f1[2] - ab[2]};
    const double be[3] = {f2[0] - bb[0], f2[1] - bb[1], 2.0 * (f2[2] - bb[2])};
    const double sg[3] = {H00 * al[0] + H01 * al[1] + H02 * al[2], H01 * al[0] + H11 * al[1] + H12 * al[2],
                          H02 * al[0] + H12 * al[1] + H22 * al[2]};
    const double mm[3] = {H00 * be[0] + H01 * be[1] + H02 * be[2], H01 * be[0] + H11 * be[1] + H12 * be[2],
                          H02 * be[0] + H12 * be[1] + H22 * be[2]};
    const double h3 = h * h * h, s = h3 * (1.0 / 12.0);
    const double en = wgt * (0.5 * h * (al[0] * sg[0] + al[1] * sg[1] + al[2] * sg[2]) +
                             0.5 * s * (be[0] * mm[0] + be[1] * mm[1] + be[2] * mm[2]));
    if (!half) e_sum += en;
    if (grad) {
      const D3 ct = mm[0] * v[2] + mm[1] * v[3] + (2.0 * mm[2]) * v[4];
      const double bt = dot(ct, a3);
      // half 0: direction 1 (with P = a_2), half 1: direction 2 (with P = a_1, other sign)
      const D3 P = half ? v[0] : v[1], own = half ? v[1] : v[0];
      const D3 ek = ((half ? -isq : isq) * s) * (cross(P, ct) - bt * cross(P, a3));
      const D3 Gk = wgt * (h * ((half ? sg[1] : sg[0]) * own + sg[2] * P) + ek);
      const double ws = wgt * s;
      const D3 Gb = (ws * (half ? mm[1] : mm[0])) * a3;
      const int k0 = half * 3, k2 = 6 + half * 3;
      W.G[g][k0] = Gk.x;
      W.G[g][k0 + 1] = Gk.y;
      W.G[g][k0 + 2] = Gk.z;
      W.G[g][k2] = Gb.x;
      W.G[g][k2 + 1] = Gb.y;
      W.G[g][k2 + 2] = Gb.z;
      if (!half) {
        const double w4 = ws * 2.0 * mm[2];
        W.G[g][12] = w4 * a3.x;
        W.G[g][13] = w4 * a3.y;
        W.G[g][14] = w4 * a3.z;
      }
      __syncwarp();
      // the contractions transposed: U[d1][gauss][b][c], then dE/dQ[a][b][c]
      double* U = W.T[0];
      for (int e2 = lane; e2 < 144; e2 += 32) {
        const int c = e2 % 3, b = (e2 / 3) % 4, gi = (e2 / 12) % 4, d1 = e2 / 48;
        const int ka = d1 == 0 ? 1 : d1 == 1 ? 0 : 2, da = d1 == 0 ? 1 : 0;
        const int kb = d1 == 0 ? 3 : 4, db = d1 == 0 ? 2 : 1;
        double u = 0.0;
#pragma unroll
        for (int gj = 0; gj < 4; ++gj) {
          u = __fma_rn(w2[(da * 4 + gj) * 4 + b], W.G[gj * 4 + gi][ka * 3 + c], u);
          if (d1 < 2) u = __fma_rn(w2[(db * 4 + gj) * 4 + b], W.G[gj * 4 + gi][kb * 3 + c], u);
        }
        U[e2] = u;
      }
      __syncwarp();
      for (int l = lane; l < 48; l += 32) {
        const int corner = l / 12, kind = (l / 3) % 4, c = l % 3;
        const int a = 2 * (corner & 1) + (kind & 1), b = 2 * (corner >> 1) + (kind >> 1);
        double t = 0.0;
#pragma unroll
        for (int dg = 0; dg < 12; ++dg) t = __fma_rn(w1[dg * 4 + a], U[(dg * 4 + b) * 3 + c], t);
        const int node = corner == 0 ? nd[0] : corner == 1 ? nd[1] : corner == 2 ? nd[2] : nd[3];
        atomicAdd(&grad[(size_t)node * 12 + kind * 3 + c], t);
      }
    }
    __syncwarp();   // W is rewritten by the next patch
  }
  // energy: CTA sum in a fixed order, then the last CTA sums the partials in CTA order
  for (int o = 16; o > 0; o >>= 1) e_sum += __shfl_xor_sync(0xffffffffu, e_sum, o);
  if (lane == 0) sred[wid] = e_sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = sred[0];
    for (int w = 1; w < WARPS; ++w) t += sred[w];
    S->partials[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(&S->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double t = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += 32 * WARPS) t += __ldcg(&S->partials[b]);
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) sred[wid] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = sred[0];
    for (int w = 1; w < WARPS; ++w) tot += sred[w];
    *energy_out = tot;
    S->ticket = 0u;
  }
}

// Device address of g_scratch, looked up once per device (with that device current) and kept for
// the life of the process; a cudaDeviceReset on that device invalidates it (documented in bhem.h).
static std::mutex g_mutex;
static Scratch* g_addr[128] = {nullptr};

static shell_status scratch_for_current_device(Scratch** out) {
  int dev = 0;
  BHEM_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 128) return fail(SHELL_ERR_ARG, "device index out of range");
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess || !p)
      return fail(SHELL_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    g_addr[dev] = reinterpret_cast<Scratch*>(p);
  }
  *out = g_addr[dev];
  return SHELL_OK;
}

}  // namespace noalloc
}  // namespace bhem

using namespace bhem;

extern "C" shell_status shell_energy_grad_noalloc(const shell_grid* grid, const shell_material* material,
                                                  const double* rest_dofs, const double* q,
                                                  double* energy, double* grad, void* stream) {
  using namespace bhem::noalloc;
  if (!grid || !material || !rest_dofs || !q || !energy) return fail(SHELL_ERR_ARG, "NULL argument");
  const shell_grid& g = *grid;
  if (g.nu < 1 || g.nv < 1 || (g.periodic_u && g.nu < 2) || (g.periodic_v && g.nv < 2) ||
      !(g.dxi1 > 0) || !(g.dxi2 > 0))
    return fail(SHELL_ERR_ARG, "invalid grid");
  const long long np = (long long)g.nu * g.nv;
  if (np > kMaxPatches)
    return fail(SHELL_ERR_ARG, "grid has " + std::to_string(np) + " patches; the allocation-free entry "
                               "point handles at most " + std::to_string(kMaxPatches));
  if (!(material->thickness > 0) || !(material->young > 0) ||
      !(material->poisson > -1.0 && material->poisson < 1.0))
    return fail(SHELL_ERR_ARG, "invalid material");
  Scratch* S = nullptr;
  BHEM_TRY(scratch_for_current_device(&S));
  cudaStream_t st = (cudaStream_t)stream;
  const long long n1 = g.periodic_u ? g.nu : g.nu + 1, n2 = g.periodic_v ? g.nv : g.nv + 1;
  BHEM_CUDA(cudaMemsetAsync(&S->ticket, 0, sizeof(unsigned), st));
  if (grad) BHEM_CUDA(cudaMemsetAsync(grad, 0, sizeof(double) * 12 * n1 * n2, st));
  const double lam = material->young * material->poisson / (1.0 - material->poisson * material->poisson);
  const double mu = material->young / (2.0 * (1.0 + material->poisson));
  const Tables tab = make_tables(g.dxi1, g.dxi2);
  if (np <= kSpreadPatches)
    k_energy_grad<1><<<(int)np, 32, 0, st>>>(tab, g.nu, g.nv, g.periodic_u, g.periodic_v, rest_dofs, q, lam, mu,
                                             material->thickness, grad, energy, S);
  else
    k_energy_grad<kWarps><<<(int)std::min<long long>((np + kWarps - 1) / kWarps, kMaxCtas), 32 * kWarps, 0, st>>>(
        tab, g.nu, g.nv, g.periodic_u, g.periodic_v, rest_dofs, q, lam, mu, material->thickness, grad, energy, S);
  BHEM_CUDA(cudaGetLastError());
  return SHELL_OK;
}
