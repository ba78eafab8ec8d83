// The linear solve of one Newton iteration (Sec. 6.1) on a shell small enough that its matrix fits
// in the SMs' shared memory: regulariser statistics and diagonal fix, block-Jacobi set-up, the PCG
// loop, and M d with the line search's dot products, in one cooperative launch.
//
// What bounds it: on small shells a PCG iteration of separate kernels is launch and memory latency
// (two kernels, 15 us an iteration at 961 and at 1,680 nodes in FP32, three and 28 us at 121 nodes in
// FP64), the statistics, the block inverses and the dot products are short latency-bound kernels with
// a host round trip each, and the matrix (5 MB at 961 nodes) is read from L2 every time. Here every SM
// keeps its rows' blocks, block-Jacobi inverses and vectors in shared memory and registers for the
// whole solve (6.6 KB per FP32 row; at most 32 rows per SM, 4,864 nodes on 152, or 17 in FP64), and
// an iteration is two exchanges between the CTAs: the two-way latency of L2, about 3 us each with the
// sums, and under 1.5 us of arithmetic. Measured per solve, statistics to dot products: 30 x 30
// patches (27 iterations) 556 -> 245 us, 280 x 5 (88) 1,480 -> 890 us, 64 x 64 (26) 640 -> 345 us,
// 10 x 10 in FP64 (41) 1,400 -> 470 us.
//
// Exchanges: a value travels as a 64-bit word {value, tag} (an FP64 value as two), written and read
// with single 64-bit accesses, so a reader that sees the expected tag has the value: no fence, no
// barrier counter, one L2 round trip. A reduction is one such partial per CTA, stored once for every
// reading CTA (so that each CTA polls cache lines of its own: with one shared set of slots the 152
// pollers of each line held up its writers, 4 to 7 us a reduction) and summed by every CTA in CTA
// order, so all CTAs hold the same totals and take the same decisions. Tags grow
// from exchange to exchange and from launch to launch (Shell::res_tag). A slot is rewritten only
// after a later reduction to which every reader of its old value has contributed, so no reader can
// miss a value: z of an iteration after the next p.q, which a CTA joins when it has received its
// neighbours' z. (Its part of r.z and r.r it sends before that, so when those sums end the loop z
// may still be on its way to a late CTA: the solution travels in words of its own.) Each wait polls at most Shell::wait_polls times; on expiry the CTA raises
// ERRBIT_TIMEOUT and leaves, and the others then expire too. The launch is cooperative, so all CTAs
// are resident.
//
// Arithmetic. FP32: that of the separate kernels on shells of these sizes (k_precond32_thread,
// k_spmv32_pcg, k_pcg32_update), operation by operation and in their order: Cholesky inverses, w =
// (A + tau D) z along a row's blocks, p = z + beta p and q = w + beta q on the own rows, alpha and beta
// as their FP64 quotients rounded to FP32. Only the double-float sums over the grid (48 bits) and the
// statistics' FP64 sums are taken in another order, so a solve has the separate kernels' bits unless
// one of its scalars lies that close to the middle of two FP32 numbers. (Sums over blocks in thirds,
// A p formed from p itself and Gauss-Jordan inverses moved 50 iterations by 5e-7 and a step to 1e-8 by
// 5e-9.) FP64: the p-update is applied by each CTA to its copies of the neighbours' p, a row is summed
// in nine pieces and the inverses are by Gauss-Jordan elimination; a step moves by 1e-14 with it.
#include <algorithm>

#include "common.cuh"

namespace bhem {

namespace {

constexpr int kRowBlocks = 9;          // blocks of a node row (a node couples to at most 9 nodes)
constexpr int kResSlotCtas = 160;      // slots per reduced value (>= CTAs, a multiple of 32)
constexpr int kResSlotWarps = kResSlotCtas / 32;
constexpr int kResThreads = 512;       // 128 registers each: the matrix pieces of a few rows fit beside the rest
constexpr int kRowsPerWarp = 2;        // rows whose DOFs a warp owns (12 lanes each)
constexpr int kResMaxRows = kRowsPerWarp * (kResThreads / 32);   // rows per CTA that have an owner
constexpr int kSlotPq = 0, kSlotRz = 1 /* r.z and r.r */, kSums = 3;   // values summed per PCG iteration

struct alignas(16) Word2 { unsigned long long a, b; };

__device__ __forceinline__ Word2 ld_word2(const Word2* p) {
  Word2 w;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];\n" : "=l"(w.a), "=l"(w.b) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void st_word2(Word2* p, Word2 w) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n" ::"l"(p), "l"(w.a), "l"(w.b) : "memory");
}
__device__ __forceinline__ unsigned long long tagged(unsigned bits, unsigned tag) {
  return ((unsigned long long)tag << 32) | bits;
}
// Sums: double-float for FP32 shells (as in the separate kernels), FP64 for FP64 shells.
template <typename R> struct Acc;
template <> struct Acc<float> {
  using T = F2;
  static __device__ __forceinline__ T zero() { return F2{0.f, 0.f}; }
  static __device__ __forceinline__ T prod(float a, float b) { return f2_prod(a, b); }
  static __device__ __forceinline__ T add(T a, T b) { return f2_add(a, b); }
  static __device__ __forceinline__ T xor_lane(T a, int o) {
    return F2{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
  }
  static __device__ __forceinline__ T lane0(T a) {
    return F2{__shfl_sync(0xffffffffu, a.hi, 0), __shfl_sync(0xffffffffu, a.lo, 0)};
  }
  static __device__ __forceinline__ double value(T a) { return (double)a.hi + (double)a.lo; }
  static __device__ __forceinline__ bool nonzero(T a) { return a.hi != 0.f || a.lo != 0.f; }
  static __device__ __forceinline__ bool positive(T a) { return a.hi > 0.f || (a.hi == 0.f && a.lo > 0.f); }
  // a / b as the separate kernels form it, the FP64 quotient rounded to FP32: an FP32 quotient q and
  // its correction d by the double-float remainder (the FP64 quotient is a chain of dependent FP64
  // operations on this GPU, about 900 cycles against 200). q + d is within a few 2^-46 of a / b (the
  // remainder is exact up to roundings of 2^-47 and d has 24 bits of at most 2^-23 q), so its rounding c
  // is that of the quotient unless q + d lies within 2^-40 of the middle between c and a neighbour,
  // or the operands leave the normal range: then the quotient is formed.
  static __device__ __forceinline__ float ratio(T a, T b) {
    const float q = __fdiv_rn(a.hi, b.hi);
    const F2 p = f2_prod(q, b.hi);
    const float rem = ((a.hi - p.hi) - p.lo) + __fmaf_rn(-q, b.lo, a.lo);
    const float d = __fdiv_rn(rem, b.hi);
    const float c = q + d, off = fabsf((q - c) + d), m = fabsf(c);
    const float below = 0.5f * (m - __int_as_float(__float_as_int(m) - 1));   // half the gaps to c's neighbours
    const float above = 0.5f * (__int_as_float(__float_as_int(m) + 1) - m);
    const float eps = 0x1p-40f * m;
    const bool sure = m > 0x1p-60f && m < 0x1p60f && fabsf(a.hi) > 0x1p-60f && fabsf(a.hi) < 0x1p60f &&
                      fabsf(b.hi) > 0x1p-60f && fabsf(b.hi) < 0x1p60f && fabsf(off - below) > eps &&
                      fabsf(off - above) > eps;
    return sure ? c : (float)(value(a) / value(b));
  }
  static __device__ __forceinline__ Word2 pack(T a, unsigned tag) {
    return Word2{tagged(__float_as_uint(a.hi), tag), tagged(__float_as_uint(a.lo), tag)};
  }
  static __device__ __forceinline__ T unpack(Word2 w) {
    return F2{__uint_as_float((unsigned)w.a), __uint_as_float((unsigned)w.b)};
  }
};
template <> struct Acc<double> {
  using T = double;
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T prod(double a, double b) { return a * b; }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ T xor_lane(T a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
  static __device__ __forceinline__ T lane0(T a) { return __shfl_sync(0xffffffffu, a, 0); }
  static __device__ __forceinline__ double value(T a) { return a; }
  static __device__ __forceinline__ bool nonzero(T a) { return a != 0.0; }
  static __device__ __forceinline__ bool positive(T a) { return a > 0.0; }
  static __device__ __forceinline__ double ratio(T a, T b) { return a / b; }
  static __device__ __forceinline__ Word2 pack(T a, unsigned tag) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(a);
    return Word2{tagged((unsigned)u, tag), tagged((unsigned)(u >> 32), tag)};
  }
  static __device__ __forceinline__ T unpack(Word2 w) {
    return __longlong_as_double((long long)((w.b << 32) | (w.a & 0xffffffffull)));
  }
};

// A node DOF in the exchanged vector: FP32 values two per Word2, FP64 values one per Word2.
template <typename R> constexpr int kDofWords = sizeof(R) / 4;   // 64-bit words per DOF

__device__ __forceinline__ void publish(unsigned long long* vec, size_t gi, float v, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;\n" ::"l"(vec + gi), "l"(tagged(__float_as_uint(v), tag)) : "memory");
}
__device__ __forceinline__ void publish(unsigned long long* vec, size_t gi, double v, unsigned tag) {
  st_word2(reinterpret_cast<Word2*>(vec) + gi, Acc<double>::pack(v, tag));
}
// DOFs gi .. gi + 3 (gi a multiple of 4); their loads are in flight together
template <int N>
__device__ __forceinline__ bool poll_words(const Word2* p, unsigned tag, int polls, Word2 (&w)[N]) {
  for (int i = 0; i < polls; ++i) {
#pragma unroll
    for (int k = 0; k < N; ++k) w[k] = ld_word2(p + k);
    bool all = true;
#pragma unroll
    for (int k = 0; k < N; ++k) all = all && (unsigned)(w[k].a >> 32) == tag && (unsigned)(w[k].b >> 32) == tag;
    if (all) return true;
  }
  return false;
}
__device__ __forceinline__ bool receive4(const unsigned long long* vec, size_t gi, unsigned tag, int polls, float v[4]) {
  Word2 w[2];
  const bool ok = poll_words(reinterpret_cast<const Word2*>(vec + gi), tag, polls, w);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    v[2 * k] = __uint_as_float((unsigned)w[k].a);
    v[2 * k + 1] = __uint_as_float((unsigned)w[k].b);
  }
  return ok;
}
__device__ __forceinline__ bool receive4(const unsigned long long* vec, size_t gi, unsigned tag, int polls, double v[4]) {
  Word2 w[4];
  const bool ok = poll_words(reinterpret_cast<const Word2*>(vec) + gi, tag, polls, w);
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = Acc<double>::unpack(w[k]);
  return ok;
}

__device__ __forceinline__ float fma_r(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_r(double a, double b, double c) { return __fma_rn(a, b, c); }

struct ResidentArgs {
  int n, per;                        // node rows, rows per CTA
  const int *rp, *col, *diag_block;
  void* val;                         // assembled matrix (its diagonal is fixed in place)
  const unsigned char* mask;
  const double* rhs;
  double rhs_sign;                   // the system's right-hand side is rhs_sign * rhs
  double tau, rtol2;
  int fixed, limit;
  int stats, fix, dots;              // take the diagonal statistics, apply the local fix, form M d and the dots
  NewtonScalars* ns;
  PcgState* st;
  double* x;                         // solution
  const double *mass, *gin;          // dots only
  double* Md;
  unsigned long long* vec;           // exchanged vector, kDofWords words per DOF
  unsigned long long* xvec;          // the same for the solution, written once per launch
  void* stat_records;                // [4][kResSlotCtas] KindStat of each CTA
  unsigned* stat_count;              // CTAs that have written theirs, over all launches
  unsigned stat_target;              // its value when those of this launch have
  Word2* slots;                      // [CTAs][kSums][kResSlotCtas] partial sums, by reader, value and writer
  double* partials;                  // [3][kResSlotCtas] dot products of each CTA
  unsigned* ticket;
  unsigned tag;                      // first tag of this launch
  int polls;
  int* err;
};

// First half of a sum over all CTAs: the warp's sums of NV values into swarp ([value][32]).
template <typename R, int NV>
__device__ __forceinline__ void warp_partials(typename Acc<R>::T (&v)[NV], typename Acc<R>::T* swarp) {
  using A = Acc<R>;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = A::add(v[i], A::xor_lane(v[i], o));
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int i = 0; i < NV; ++i) swarp[i * 32 + (threadIdx.x >> 5)] = v[i];
}

// Second half, by one warp: the CTA's sum of the first `warps` partials goes to every CTA's slots of
// this value, the CTAs' sums come back and are added in the same order everywhere. All lanes get it.
template <typename R>
__device__ __forceinline__ bool exchange_sum(const typename Acc<R>::T* partial, int warps, int value, Word2* slots,
                                             unsigned tag, int polls, typename Acc<R>::T& total) {
  using A = Acc<R>;
  const int lane = threadIdx.x & 31, G = gridDim.x;
  typename A::T s = lane < warps ? partial[lane] : A::zero();
  for (int o = warps > 16 ? 16 : warps > 8 ? 8 : warps > 4 ? 4 : warps > 2 ? 2 : 1; o > 0; o >>= 1)
    s = A::add(s, A::xor_lane(s, o));
  s = A::lane0(s);
  const Word2 mine = A::pack(s, tag);
  for (int b = lane; b < G; b += 32) st_word2(slots + ((size_t)b * kSums + value) * kResSlotCtas + blockIdx.x, mine);
  const Word2* in = slots + ((size_t)blockIdx.x * kSums + value) * kResSlotCtas + lane;
  Word2 w[kResSlotWarps];
  bool ok = false;
  for (int i = 0; i < polls && !ok; ++i) {   // the lane's slots in flight together
#pragma unroll
    for (int j = 0; j < kResSlotWarps; ++j)
      if (lane + 32 * j < G) w[j] = ld_word2(in + 32 * j);
    ok = true;
#pragma unroll
    for (int j = 0; j < kResSlotWarps; ++j)
      ok = ok && (lane + 32 * j >= G || ((unsigned)(w[j].a >> 32) == tag && (unsigned)(w[j].b >> 32) == tag));
  }
  total = lane < G ? A::unpack(w[0]) : A::zero();
#pragma unroll
  for (int j = 1; j < kResSlotWarps; ++j)
    if (lane + 32 * j < G) total = A::add(total, A::unpack(w[j]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) total = A::add(total, A::xor_lane(total, o));
  return __all_sync(0xffffffffu, ok);
}

__device__ __forceinline__ float min_r(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double min_r(double a, double b) { return fmin(a, b); }

// One CTA's diagonal statistics of a DOF kind over its free DOFs.
template <typename R> struct alignas(16) KindStat { double sum; R mn; int count; };

// Diagonal statistics (per DOF kind: sum |A_ii|, count, min A_ii over free DOFs) over all CTAs into
// stat12 (shared); each CTA's diagonal is in its copy of the matrix. The CTAs write their records,
// count themselves in on one counter (2,500 cycles for 152 CTAs) and read all records.
template <typename R>
__device__ bool all_stats(const ResidentArgs& P, const R* sA, const int* sdiag, int i0, int rows, double* stat12) {
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  KindStat<R>* all = reinterpret_cast<KindStat<R>*>(P.stat_records);   // [4][kResSlotCtas]
  __shared__ KindStat<R> part[4 * kResSlotWarps];
  bool ok = true;
  if (wid == 0) {   // 8 lanes per kind
    const int kind = lane >> 3, sub = lane & 7;
    KindStat<R> k{0.0, R(INFINITY), 0};
    for (int r = sub; r < rows; r += 8)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int d = 3 * kind + c;
        if (P.mask && P.mask[(size_t)(i0 + r) * 12 + d]) continue;
        const R v = sA[(size_t)(r * kRowBlocks + sdiag[r]) * 144 + d * 13];
        k.sum += fabs((double)v);
        k.mn = min_r(k.mn, v);
        ++k.count;
      }
    for (int o = 4; o > 0; o >>= 1) {
      k.sum += __shfl_xor_sync(0xffffffffu, k.sum, o);
      k.mn = min_r(k.mn, __shfl_xor_sync(0xffffffffu, k.mn, o));
      k.count += __shfl_xor_sync(0xffffffffu, k.count, o);
    }
    if (sub == 0) {
      all[kind * kResSlotCtas + blockIdx.x] = k;
      __threadfence();
    }
    __syncwarp();
    if (lane == 0) {
      ok = false;
      unsigned n;
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(P.stat_count) : "memory");
      for (int i = 0; i < P.polls && !ok; ++i) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(n) : "l"(P.stat_count) : "memory");
        ok = (int)(n - P.stat_target) >= 0;
      }
    }
  }
  if (__syncthreads_or(!ok)) return false;
  for (int k = t; k < 4 * kResSlotCtas; k += blockDim.x) {   // at least 10 warps
    const int b = k % kResSlotCtas;
    KindStat<R> v{0.0, R(INFINITY), 0};
    if (b < (int)gridDim.x) {
      const KindStat<R>* p = all + k;
      v.sum = __ldcg(&p->sum);
      v.mn = __ldcg(&p->mn);
      v.count = __ldcg(&p->count);
    }
    for (int o = 16; o > 0; o >>= 1) {
      v.sum += __shfl_xor_sync(0xffffffffu, v.sum, o);
      v.mn = min_r(v.mn, __shfl_xor_sync(0xffffffffu, v.mn, o));
    }
    v.count = __reduce_add_sync(0xffffffffu, v.count);
    if (lane == 0) part[k >> 5] = v;
  }
  __syncthreads();
  if (t < 4) {
    KindStat<R> v = part[t * kResSlotWarps];
    for (int j = 1; j < kResSlotWarps; ++j) {
      const KindStat<R> y = part[t * kResSlotWarps + j];
      v.sum += y.sum;
      v.mn = min_r(v.mn, y.mn);
      v.count += y.count;
    }
    stat12[3 * t] = v.sum;
    stat12[3 * t + 1] = (double)v.count;
    stat12[3 * t + 2] = (double)v.mn;
    if (blockIdx.x == 0)
      for (int j = 0; j < 3; ++j) P.ns->diag_stats[3 * t + j] = stat12[3 * t + j];
  }
  __syncthreads();
  return true;
}

// Row l of a node's 12 x 12 block in m becomes row l of its inverse (lanes 0-11 of each half warp; all 32
// lanes call it); false in every lane of the half when the block is not SPD (m is then void).
// By Cholesky, A = L L^T, W = L^{-1}, A^{-1} = W^T W: the operations of k_precond32_thread on every entry, in
// its order. Lane a holds row a of L, then column a of W.
__device__ __forceinline__ bool cholesky_inverse_row(float (&m)[12], int l) {
  bool spd = true;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const float piv = __shfl_sync(0xffffffffu, m[k], k, 16);
    if (!(piv > 0.f)) spd = false;
    const float r = sqrtf(piv);
    m[k] = l == k ? r : m[k] / r;
#pragma unroll
    for (int j = k + 1; j < 12; ++j)   // entries above the diagonal are never read
      m[j] = __fmaf_rn(-m[k], __shfl_sync(0xffffffffu, m[k], j, 16), m[j]);
  }
  float w[12];
#pragma unroll
  for (int r = 0; r < 12; ++r) {
    float u = r == l ? 1.f : 0.f;
#pragma unroll
    for (int k = 0; k < r; ++k) u = __fmaf_rn(-__shfl_sync(0xffffffffu, m[k], r, 16), w[k], u);   // w[k] = 0 for k < l
    w[r] = u / __shfl_sync(0xffffffffu, m[r], r, 16);
  }
#pragma unroll
  for (int b = 0; b < 12; ++b) {
    float s = 0.f;
#pragma unroll
    for (int k = b; k < 12; ++k) s = __fmaf_rn(w[k], __shfl_sync(0xffffffffu, w[k], b, 16), s);
    m[b] = s;
  }
  return spd;
}

// By Gauss-Jordan elimination without pivoting; its pivots are the squared pivots of a Cholesky
// factorisation.
__device__ __forceinline__ bool gauss_jordan_row(double (&m)[12], int l) {
  bool spd = true;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const double piv = __shfl_sync(0xffffffffu, m[k], k, 16);
    if (!(piv > 0.0)) spd = false;
    const double inv = 1.0 / piv, f = m[k];
    if (l == k) {   // the pivot row is scaled once, then broadcast
      m[k] = 1.0;
#pragma unroll
      for (int b = 0; b < 12; ++b) m[b] *= inv;
    }
#pragma unroll
    for (int b = 0; b < 12; ++b) {
      const double rk = __shfl_sync(0xffffffffu, m[b], k, 16);
      if (l != k) m[b] = b == k ? -f * rk : __fma_rn(-f, rk, m[b]);
    }
  }
  return spd;
}

// How a row's product is shared out. A piece covers 4 entries of one matrix row in each of kBlocks blocks:
// FP32 all nine, one chain of products as in k_spmv32_pcg (36 pieces per row); FP64 three (108 pieces).
// Piece e of a CTA is piece e % kPieces of row e / kPieces; its matrix row's kSums sums lie side by side.
template <typename R> struct Product {
  static constexpr int kBlocks = sizeof(R) == 4 ? kRowBlocks : 3;
  static constexpr int kEntries = 4 * kBlocks;
  static constexpr int kSums = 3 * kRowBlocks / kBlocks;
  static constexpr int kPieces = 12 * kSums;
};
// first block, matrix row and first column of piece w of a row
template <typename R> __device__ __forceinline__ int3 piece_of(int w) {
  using P = Product<R>;
  return make_int3(w % P::kSums / 3 * P::kBlocks, w / P::kSums, w % 3 * 4);
}

template <typename R>
__host__ __device__ constexpr size_t resident_row_bytes() {
  // matrix, block-Jacobi inverse, staged vector of the row's columns, partial sums of the product
  return sizeof(R) * (kRowBlocks * 144 + 144 + kRowBlocks * 12 + 12 * Product<R>::kSums + 12) + sizeof(int) * (kRowBlocks + 1);
}

// A row's product is Product<R>::kPieces pieces, of which a thread has up to PASSES, in registers for the
// whole loop; PASSES 0: read from shared memory. Of the neighbours' exchanged values (27 pieces of 4
// DOFs per row) a thread of warps 2 and up has up to PIECES.
template <typename R, int PASSES, int PIECES>
__global__ void __launch_bounds__(kResThreads, 1) k_solve_resident(ResidentArgs P) {
  using A = Acc<R>;
  using AT = typename A::T;
  extern __shared__ __align__(16) unsigned char sraw[];
  R* sA = reinterpret_cast<R*>(sraw);                      // [per][9][12][12]
  R* sD = sA + (size_t)P.per * kRowBlocks * 144;           // [per][12][12]
  R* sx = sD + (size_t)P.per * 144;                        // [per][9][12] z (FP64: p) of each block's column
  R* sacc = sx + (size_t)P.per * kRowBlocks * 12;          // [per][12][kSums]
  R* sr = sacc + (size_t)P.per * 12 * Product<R>::kSums;   // [per][12]
  int* scol = reinterpret_cast<int*>(sr + (size_t)P.per * 12);   // [per][9]
  int* sdiag = scol + P.per * kRowBlocks;                  // [per] slot of the diagonal block
  __shared__ double swarp_d[96];                           // warp partials of up to three sums
  __shared__ double s_stat[12];
  __shared__ R s_td[4], s_floor[4], s_scal;
  __shared__ int s_flag, s_stop, s_fail;
  AT* swarp = reinterpret_cast<AT*>(swarp_d);
  constexpr int nt = kResThreads;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int i0 = blockIdx.x * P.per, rows = min(P.per, P.n - i0);
  R* val = reinterpret_cast<R*>(P.val);
  if (t == 0) s_fail = 0;

  // ---- the CTA's rows: columns and blocks (absent blocks are zero)
  for (int e = t; e < rows * kRowBlocks; e += nt) {
    const int row = e / kRowBlocks, u = e % kRowBlocks, k = P.rp[i0 + row] + u;
    scol[e] = k < P.rp[i0 + row + 1] ? P.col[k] : -1;
    if (u == 0) sdiag[row] = P.diag_block[i0 + row] - k;
  }
  constexpr int kVec = 16 / sizeof(R), kBlockVecs = 144 / kVec;
  for (int e = t; e < rows * kRowBlocks * kBlockVecs; e += nt) {
    const int b = e / kBlockVecs, w = e % kBlockVecs, row = b / kRowBlocks, u = b % kRowBlocks;
    const int k = P.rp[i0 + row] + u;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < P.rp[i0 + row + 1]) v = __ldcg(reinterpret_cast<const float4*>(val + (size_t)k * 144) + w);
    reinterpret_cast<float4*>(sA + (size_t)b * 144)[w] = v;
  }
  for (int e = t; e < rows * kRowBlocks * 12; e += nt) sx[e] = R(0);
  __syncthreads();

  // ---- regulariser: kind statistics, shift tau D_k, local fix of the diagonal (Sec. 6.1)
  if (P.stats) {
    if (!all_stats<R>(P, sA, sdiag, i0, rows, s_stat)) {
      if (t == 0) atomicOr(P.err, ERRBIT_TIMEOUT);
      return;
    }
  } else {
    if (t < 12) s_stat[t] = P.ns->diag_stats[t];
    __syncthreads();
  }
  if (t < 4) {
    const double cnt = s_stat[3 * t + 1], dbar = cnt > 0.0 ? s_stat[3 * t] / cnt : 1.0;
    s_td[t] = (R)(P.tau * dbar);
    s_floor[t] = (R)(1e-8 * dbar);
  }
  if (t == 0) {
    bool any = false;
    for (int q = 0; q < 4; ++q) any = any || (s_stat[3 * q + 1] > 0.0 && s_stat[3 * q + 2] <= 0.0);
    s_flag = any;
  }
  __syncthreads();
  // a DOF of the CTA's rows per thread, two rows per warp (lanes 0-11, 12-23): a row's 12 values are
  // exchanged within the warp
  const int myrow = kRowsPerWarp * wid + lane / 12, a = lane % 12;
  const bool own = lane < 12 * kRowsPerWarp && myrow < rows;
  const int own_warps = (rows + kRowsPerWarp - 1) / kRowsPerWarp;
  const size_t gi = (size_t)(i0 + myrow) * 12 + a;
  const bool fixed_dof = own && P.mask && P.mask[gi];
  if (P.fix && s_flag) {
    if (own && !fixed_dof) {
      R* d = sA + (size_t)(myrow * kRowBlocks + sdiag[myrow]) * 144 + a * 13;
      const R v = *d;
      if (v <= R(0)) {
        const R f = s_floor[a / 3], w = -v > f ? -v : f;
        *d = w;
        val[(size_t)P.diag_block[i0 + myrow] * 144 + a * 13] = w;
        atomicAdd(&P.ns->diag_fixes, 1);
      }
    }
    __syncthreads();
  }

  // ---- block-Jacobi: (A_ii masked + tau D)^{-1}, one row per lane, two nodes per warp. A block that is
  // not SPD falls back to the inverse of its diagonal.
  for (int base = wid * 2; base < rows; base += (nt >> 5) * 2) {
    const int l = lane & 15, row = base + (lane >> 4);
    const bool act = row < rows && l < 12;
    R m[12];
    R dg = R(1);
    const bool fa = act && P.mask && P.mask[(size_t)(i0 + row) * 12 + l];
#pragma unroll
    for (int b = 0; b < 12; ++b) {
      R v = (l == b) ? R(1) : R(0);
      if (act && !fa && !(P.mask && P.mask[(size_t)(i0 + row) * 12 + b])) {
        v = sA[(size_t)(row * kRowBlocks + sdiag[row]) * 144 + l * 12 + b];
        if (l == b) v += s_td[b / 3];
      }
      m[b] = v;
      if (l == b) dg = v;
    }
    bool spd = true;
    if constexpr (sizeof(R) == 4) spd = cholesky_inverse_row(m, l);
    else spd = gauss_jordan_row(m, l);
    if (act) {
      if (!spd) {
#pragma unroll
        for (int b = 0; b < 12; ++b) m[b] = (l == b) ? (dg > R(0) ? R(1) / dg : R(1)) : R(0);
      }
#pragma unroll
      for (int b = 0; b < 12; ++b) sD[(size_t)row * 144 + l * 12 + b] = m[b];
    }
    __syncwarp();
    if constexpr (sizeof(R) == 8) {   // exactly symmetric: the mean of the two triangles
      if (act) {
#pragma unroll
        for (int b = 0; b < 12; ++b) m[b] = R(0.5) * (m[b] + sD[(size_t)row * 144 + b * 12 + l]);
      }
      __syncwarp();
      if (act) {
#pragma unroll
        for (int b = 0; b < 12; ++b) sD[(size_t)row * 144 + l * 12 + b] = m[b];
      }
    }
  }

  // this thread's pieces of the products
  using PR = Product<R>;
  R areg[PASSES > 0 ? PASSES : 1][PR::kEntries];
  int xoff[PASSES > 0 ? PASSES : 1];   // the piece's entries of the staged vector; its sum goes to sacc[t + s nt]
  if (PASSES > 0) {
#pragma unroll
    for (int s = 0; s < PASSES; ++s) {
      const int e = t + s * nt, row = e / PR::kPieces;
      const int3 w = piece_of<R>(e % PR::kPieces);
      xoff[s] = row < rows ? (row * kRowBlocks + w.x) * 12 + w.z : 0;
#pragma unroll
      for (int k = 0; k < PR::kEntries; ++k)
        areg[s][k] = row < rows ? sA[(size_t)(row * kRowBlocks + w.x + k / 4) * 144 + w.y * 12 + w.z + k % 4] : R(0);
    }
  }
  // this thread's pieces of the neighbours' vectors: z as received, p (FP64), and the first DOF (-1: none)
  R zn[PIECES][4] = {}, pn[PIECES][4] = {};
  int piece_gi[PIECES];
#pragma unroll
  for (int s = 0; s < PIECES; ++s) {
    const int e = t - 64 + s * (nt - 64);
    const int j = t >= 64 && e < rows * 27 ? scol[e / 3] : -1;
    piece_gi[s] = j < 0 ? -1 : j * 12 + (e % 3) * 4;
  }
  auto receive_pieces = [&](const unsigned long long* vec, unsigned tag) -> bool {
    bool ok = true;
#pragma unroll
    for (int s = 0; s < PIECES; ++s)
      if (piece_gi[s] >= 0) ok = receive4(vec, piece_gi[s], tag, P.polls, zn[s]) && ok;
    return ok;
  };

  // ---- start: x = 0, r = rhs, z = D r
  R xv = R(0), rv = R(0), zv = R(0), pv = R(0), qv = R(0);
  AT rz = A::zero(), pq = A::zero();   // warp 0
  double rr = 0.0, bb = 0.0;           // thread 32
  int iters = 0, negcurv = 0, done = 0;
  // z = D r of the own DOFs, sent to the neighbours, and the sums r.z and r.r over all CTAs, while
  // the warps that need no sum receive the neighbours' z; then beta, the stopping test
  auto precond_and_sums = [&](unsigned tag, bool first) -> bool {
    if (own) sr[myrow * 12 + a] = rv;
    __syncwarp();
    if (own) {
      const R* D = sD + (size_t)myrow * 144 + a * 12;
      const R* q = sr + myrow * 12;
      zv = R(0);
      if (!fixed_dof) {
        zv = D[0] * q[0];
#pragma unroll
        for (int c = 1; c < 12; ++c) zv = fma_r(D[c], q[c], zv);
      }
      publish(P.vec, gi, zv, tag);
    }
    if (wid < own_warps) {
      AT v[2] = {A::prod(rv, zv), A::prod(rv, rv)};
      warp_partials<R, 2>(v, swarp);
    }
    __syncthreads();
    bool ok = true;
    if (wid < 2) {
      AT tot;
      ok = exchange_sum<R>(swarp + wid * 32, own_warps, kSlotRz + wid, P.slots, tag, P.polls, tot);
      if (t == 0) {
        s_scal = first ? R(0) : A::ratio(tot, rz);   // beta
        rz = tot;
        s_flag = (!first && !A::nonzero(tot)) || iters >= P.limit;
      }
      if (t == 32) {
        rr = A::value(tot);
        if (first) bb = rr;
        s_stop = first ? bb == 0.0 : (P.fixed == 0 && rr <= P.rtol2 * bb);
      }
    } else {
      ok = receive_pieces(P.vec, tag);
    }
    if (!ok) s_fail = 1;
    __syncthreads();
    done = s_flag | s_stop;
    return !s_fail;
  };
  if (own) rv = fixed_dof ? R(0) : (R)(P.rhs_sign * P.rhs[gi]);
  if (!precond_and_sums(P.tag + 1, true)) {
    if (t == 0) atomicOr(P.err, ERRBIT_TIMEOUT);
    return;
  }

  // ---- PCG
  while (!done) {
    // z (FP64: p = z + beta p) of every block's column
    const R beta = s_scal;
#pragma unroll
    for (int s = 0; s < PIECES; ++s)
      if (piece_gi[s] >= 0) {
        R* x = sx + (t - 64 + s * (nt - 64)) * 4;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if constexpr (sizeof(R) == 8) x[k] = pn[s][k] = fma_r(beta, pn[s][k], zn[s][k]);
          else x[k] = zn[s][k];
        }
      }
    __syncthreads();
    if (PASSES > 0) {
#pragma unroll
      for (int s = 0; s < PASSES; ++s) {
        const int e = t + s * nt;
        const R* x = sx + xoff[s];
        R acc = R(0);
#pragma unroll
        for (int k = 0; k < PR::kEntries; ++k) acc = fma_r(areg[s][k], x[(k / 4) * 12 + k % 4], acc);
        if (e < rows * PR::kPieces) sacc[e] = acc;
      }
    } else {
      for (int e = t; e < rows * PR::kPieces; e += nt) {
        const int row = e / PR::kPieces;
        const int3 w = piece_of<R>(e % PR::kPieces);
        const R* m = sA + (size_t)(row * kRowBlocks + w.x) * 144 + w.y * 12 + w.z;
        const R* x = sx + (row * kRowBlocks + w.x) * 12 + w.z;
        R acc = R(0);
#pragma unroll
        for (int k = 0; k < PR::kEntries; ++k) acc = fma_r(m[(k / 4) * 144 + k % 4], x[(k / 4) * 12 + k % 4], acc);
        sacc[e] = acc;
      }
    }
    __syncthreads();
    if (wid < own_warps) {
      AT v[1] = {A::zero()};
      if (own) {
        const R* s = sacc + (size_t)(myrow * 12 + a) * PR::kSums;
        if constexpr (sizeof(R) == 8) {
          R y = (((s[0] + s[1]) + s[2]) + ((s[3] + s[4]) + s[5])) + ((s[6] + s[7]) + s[8]);
          pv = sx[(myrow * kRowBlocks + sdiag[myrow]) * 12 + a];
          y = fma_r(s_td[a / 3], pv, y);
          qv = fixed_dof ? R(0) : y;
        } else {   // w = (A + tau D) z, p = z + beta p, q = w + beta q (= A p by linearity)
          R w = (s[0] + s[1]) + s[2];
          w = fma_r(s_td[a / 3], zv, w);
          if (fixed_dof) w = R(0);
          pv = fma_r(beta, pv, zv);
          qv = fma_r(beta, qv, w);
        }
        v[0] = A::prod(pv, qv);
      }
      warp_partials<R, 1>(v, swarp);
    }
    __syncthreads();
    if (wid == 0) {
      const bool ok = exchange_sum<R>(swarp, own_warps, kSlotPq, P.slots, P.tag + 2 + iters, P.polls, pq);
      if (t == 0) {
        const bool neg = !A::positive(pq);
        s_scal = neg ? R(0) : A::ratio(rz, pq);   // alpha
        s_flag = neg;
        if (!ok) s_fail = 1;
      }
    }
    __syncthreads();
    if (s_fail) {
      if (t == 0) atomicOr(P.err, ERRBIT_TIMEOUT);
      return;
    }
    if (s_flag) {
      negcurv = 1;
      break;
    }
    const R alpha = s_scal;
    xv = fma_r(alpha, pv, xv);
    rv = fma_r(-alpha, qv, rv);
    ++iters;
    if (!precond_and_sums(P.tag + 1 + iters, false)) {
      if (t == 0) atomicOr(P.err, ERRBIT_TIMEOUT);
      return;
    }
  }

  // ---- results
  if (own) P.x[gi] = (double)xv;
  if (blockIdx.x == 0 && t == 0) {
    P.st->iters = iters;
    P.st->rz = A::value(rz);
    P.st->pq = A::value(pq);
    P.st->negcurv = negcurv;
    P.st->done = 1;
  }
  if (blockIdx.x == 0 && t == 32) {
    P.st->rr = rr;
    P.st->bb = bb;
  }
  if (!P.dots || negcurv) return;
  // M d on the own rows and d.Md, d.gin, g.d (rhs = -g) for the line search, in FP64
  const unsigned tagx = P.tag + (unsigned)max(P.limit, 0) + 3u;
  if (own) publish(P.xvec, gi, xv, tagx);
  bool ok = true;
  if (wid >= 2) ok = receive_pieces(P.xvec, tagx);
#pragma unroll
  for (int s = 0; s < PIECES; ++s)
    if (piece_gi[s] >= 0) {
      R* x = sx + (t - 64 + s * (nt - 64)) * 4;
#pragma unroll
      for (int k = 0; k < 4; ++k) x[k] = zn[s][k];
    }
  if (__syncthreads_or(!ok)) {
    if (t == 0) atomicOr(P.err, ERRBIT_TIMEOUT);
    return;
  }
  double v3[3] = {0.0, 0.0, 0.0};
  if (own) {
    const int r = a / 3, c = a % 3, k0 = P.rp[i0 + myrow];
    double s = 0.0;
    for (int u = 0; u < kRowBlocks && scol[myrow * kRowBlocks + u] >= 0; ++u) {
      const double* mb = P.mass + (size_t)(k0 + u) * 16 + r * 4;
      const R* d = sx + (myrow * kRowBlocks + u) * 12 + c;
#pragma unroll
      for (int q = 0; q < 4; ++q) s += mb[q] * (double)d[q * 3];
    }
    P.Md[gi] = s;
    const double d = (double)xv;
    v3[0] = d * s;
    v3[1] = d * P.gin[gi];
    v3[2] = d * (-P.rhs_sign < 0.0 ? -P.rhs[gi] : P.rhs[gi]);
  }
  if (wid < own_warps) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      for (int o = 16; o > 0; o >>= 1) v3[i] += __shfl_xor_sync(0xffffffffu, v3[i], o);
      if (lane == 0) swarp_d[i * 32 + wid] = v3[i];
    }
  }
  __syncthreads();
  if (wid < 3) {
    double s = lane < own_warps ? swarp_d[wid * 32 + lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      P.partials[wid * kResSlotCtas + blockIdx.x] = s;
      __threadfence();
    }
  }
  __syncthreads();
  if (t == 0) s_flag = atomicAdd(P.ticket, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!s_flag) return;
  __threadfence();
  if (wid < 3) {   // the last CTA: the CTAs' sums in one order
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < kResSlotWarps; ++j)
      if (lane + 32 * j < (int)gridDim.x) s += __ldcg(P.partials + wid * kResSlotCtas + lane + 32 * j);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) P.ns->dots[wid] = s;
  }
  if (t == 0) *P.ticket = 0u;
}

size_t resident_slot_bytes(int ctas) {
  return sizeof(Word2) * kResSlotCtas * kSums * ctas;
}

// the exchanged vectors: z and the solution
size_t resident_vec_bytes(const Shell& s) {
  return 2 * sizeof(unsigned long long) * (s.val_fp64 ? kDofWords<double> : kDofWords<float>) * (size_t)s.n_dof;
}

// the statistics' records, the dot products' partials, two counters
size_t resident_tail_bytes() {
  return sizeof(KindStat<double>) * 4 * kResSlotCtas + sizeof(double) * 3 * kResSlotCtas + sizeof(unsigned) * 4;
}

using ResidentKernel = void (*)(ResidentArgs);

// The kernel for `per` rows per CTA: passes of 512 threads over a row's pieces of the product (36 in FP32,
// 108 in FP64), pieces of 448 threads over 27 per row. FP32 holds two passes of the matrix in registers
// (72), FP64 two (24 FP64 values).
template <typename R> ResidentKernel resident_kernel(int per);
template <> ResidentKernel resident_kernel<float>(int per) {
  if (per <= 14) return k_solve_resident<float, 1, 1>;
  if (per <= 28) return k_solve_resident<float, 2, 2>;
  return k_solve_resident<float, 0, 2>;
}
template <> ResidentKernel resident_kernel<double>(int per) {
  if (per <= 9) return k_solve_resident<double, 2, 1>;
  return k_solve_resident<double, 0, 2>;
}
static_assert(27 * kResMaxRows <= 2 * (kResThreads - 64), "the last forms' PIECES cover every row accepted");

// Rows per CTA. An exchange grows with the CTAs (alone: 2,500 cycles for 64, 3,500 for 152), a CTA's
// products with its rows, so FP32 takes at least 9 rows per CTA (30 x 30 nodes' solve of 27
// iterations: 266 us with 7 rows, 244 with 9, 280 with 18; 1,680 nodes, 88 iterations: 890 us with
// 12 rows, 960 with 28) and FP64 at least 2 (121 nodes, 41 iterations: 488 us with 1, 470 with 2, 478
// with 4).
template <typename R>
int resident_rows(int n, int sms) {
  const int least = (n + sms - 1) / sms;
  if (sizeof(R) == 8) return std::max(least, 2);
  return least <= 9 ? 9 : least;
}

template <typename R>
shell_status resident_setup(Shell& s) {
  int coop = 0, optin = 0, occ = 0;
  BHEM_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, s.device));
  BHEM_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, s.device));
  const int sms = std::min(s.num_sms, kResSlotCtas);
  if (!coop || sms < 1 || s.max_row > kRowBlocks) return SHELL_OK;
  const int per = resident_rows<R>(s.n_nodes, sms);
  const ResidentKernel k = resident_kernel<R>(per);
  cudaFuncAttributes fa;
  BHEM_CUDA(cudaFuncGetAttributes(&fa, (const void*)k));
  const size_t smem = per * resident_row_bytes<R>();
  if (smem + fa.sharedSizeBytes > (size_t)optin || per > kResMaxRows) return SHELL_OK;
  BHEM_CUDA(cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes));
  BHEM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)k, kResThreads, smem));
  const int ctas = (s.n_nodes + per - 1) / per;
  if (occ < 1 || ctas > sms) return SHELL_OK;
  const size_t bytes = resident_slot_bytes(ctas) + resident_vec_bytes(s) + resident_tail_bytes();
  if (cudaMalloc(&s.d_resident, bytes) != cudaSuccess) {
    cudaGetLastError();
    s.d_resident = nullptr;
    return fail(SHELL_ERR_OOM, "cudaMalloc: resident solve");
  }
  s.res_per = per;
  return SHELL_OK;
}

}  // namespace

// Mixed precision or FP64 shells whose rows fit one CTA per SM (FP32: kResMaxRows per SM, FP64: 17);
// only where the caller has not selected another form of the solve (shell_options.spmv,
// BHEM_PCG_LOOP, BHEM_PCG_HOST_LOOP, BHEM_PCG_PUPDATE).
shell_status setup_resident(Shell& s) {
  return s.val_fp64 ? resident_setup<double>(s) : resident_setup<float>(s);
}

shell_status launch_solve_resident(Shell& s, const unsigned char* mask, const double* rhs, double rhs_sign, double tau,
                                   double rtol, int fixed, int limit, bool stats, bool fix, bool dots, double* x,
                                   bool* launched) {
  const int ctas = (s.n_nodes + s.res_per - 1) / s.res_per;
  const size_t slot_bytes = resident_slot_bytes(ctas);
  const size_t vec_bytes = resident_vec_bytes(s);
  const unsigned used = (unsigned)std::max(limit, 0) + 8u;
  if (s.res_reset || s.res_tag > 0xffffffffu - used) {   // first use, after an error, or the tags wrap
    BHEM_CUDA(cudaMemsetAsync(s.d_resident, 0, slot_bytes + vec_bytes + resident_tail_bytes(), s.stream));
    s.res_tag = 1;
    s.res_stat_count = 0;
    s.res_reset = false;
  }
  ResidentArgs P{};
  P.n = s.n_nodes;
  P.per = s.res_per;
  P.rp = s.d_row_ptr;
  P.col = s.d_col;
  P.diag_block = s.d_diag_block;
  P.val = s.d_val;
  P.mask = mask;
  P.rhs = rhs;
  P.rhs_sign = rhs_sign;
  P.tau = tau;
  P.rtol2 = fixed > 0 ? 0.0 : rtol * rtol;
  P.fixed = fixed;
  P.limit = limit;
  P.stats = stats;
  P.fix = fix;
  P.dots = dots;
  P.ns = s.d_ns;
  P.st = s.d_pcg;
  P.x = x;
  P.mass = s.d_mass;
  P.gin = s.d_gin;
  P.Md = s.d_Md;
  char* base = (char*)s.d_resident;
  P.slots = (Word2*)base;
  P.vec = (unsigned long long*)(base + slot_bytes);
  P.xvec = (unsigned long long*)(base + slot_bytes + vec_bytes / 2);
  P.stat_records = base + slot_bytes + vec_bytes;
  P.partials = (double*)(base + slot_bytes + vec_bytes + sizeof(KindStat<double>) * 4 * kResSlotCtas);
  P.ticket = (unsigned*)(P.partials + 3 * kResSlotCtas);
  P.stat_count = P.ticket + 1;
  P.stat_target = s.res_stat_count + (unsigned)ctas;
  P.tag = s.res_tag;
  P.polls = s.wait_polls;
  P.err = s.d_err;
  void* args[] = {(void*)&P};
  const size_t smem = s.res_per * (s.val_fp64 ? resident_row_bytes<double>() : resident_row_bytes<float>());
  const void* k = s.val_fp64 ? (const void*)resident_kernel<double>(s.res_per) : (const void*)resident_kernel<float>(s.res_per);
  const cudaError_t e =
      cudaLaunchCooperativeKernel(k, dim3(ctas), dim3(kResThreads), args, smem, s.stream);
  *launched = e == cudaSuccess;
  if (e == cudaErrorCooperativeLaunchTooLarge) {   // fewer SMs than the device has (a partition): the general path
    cudaGetLastError();
    s.res_per = 0;
    return SHELL_OK;
  }
  BHEM_CUDA(e);
  s.res_tag += used;
  if (stats) s.res_stat_count += (unsigned)ctas;
  ++s.launches;
  return SHELL_OK;
}

}  // namespace bhem
