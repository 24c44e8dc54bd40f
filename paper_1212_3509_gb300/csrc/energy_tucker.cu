// Demag energy of a Tucker magnetization from its potential in Tucker form,
// without forming a full tensor (Alg. 2 and the energy study after it).
//
// m^(q) = [[G^(q); V^(q,1), V^(q,2), V^(q,3)]] (Eq. tucker_rep) and
// phi = sum_t w_t [[C_t; W_t1, W_t2, W_t3]]: either the terms (k, q') of the
// Tucker application (core G^(q'), factors T_{k,q',p} V^(q',p), weight
// c s omega_k; Eq. kron_eval_tuck) or one Tucker tensor (the approximate sum
// of Alg. 2).  The stray field is -D phi with the second-order stencils of
// energy.cu; along axis q the difference acts on the factors of that axis
// only, so with W'_tp = D_q W_tp (p = q) or W_tp (p != q)
//   E = 1/2 h1 h2 h3 sum_q sum_t w_t < m^(q), [[C_t; W'_t1, W'_t2, W'_t3]] >.
// The inner product of two Tucker tensors contracts the cores through the
// factor Grams M_p = V^(q,p)^T W'_tp:
//   <[[G; V]], [[C; W']]> = sum_{a,b} G[a] C[b] prod_p M_p[a_p][b_p].
// One block per (term, component): the Grams in shared memory, the core
// contraction mode by mode in FP64 (intermediates in shared memory, or in a
// global workspace at large ranks); the per-block values are summed in a fixed
// order.
#include <type_traits>

#include "internal.h"

namespace demag {

constexpr int kEnMaxRank = 64;
constexpr int kEnWarps = 8;
constexpr size_t kEnSmemMax = 200 * 1024;  // largest dynamic request (Grams, and the contraction where it fits)

__device__ __forceinline__ double en_warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename F>
struct EnTuckerT {
  int n[3];
  double inv2h[3];   // 1 / (2 h_p)
  int r[3];          // multilinear ranks of m
  const F* G;        // [3][r3][r2][r1]
  const F* V;        // blocks (q, p), each [r_p][n_p]
  int s[3];          // ranks of every phi term
  const F* C;        // term cores [s3][s2][s1]: C + (core_by_q ? t % 3 : 0) * s1 s2 s3
  int core_by_q;
  const F* W[3];     // term t, mode p: rows W[p] + t * s_p * n_p
  const F* w;        // term weights (NULL: 1)
  int T;             // number of terms
  double* ws;        // per block r1 s3 (s2 + r2) doubles; NULL: behind the Grams in shared memory
  double* part;      // [T][3]
};
using EnTucker = EnTuckerT<float>;

// 2 h (D w)[i] of one factor row at an end, in FP64 (3-point one-sided, two-point for n = 2, zero for
// n = 1); between the ends it is w[i + 1] - w[i - 1], one rounding
template <typename F>
__device__ __forceinline__ F fd_end(const F* w, int i, int n) {
  if (n == 1) return F(0);
  if (n == 2) return (F)(2.0 * ((double)w[1] - (double)w[0]));
  if (i == 0) return (F)(-3.0 * (double)w[0] + 4.0 * (double)w[1] - (double)w[2]);
  return (F)(3.0 * (double)w[n - 1] - 4.0 * (double)w[n - 2] + (double)w[n - 3]);
}

// An unevaluated sum hi + lo: FP32 values added without loss on the FP32 pipe
// (Knuth's two-sum), where an FP64 addition would take 64 times as long; FP64
// values as they are.
template <typename F> struct EnSum;
template <> struct EnSum<float> {
  float hi, lo;
  __device__ __forceinline__ void set(float v) { hi = v; lo = 0.f; }
  __device__ __forceinline__ void add(float h, float l) {
    const float s = __fadd_rn(hi, h), bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h, bb));
    hi = s;
    lo = __fadd_rn(__fadd_rn(lo, l), e);
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
template <> struct EnSum<double> {
  double hi, lo;
  __device__ __forceinline__ void set(double v) { hi = v; lo = 0.0; }
  __device__ __forceinline__ void add(double h, double) { hi += h; }
  __device__ __forceinline__ double value() const { return hi; }
};

// One step of the transposing reduction: of C sums, a lane keeps the half that
// its bit `off` selects and adds its partner's values of them.
template <int C, typename F>
__device__ __forceinline__ void en_halve(EnSum<F>* v, int off) {
  const bool up = (threadIdx.x & off) != 0;
#pragma unroll
  for (int j = 0; j < C / 2; ++j) {
    const EnSum<F> give = up ? v[j] : v[j + C / 2];
    EnSum<F> keep = up ? v[j + C / 2] : v[j];
    const F h = __shfl_xor_sync(0xffffffffu, give.hi, off);
    F l = F(0);
    if constexpr (C < 64 && std::is_same<F, float>::value) l = __shfl_xor_sync(0xffffffffu, give.lo, off);
    keep.add(h, l);
    v[j] = keep;
  }
}

// One Gram M[a][b] = sum_i A[a][i] B'[b][i] of ra and rb rows of length n (B' = D B when deriv,
// scale = 1 / (2 h)).
template <typename F>
struct EnGram {
  const F *A, *B;
  int ra, rb, n;
  bool deriv;
  double scale;
  double* M;
};

// Static shared memory of the energy kernels; its size counts against the 48 KB that a launch may ask
// for without the attribute.
template <typename F>
struct EnShared {
  double red[32];             // the block's sum
  double part[kEnWarps * 64]; // partial Gram blocks of block_grams
  EnGram<F> gram[3];
};

constexpr float kEnLarge = 1.3e36f;  // about 2^120: 32 of them stay finite

// The three Grams g[0..2] (in shared memory) by the whole block.  The work is cut into items, 8 x 8
// outputs over one segment of columns (at most 1024, so that the FP32 sums of a lane stay at 32
// products), one warp each, 8 at a time: a lane takes every 32nd column of the segment, its 8 + 8
// entries (read along the rows, coalesced) feed 64 products summed in registers, the lanes' sums are
// added without loss (EnSum) by a transposing reduction, and segments in FP64 in a fixed order.  Lane
// sums beyond kEnLarge, infinite or not a number, whose two-sum would overflow or turn an infinity into
// NaN, are added in FP64 instead.
// Bound: the latency of an item's loads and reduction, so small ranks split the columns until every
// warp has an item.  1024^3, ranks 8, R = 61 (270 blocks): 661 us when 64 x 64 tiles padded every
// rank and each partial sum and derivative was formed in FP64; 33 us now.
template <typename F>
__device__ void block_grams(const EnGram<F>* g, double* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int blocks = 0, first[4];
#pragma unroll
  for (int p = 0; p < 3; ++p) blocks += ((g[p].ra + 7) >> 3) * ((g[p].rb + 7) >> 3);
  const int want = blocks < kEnWarps ? kEnWarps / blocks : 1;  // segments per 8 x 8 block, at least
  int seg[3], segs[3], items = 0;
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    seg[p] = min(1024, ((g[p].n + want - 1) / want + 31) & ~31);
    segs[p] = (g[p].n + seg[p] - 1) / seg[p];
    first[p] = items;
    items += ((g[p].ra + 7) >> 3) * ((g[p].rb + 7) >> 3) * segs[p];
  }
  first[3] = items;
  // item -> Gram, 8 x 8 block, segment (segments of a block are consecutive)
  auto locate = [&](int item, int& p, int& a0, int& b0, int& sg) {
    p = item < first[1] ? 0 : item < first[2] ? 1 : 2;
    const int ns = p == 0 ? segs[0] : p == 1 ? segs[1] : segs[2];
    const int e = item - (p == 0 ? first[0] : p == 1 ? first[1] : first[2]);
    const int nb = (g[p].rb + 7) >> 3, blk = e / ns;
    sg = e - blk * ns;
    a0 = blk / nb * 8;
    b0 = (blk - blk / nb * nb) * 8;
  };
  for (int base = 0; base < items; base += kEnWarps) {
    if (base + warp < items) {
      int p, a0, b0, sg;
      locate(base + warp, p, a0, b0, sg);
      const F *A = g[p].A, *B = g[p].B;
      const int ra = g[p].ra, rb = g[p].rb, n = g[p].n, len = p == 0 ? seg[0] : p == 1 ? seg[1] : seg[2];
      const bool deriv = g[p].deriv;
      F acc[8][8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = F(0);
      const int iend = min(n, (sg + 1) * len);
      for (int i = sg * len + lane; i < iend; i += 32) {
        const int hi = deriv ? min(i + 1, n - 1) : i;
        F av[8], bv[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          av[r] = a0 + r < ra ? A[(long)(a0 + r) * n + i] : F(0);
          bv[r] = b0 + r < rb ? B[(long)(b0 + r) * n + hi] : F(0);
        }
        if (deriv) {  // the entries one to the right are there; those one to the left follow in one batch
          F left[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) left[r] = b0 + r < rb ? B[(long)(b0 + r) * n + max(i - 1, 0)] : F(0);
#pragma unroll
          for (int r = 0; r < 8; ++r) bv[r] = bv[r] - left[r];
          if (i == 0 || i == n - 1) {
#pragma unroll
            for (int r = 0; r < 8; ++r)
              if (b0 + r < rb) bv[r] = fd_end(B + (long)(b0 + r) * n, i, n);
          }
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int c = 0; c < 8; ++c) acc[r][c] = fma(av[r], bv[c], acc[r][c]);
      }
      bool large = false;
      if constexpr (std::is_same<F, float>::value) {
#pragma unroll
        for (int j = 0; j < 64; ++j) large = large || !(fabsf(acc[j / 8][j % 8]) <= kEnLarge);
      }
      if (__any_sync(0xffffffffu, large)) {
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          const double s = en_warp_sum((double)acc[j / 8][j % 8]);
          if (lane == 0) part[warp * 64 + j] = s;
        }
      } else {
        EnSum<F> v[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) v[j].set(acc[j / 8][j % 8]);
        en_halve<64>(v, 16);
        en_halve<32>(v, 8);
        en_halve<16>(v, 4);
        en_halve<8>(v, 2);
        en_halve<4>(v, 1);
        // a lane is left with outputs 2 lane and 2 lane + 1
        part[warp * 64 + 2 * lane] = v[0].value();
        part[warp * 64 + 2 * lane + 1] = v[1].value();
      }
    }
    __syncthreads();
    if (threadIdx.x < 64) {
      for (int w = 0; w < kEnWarps && base + w < items; ++w) {
        int p, a0, b0, sg;
        locate(base + w, p, a0, b0, sg);
        const int ia = a0 + threadIdx.x / 8, ib = b0 + threadIdx.x % 8;
        if (ia < g[p].ra && ib < g[p].rb) {
          double* o = g[p].M + ia * g[p].rb + ib;
          const double v = part[w * 64 + threadIdx.x];
          *o = (sg ? *o : 0.0) + (g[p].deriv ? g[p].scale * v : v);
        }
      }
    }
    __syncthreads();
  }
}

template <typename F>
__global__ void __launch_bounds__(32 * kEnWarps) tucker_energy_kernel(const __grid_constant__ EnTuckerT<F> a) {
  extern __shared__ double Mg[];
  __shared__ EnShared<F> sh;
  double* const red = sh.red;
  EnGram<F>* const gram = sh.gram;
  const int t = blockIdx.x, q = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int r1 = a.r[0], r2 = a.r[1], r3 = a.r[2];
  const int s1 = a.s[0], s2 = a.s[1], s3 = a.s[2];
  const int size_c = s1 * s2 * s3;
  const F* Ct = a.C + (a.core_by_q ? (long)(t % 3) * size_c : 0L);
  const int moff[4] = {0, r1 * s1, r1 * s1 + r2 * s2, r1 * s1 + r2 * s2 + r3 * s3};
  // 1. Grams M_p [r_p][s_p]
  if (threadIdx.x < 3) {
    const int p = threadIdx.x;
    long voff = (long)q * ((long)r1 * a.n[0] + (long)r2 * a.n[1] + (long)r3 * a.n[2]);
    for (int pp = 0; pp < p; ++pp) voff += (long)a.r[pp] * a.n[pp];
    gram[p] = {a.V + voff, a.W[p] + (long)t * a.s[p] * a.n[p], a.r[p],   a.s[p],
               a.n[p],     p == q,                             a.inv2h[p], Mg + moff[p]};
  }
  // the term's core in FP64, once
  double* Cd = a.ws ? nullptr : Mg + moff[3];
  if (Cd)
    for (int i = threadIdx.x; i < size_c; i += blockDim.x) Cd[i] = (double)Ct[i];
  __syncthreads();
  block_grams(gram, sh.part);
  const double *M1 = Mg, *M2 = Mg + moff[1], *M3 = Mg + moff[2];
  double* Y1 = a.ws ? a.ws + ((long)t * 3 + q) * ((long)r1 * s3 * (s2 + r2)) : Cd + size_c;
  double* Y2 = Y1 + r1 * s2 * s3;
  // 2. Y1[b3][b2][a1] = sum_b1 M1[a1][b1] C[b3][b2][b1]
  for (int idx = threadIdx.x; idx < s3 * s2 * r1; idx += blockDim.x) {
    const int bb = idx / r1, a1 = idx - bb * r1;  // b3 s2 + b2
    double acc = 0.0;
    if (Cd) {
      for (int b1 = 0; b1 < s1; ++b1) acc += M1[a1 * s1 + b1] * Cd[bb * s1 + b1];
    } else {
      for (int b1 = 0; b1 < s1; ++b1) acc += M1[a1 * s1 + b1] * (double)Ct[bb * s1 + b1];
    }
    Y1[idx] = acc;
  }
  __syncthreads();
  // 3. Y2[b3][a2][a1] = sum_b2 M2[a2][b2] Y1[b3][b2][a1]
  for (int idx = threadIdx.x; idx < s3 * r2 * r1; idx += blockDim.x) {
    const int ba = idx / r1, a1 = idx - ba * r1;
    const int b3 = ba / r2, a2 = ba - b3 * r2;
    double acc = 0.0;
    for (int b2 = 0; b2 < s2; ++b2) acc += M2[a2 * s2 + b2] * Y1[(b3 * s2 + b2) * r1 + a1];
    Y2[idx] = acc;
  }
  __syncthreads();
  // 4. X = sum_a G^(q)[a3][a2][a1] sum_b3 M3[a3][b3] Y2[b3][a2][a1]
  const F* Gq = a.G + (long)q * r1 * r2 * r3;
  double x = 0.0;
  for (int idx = threadIdx.x; idx < r3 * r2 * r1; idx += blockDim.x) {
    const int a3 = idx / (r2 * r1), a21 = idx - a3 * (r2 * r1);
    double acc = 0.0;
    for (int b3 = 0; b3 < s3; ++b3) acc += M3[a3 * s3 + b3] * Y2[b3 * r2 * r1 + a21];
    x += (double)Gq[idx] * acc;
  }
  x = en_warp_sum(x);
  if (lane == 0) red[warp] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < nw; ++i) v += red[i];
    a.part[(long)t * 3 + q] = (a.w ? (double)a.w[t] : 1.0) * v;
  }
}

// The same energy for a TT magnetization (Eq. tt_3d_1) and the 3M trains of its potential: one
// block per (term t, component q); the inner product of two trains contracts the first-core Gram
// M1[a1][b1], the middle-core Gram M2[(a1 a2)][(b1 b2)] and the last-core Gram M3[a2][b2]:
//   <A, B'> = sum_{a2, b2} M3[a2][b2] sum_{a1, b1} M1[a1][b1] M2[(a1 a2)][(b1 b2)],
// with D_q applied to the axis-q core of the term.
struct EnTT {
  int n[3];
  double inv2h[3];
  int r1, r2;                    // ranks of the magnetization and of every term
  const float* A[3];             // magnetization cores, component q at A[p] + q * (size of core p)
  const float* B[3];             // term cores, term t at B[p] + t * (size of core p)
  const float* w;                // term weights
  int T;
  double* part;                  // [T][3]
};

__global__ void __launch_bounds__(32 * kEnWarps) tt_energy_kernel(const __grid_constant__ EnTT a) {
  extern __shared__ double sg[];
  __shared__ EnShared<float> sh;
  double* const red = sh.red;
  EnGram<float>* const gram = sh.gram;
  const int t = blockIdx.x, q = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int r1 = a.r1, r2 = a.r2, r12 = r1 * r2;
  double* Mg[3] = {sg, sg + r1 * r1, sg + r1 * r1 + (long)r12 * r12};
  if (threadIdx.x < 3) {
    const int p = threadIdx.x, n = a.n[p], rp = p == 0 ? r1 : p == 1 ? r12 : r2;
    gram[p] = {a.A[p] + (long)q * rp * n, a.B[p] + (long)t * rp * n, rp, rp, n, p == q, a.inv2h[p], Mg[p]};
  }
  __syncthreads();
  block_grams(gram, sh.part);
  double x = 0.0;
  for (int e = threadIdx.x; e < r2 * r2; e += blockDim.x) {
    const int a2 = e / r2, b2 = e % r2;
    double s = 0.0;
    for (int a1 = 0; a1 < r1; ++a1)
      for (int b1 = 0; b1 < r1; ++b1) s += Mg[0][a1 * r1 + b1] * Mg[1][(long)(a1 * r2 + a2) * r12 + b1 * r2 + b2];
    x += s * Mg[2][e];
  }
  x = en_warp_sum(x);
  if (lane == 0) red[warp] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < nw; ++i) v += red[i];
    a.part[(long)t * 3 + q] = (double)a.w[t] * v;
  }
}

// energy = scale * sum part[0..count) in a fixed order (one block)
__global__ void __launch_bounds__(256) energy_sum_kernel(long count, const double* part, double scale, double* energy) {
  __shared__ double red[32];
  double acc = 0.0;
  for (long i = threadIdx.x; i < count; i += blockDim.x) acc += part[i];
  acc = en_warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) v += red[i];
    *energy = scale * v;
  }
}

// Scratch of one call, ordered on its stream (give it back with cudaFreeAsync).
// It comes from a memory pool of the plan that keeps up to 64 MiB of what was
// given back: with the device's default pool, which returns everything at each
// synchronisation, a call that is waited for spent 200 us on mapping it again.
// The pool dies with the plan.  Under stream capture the default pool is used.
static demag_status scratch_alloc(demag_plan* P, void** mem, size_t bytes, cudaStream_t st) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(st, &cap);
  if (cap == cudaStreamCaptureStatusNone && !P->pool) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    if (cudaMemPoolCreate(&P->pool, &props) != cudaSuccess) {
      P->pool = nullptr;
      cudaGetLastError();  // the default pool serves
    } else {
      unsigned long long keep = 64ull << 20;
      cudaMemPoolSetAttribute(P->pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
  }
  if (cap == cudaStreamCaptureStatusNone && P->pool)
    DEMAG_CUDA(P, cudaMallocFromPoolAsync(mem, bytes, P->pool, st));
  else
    DEMAG_CUDA(P, cudaMallocAsync(mem, bytes, st));
  return DEMAG_OK;
}

void scratch_destroy(demag_plan* P) {
  if (P->pool) cudaMemPoolDestroy(P->pool);
  P->pool = nullptr;
}

template <typename F>
static demag_status run_tucker_energy(demag_plan* P, EnTuckerT<F>& a, double* energy, cudaStream_t st,
                                      const char* who) {
  for (int p = 0; p < 3; ++p)
    if (a.r[p] < 1 || a.r[p] > kEnMaxRank || a.s[p] < 1 || a.s[p] > kEnMaxRank)
      return set_error(P, DEMAG_EINVAL, "%s: ranks must be in [1, %d]", who, kEnMaxRank);
  for (int p = 0; p < 3; ++p) {
    a.n[p] = P->n[p];
    a.inv2h[p] = 0.5 / P->h[p];
  }
  // The contraction's intermediates stay in shared memory beside the Grams where they fit (ranks up
  // to about 15), in global memory otherwise.
  const size_t grams = (size_t)a.r[0] * a.s[0] + (size_t)a.r[1] * a.s[1] + (size_t)a.r[2] * a.s[2];
  const long per = (long)a.r[0] * a.s[2] * (a.s[1] + a.r[1]), core = (long)a.s[0] * a.s[1] * a.s[2];
  const bool in_smem = sizeof(double) * (grams + per + core) <= 96 * 1024;
  const size_t smem = sizeof(double) * (grams + (in_smem ? per + core : 0));
  if (smem + sizeof(EnShared<F>) > 48 * 1024) {
    static unsigned long long done = 0;  // one per instantiation
    int dev = 0;
    cudaGetDevice(&dev);
    if (!(done & (1ull << (dev & 63)))) {
      DEMAG_CUDA(P, cudaFuncSetAttribute(tucker_energy_kernel<F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kEnSmemMax));
      done |= 1ull << (dev & 63);
    }
  }
  const long blocks = (long)a.T * 3;
  void* mem = nullptr;
  demag_status s = scratch_alloc(P, &mem, sizeof(double) * (size_t)(blocks * (in_smem ? 0 : per) + blocks), st);
  if (s != DEMAG_OK) return s;
  a.part = static_cast<double*>(mem);
  a.ws = in_smem ? nullptr : a.part + blocks;
  DEMAG_LAUNCH(P, kFamEnergy, st, tucker_energy_kernel<F><<<dim3(a.T, 3), 32 * kEnWarps, smem, st>>>(a));
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    const double vol = P->h[0] * P->h[1] * P->h[2];
    DEMAG_LAUNCH(P, kFamEnergy, st, energy_sum_kernel<<<1, 256, 0, st>>>(blocks, a.part, 0.5 * vol, energy));
    e = cudaGetLastError();
  }
  cudaFreeAsync(mem, st);
  if (e != cudaSuccess) return cuda_error(P, e, who);
  return DEMAG_OK;
}

constexpr int kEnMaxTTRank = 64;  // r1 r2: the middle core's rows, at most 64 per Gram side

// The Tucker application in FP64 for the energy study after Alg. 2: with FP32 factors the
// study's energy error stops falling near 5e-7 (n >= 2048), while the method's own error keeps
// falling.  Every factor T_{k,q,p} V^(q,p) (Eq. kron_eval_tuck; T Toeplitz with
// T[i][j] = gen[i - j], E off the component's axis, F on it) is summed directly in FP64: one
// block per (column, node), the generator row and the input column in shared memory, each
// thread a set of outputs i, each sum over j in a fixed order.
struct TuckDirect {
  int n[3], r[3];
  int glen;
  const double* gen;   // [M][2][3][glen], type 0 = E, 1 = F, entry d + n_p - 1
  const double* V;     // blocks (q, p), each [r_p][n_p]
  double* out[3];      // axis p: [M][3][r_p][n_p]
};

__global__ void __launch_bounds__(256) tucker_direct_fp64_kernel(const __grid_constant__ TuckDirect a) {
  extern __shared__ double sh[];
  const int k = blockIdx.y;
  const int per_q = a.r[0] + a.r[1] + a.r[2];
  int j = blockIdx.x;
  const int q = j / per_q;
  j -= q * per_q;
  int p = 0;
  while (j >= a.r[p]) {
    j -= a.r[p];
    ++p;
  }
  const int n = a.n[p];
  const int type = p == q ? 1 : 0;
  const double* g = a.gen + (((long)k * 2 + type) * 3 + p) * a.glen;
  long voff = (long)q * ((long)a.r[0] * a.n[0] + (long)a.r[1] * a.n[1] + (long)a.r[2] * a.n[2]);
  for (int pp = 0; pp < p; ++pp) voff += (long)a.r[pp] * a.n[pp];
  const double* v = a.V + voff + (long)j * n;
  double* vs = sh;      // [n]
  double* gs = sh + n;  // [2 n - 1]
  for (int i = threadIdx.x; i < n; i += blockDim.x) vs[i] = v[i];
  for (int i = threadIdx.x; i < 2 * n - 1; i += blockDim.x) gs[i] = g[i];
  __syncthreads();
  double* out = a.out[p] + (((long)k * 3 + q) * a.r[p] + j) * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double* gi = gs + i + n - 1;  // gi[-jj] = gen[i - jj]
    double acc = 0.0;
    for (int jj = 0; jj < n; ++jj) acc = fma(gi[-jj], vs[jj], acc);
    out[i] = acc;
  }
}

// term weights of the Tucker application, w[k][q] = c s omega_k
__global__ void tucker_weights_fp64_kernel(int M, const double* scale, double* w) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 3 * M; i += gridDim.x * blockDim.x) w[i] = scale[i / 3];
}

constexpr size_t kDirectSmemMax = 200 * 1024;  // 8 (3 nmax - 1) bytes: nmax up to 8533

}  // namespace demag

using namespace demag;

extern "C" demag_status demag_energy_tt(demag_plan* P, const int r[2], const float* G1, const float* G2,
                                        const float* G3, const float* out_w, const float* oG1, const float* oG2,
                                        const float* oG3, double* energy, void* stream) {
  if (!P) return set_error(nullptr, DEMAG_EINVAL, "demag_energy_tt: plan is NULL");
  if (!r || !G1 || !G2 || !G3 || !out_w || !oG1 || !oG2 || !oG3 || !energy)
    return set_error(P, DEMAG_EINVAL, "demag_energy_tt: NULL pointer");
  demag_status u = require_uniform(P, "demag_energy_tt");
  if (u != DEMAG_OK) return u;
  if (r[0] < 1 || r[1] < 1 || r[0] > kEnMaxRank || r[1] > kEnMaxRank || r[0] * r[1] > kEnMaxTTRank)
    return set_error(P, DEMAG_EINVAL, "demag_energy_tt: ranks must be in [1, %d] with r1 r2 <= %d", kEnMaxRank,
                     kEnMaxTTRank);
  cudaStream_t st = (cudaStream_t)stream;
  EnTT a{};
  for (int p = 0; p < 3; ++p) {
    a.n[p] = P->n[p];
    a.inv2h[p] = 0.5 / P->h[p];
  }
  a.r1 = r[0];
  a.r2 = r[1];
  a.A[0] = G1;
  a.A[1] = G2;
  a.A[2] = G3;
  a.B[0] = oG1;
  a.B[1] = oG2;
  a.B[2] = oG3;
  a.w = out_w;
  a.T = 3 * P->M;
  const int r12 = r[0] * r[1];
  const size_t smem = sizeof(double) * ((size_t)r[0] * r[0] + (size_t)r12 * r12 + (size_t)r[1] * r[1]);
  if (smem + sizeof(EnShared<float>) > 48 * 1024) {
    static unsigned long long done = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (!(done & (1ull << (dev & 63)))) {
      // largest request: r1, r2 <= 64 and r1 r2 <= 64 give at most 3 * 64^2 doubles (96 KB)
      const int cap = (int)(sizeof(double) * ((size_t)kEnMaxTTRank * kEnMaxTTRank + 2 * kEnMaxRank * kEnMaxRank));
      DEMAG_CUDA(P, cudaFuncSetAttribute(tt_energy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, cap));
      done |= 1ull << (dev & 63);
    }
  }
  const long blocks = (long)a.T * 3;
  void* mem = nullptr;
  demag_status s = scratch_alloc(P, &mem, sizeof(double) * (size_t)blocks, st);
  if (s != DEMAG_OK) return s;
  a.part = static_cast<double*>(mem);
  DEMAG_LAUNCH(P, kFamEnergy, st, tt_energy_kernel<<<dim3(a.T, 3), 256, smem, st>>>(a));
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    const double vol = P->h[0] * P->h[1] * P->h[2];
    DEMAG_LAUNCH(P, kFamEnergy, st, energy_sum_kernel<<<1, 256, 0, st>>>(blocks, a.part, 0.5 * vol, energy));
    e = cudaGetLastError();
  }
  cudaFreeAsync(mem, st);
  if (e != cudaSuccess) return cuda_error(P, e, "demag_energy_tt");
  return DEMAG_OK;
}

extern "C" demag_status demag_energy_tucker(demag_plan* P, const int r[3], const float* core, const float* V,
                                            const float* out_w, const float* out_V, double* energy, void* stream) {
  if (!P) return set_error(nullptr, DEMAG_EINVAL, "demag_energy_tucker: plan is NULL");
  if (!r || !core || !V || !out_w || !out_V || !energy)
    return set_error(P, DEMAG_EINVAL, "demag_energy_tucker: NULL pointer");
  demag_status u = require_uniform(P, "demag_energy_tucker");  // uniform stencils and cell volume
  if (u != DEMAG_OK) return u;
  EnTucker a{};
  for (int p = 0; p < 3; ++p) a.r[p] = a.s[p] = r[p];
  a.G = core;
  a.V = V;
  a.C = core;
  a.core_by_q = 1;
  const long per_mode[3] = {(long)P->M * 3 * r[0] * P->n[0], (long)P->M * 3 * r[1] * P->n[1],
                            (long)P->M * 3 * r[2] * P->n[2]};
  a.W[0] = out_V;
  a.W[1] = out_V + per_mode[0];
  a.W[2] = out_V + per_mode[0] + per_mode[1];
  a.w = out_w;
  a.T = 3 * P->M;
  return run_tucker_energy(P, a, energy, (cudaStream_t)stream, "demag_energy_tucker");
}

extern "C" demag_status demag_energy_tucker_phi(demag_plan* P, const int r[3], const float* core, const float* V,
                                                const int rho[3], const float* phi_core, const float* phi_U,
                                                double* energy, void* stream) {
  if (!P) return set_error(nullptr, DEMAG_EINVAL, "demag_energy_tucker_phi: plan is NULL");
  if (!r || !core || !V || !rho || !phi_core || !phi_U || !energy)
    return set_error(P, DEMAG_EINVAL, "demag_energy_tucker_phi: NULL pointer");
  demag_status u = require_uniform(P, "demag_energy_tucker_phi");
  if (u != DEMAG_OK) return u;
  EnTucker a{};
  for (int p = 0; p < 3; ++p) {
    a.r[p] = r[p];
    a.s[p] = rho[p];
  }
  a.G = core;
  a.V = V;
  a.C = phi_core;
  a.core_by_q = 0;
  a.W[0] = phi_U;
  a.W[1] = phi_U + (long)rho[0] * P->n[0];
  a.W[2] = a.W[1] + (long)rho[1] * P->n[1];
  a.w = nullptr;
  a.T = 1;
  return run_tucker_energy(P, a, energy, (cudaStream_t)stream, "demag_energy_tucker_phi");
}

extern "C" demag_status demag_energy_tucker_fp64(demag_plan* P, const int r[3], const double* core, const double* V,
                                                 double* energy, void* stream) {
  if (!P) return set_error(nullptr, DEMAG_EINVAL, "demag_energy_tucker_fp64: plan is NULL");
  if (!r || !core || !V || !energy) return set_error(P, DEMAG_EINVAL, "demag_energy_tucker_fp64: NULL pointer");
  demag_status u = require_uniform(P, "demag_energy_tucker_fp64");
  if (u != DEMAG_OK) return u;
  for (int p = 0; p < 3; ++p)
    if (r[p] < 1 || r[p] > kEnMaxRank)
      return set_error(P, DEMAG_EINVAL, "demag_energy_tucker_fp64: ranks must be in [1, %d]", kEnMaxRank);
  const size_t smem = sizeof(double) * (3 * (size_t)P->nmax - 1);
  if (smem > kDirectSmemMax)
    return set_error(P, DEMAG_EUNSUPPORTED, "demag_energy_tucker_fp64: %d cells per axis exceed the limit of %d",
                     P->nmax, (int)((kDirectSmemMax / sizeof(double) + 1) / 3));
  cudaStream_t st = (cudaStream_t)stream;
  if (smem > 48 * 1024) {
    static unsigned long long done = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    if (!(done & (1ull << (dev & 63)))) {
      DEMAG_CUDA(P, cudaFuncSetAttribute(tucker_direct_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kDirectSmemMax));
      done |= 1ull << (dev & 63);
    }
  }
  const int M = P->M;
  const long per_mode[3] = {(long)M * 3 * r[0] * P->n[0], (long)M * 3 * r[1] * P->n[1],
                            (long)M * 3 * r[2] * P->n[2]};
  void* mem = nullptr;
  demag_status s = scratch_alloc(P, &mem, sizeof(double) * (size_t)(per_mode[0] + per_mode[1] + per_mode[2] + 3 * M),
                                 st);
  if (s != DEMAG_OK) return s;
  double* outV = static_cast<double*>(mem);
  double* w = outV + per_mode[0] + per_mode[1] + per_mode[2];
  TuckDirect d{};
  for (int p = 0; p < 3; ++p) {
    d.n[p] = P->n[p];
    d.r[p] = r[p];
  }
  d.glen = P->glen;
  d.gen = P->gen64;
  d.V = V;
  d.out[0] = outV;
  d.out[1] = outV + per_mode[0];
  d.out[2] = outV + per_mode[0] + per_mode[1];
  DEMAG_LAUNCH(P, kFamEnergy, st,
               tucker_direct_fp64_kernel<<<dim3(3 * (r[0] + r[1] + r[2]), M), 256, smem, st>>>(d));
  DEMAG_LAUNCH(P, kFamEnergy, st, tucker_weights_fp64_kernel<<<1, 256, 0, st>>>(M, P->scale, w));
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    cudaFreeAsync(mem, st);
    return cuda_error(P, e, "demag_energy_tucker_fp64");
  }
  EnTuckerT<double> a{};
  for (int p = 0; p < 3; ++p) a.r[p] = a.s[p] = r[p];
  a.G = core;
  a.V = V;
  a.C = core;
  a.core_by_q = 1;
  a.W[0] = d.out[0];
  a.W[1] = d.out[1];
  a.W[2] = d.out[2];
  a.w = w;
  a.T = 3 * M;
  s = run_tucker_energy(P, a, energy, st, "demag_energy_tucker_fp64");
  cudaFreeAsync(mem, st);
  return s;
}
