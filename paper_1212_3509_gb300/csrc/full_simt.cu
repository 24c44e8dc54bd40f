// Full format: the Kronecker operator by chained mode products on CUDA cores.
//
// Cor. 3 (Eq. kron_operator) with the mode product of Sec. 2.2 (Eq. modemul):
// per node k and component q the three Toeplitz factors act along i1, i2, i3.
// The modes are applied in the order 3, 2, 1.  Per node the nine products
// share work (8 products of n^4 multiply-adds):
//   axis 3:  Y_q = m_q x_3 E (q = 1, 2),  Y_3 = m_3 x_3 F
//   axis 2:  U = Y_2 x_2 F + Y_3 x_2 E,  V = Y_1 x_2 E
//   axis 1:  phi = sum_k (U_k x_1 S_k E + V_k x_1 S_k F),  S_k = c s omega_k
// (S_k reaches 10^4 where E is small, so it goes with the last product: before it no field outgrows the
// input's, E and F being integrals over a part of [-1, 1]).
// and the node sum of the last stage is one contraction of length 2 n1 M.
// Every field stays in the caller's layout [i3][i2][i1]: along axes 3 and 2
// the rows of a product (everything but the contracted index) are contiguous
// or in contiguous runs of n1, so nothing is ever transposed; only the last
// stage reads its contraction index contiguously.
//
// Even / odd halves.  With x+_j = x_j + x_{n-1-j} and x-_j = x_j - x_{n-1-j}
// (j < h = ceil(n/2)) a symmetric Toeplitz factor maps x+ to the even half
// p_a = (y_a + y_{n-1-a})/2 of the output and x- to the odd half
// q_a = (y_a - y_{n-1-a})/2, a skew one the other way round, so a product
// takes half the multiply-adds of the dense factor.  The sums x+- are formed
// while a tile is loaded and y_a = p_a + q_a, y_{n-1-a} = p_a - q_a in its
// epilogue: no folded copy of any field exists.  A factor without that
// symmetry (non-uniform grid) is the sum of two such parts.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cooperative_groups.h>
#include <mutex>
#include <type_traits>

#include "internal.h"

namespace demag {

constexpr int kMaxPairs = 4;  // (field, factor part) pairs summed by one output field of one node

// One launch: outputs (node, job), each sum over its pairs of a half-matrix
// product along one axis.  Element (row r, index j) of a field is at
// (r / inner) * ostride + r % inner + j * kstride.
struct ModeStage {
  int n, h, ldh;          // contracted axis, ceil(n / 2), leading dimension of the factor parts
  int inner;              // contiguous rows
  unsigned inner_mul, inner_shift;  // r / inner = (umulhi(r, inner_mul) + r) >> inner_shift
  long ostride, kstride;
  int rows;               // rows of one field
  long N;                 // elements of one field
  const void* A;          // input fields
  const void* B;          // factor parts of this axis, first node of the launch
  void* C;                // output fields
  long b_node;            // elements between the factor parts of consecutive nodes
  int nodes;              // nodes of this launch: one output per node, or summed (SUM)
  int a_node, c_node;     // fields per node in A (0: shared by the nodes) and C
  int njobs;              // outputs per node
  int npairs[3];          // pairs per output
  int a_field[3][kMaxPairs];
  long b_off[3][kMaxPairs];
  int swap[3][kMaxPairs]; // 0: even half from x+, odd from x-; 1: the other way round
  int tiles_n;
  int split;              // SUM: node ranges, one per block of a cluster
  float alpha;            // SUM: scale of the result
};

// ---------------------------------------------------------------- the kernel
//
// Bound: the FP32 (FP64) pipe, and close behind it the words that shared
// memory delivers to registers (32 per cycle and SM against 128 multiply-adds).
// A block owns BM rows x BN columns of both output halves, a thread TM x TN of
// each.  The two halves travel as pairs: (x+, x-) of a row and (even, odd) of a
// factor entry are neighbours in shared memory and one packed operand of
// fma.rn.f32x2, whose result is the pair of accumulators (the roundings of two
// fmaf).  2 (TM + TN) words then feed 2 TM TN multiply-adds: with 8 x 8 both
// pipes are equally full, which is why the widest tile has 128 accumulators.
// Factor parts go to shared memory by cp.async in their global layout; x+- are
// formed from registers loaded while the previous operands are used.
constexpr int kBK = 8;

template <typename T, int BM_, int BN_, int TM_, int TN_, int OCC_>
struct ModeCfg {
  static constexpr int OCC = OCC_;                 // resident blocks the registers are bounded for
  static constexpr int BM = BM_, BN = BN_, TM = TM_, TN = TN_;
  static constexpr int WR = BM / (8 * TM), WC = BN / (4 * TN);  // warps along rows and columns, 8 x 4 threads each
  static constexpr int NT = 32 * WR * WC;
  static constexpr int VA = 8 / (int)sizeof(T);    // pairs per 16-byte read
  static constexpr int LDA = BM + 2;               // 16-byte rows; the offset spreads transposed stores over the banks
  static constexpr int LA = BM * kBK / NT;
  static constexpr int LB = BN * kBK / VA;         // 16-byte copies of a factor block
  static constexpr size_t operands = (size_t)2 * kBK * (LDA + BN) * 2 * sizeof(T);
  static constexpr size_t reduce = (size_t)2 * BM * BN * sizeof(T);
  static_assert(LA * NT == BM * kBK && WR * 8 * TM == BM && WC * 4 * TN == BN, "tiles divide evenly");
};

// r / inner and r % inner by multiplication (rows stay below 2^31)
template <int KIND>
__device__ __forceinline__ long row_offset(const ModeStage& S, int r) {
  if (KIND == 0) return r;  // axis 3: all rows are one run
  if (KIND == 2) return r * S.ostride;
  const int q = (int)((__umulhi((unsigned)r, S.inner_mul) + (unsigned)r) >> S.inner_shift);
  return q * S.ostride + (r - q * S.inner);
}

__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// A thread's accumulators of both halves: TM x TN pairs.
template <typename Cfg, typename T> struct ModeAcc;
template <typename Cfg> struct ModeAcc<Cfg, float> {
  unsigned long long v[Cfg::TM][Cfg::TN];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < Cfg::TM; ++i)
#pragma unroll
      for (int j = 0; j < Cfg::TN; ++j) v[i][j] = 0ull;
  }
  __device__ __forceinline__ float get(int s, int i, int j) const {
    return __uint_as_float((unsigned)(s ? v[i][j] >> 32 : v[i][j] & 0xffffffffull));
  }
  // += pairs of rows (at ax) * pairs of factor entries (at bx)
  __device__ __forceinline__ void step(const float2* ax, const float2* bx) {
    unsigned long long a[Cfg::TM], b[Cfg::TN];
#pragma unroll
    for (int c = 0; c < Cfg::TM / 2; ++c) {
      const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(ax + c * 16);
      a[2 * c] = u.x;
      a[2 * c + 1] = u.y;
    }
#pragma unroll
    for (int j = 0; j < Cfg::TN / 2; ++j) {
      const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(bx + 2 * j);
      b[2 * j] = u.x;
      b[2 * j + 1] = u.y;
    }
#pragma unroll
    for (int i = 0; i < Cfg::TM; ++i)
#pragma unroll
      for (int j = 0; j < Cfg::TN; ++j) fma2(v[i][j], a[i], b[j]);
  }
};
template <typename Cfg> struct ModeAcc<Cfg, double> {
  double v[2][Cfg::TM][Cfg::TN];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int i = 0; i < Cfg::TM; ++i)
#pragma unroll
        for (int j = 0; j < Cfg::TN; ++j) v[s][i][j] = 0.0;
  }
  __device__ __forceinline__ double get(int s, int i, int j) const { return v[s][i][j]; }
  __device__ __forceinline__ void step(const double2* ax, const double2* bx) {
    double2 a[Cfg::TM], b[Cfg::TN];
#pragma unroll
    for (int i = 0; i < Cfg::TM; ++i) a[i] = ax[i * 8];
#pragma unroll
    for (int j = 0; j < Cfg::TN; ++j) b[j] = bx[j];
#pragma unroll
    for (int i = 0; i < Cfg::TM; ++i)
#pragma unroll
      for (int j = 0; j < Cfg::TN; ++j) {
        v[0][i][j] = fma(a[i].x, b[j].x, v[0][i][j]);
        v[1][i][j] = fma(a[i].y, b[j].y, v[1][i][j]);
      }
  }
};

template <typename T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

// 16 bytes to shared memory, zeros instead when !ok
__device__ __forceinline__ void copy16(void* dst, const void* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// KIND 0: axis 3 (reads the caller's FP32 fields), 1: axis 2, 2: axis 1 with the node sum (contraction
// index contiguous; writes the caller's FP32 fields; the node ranges of a cluster's blocks are added in
// rank order through distributed shared memory)
template <typename T, typename Cfg, int KIND>
__global__ void __launch_bounds__(Cfg::NT, Cfg::OCC) mode_kernel(const __grid_constant__ ModeStage S) {
  constexpr bool SUM = KIND == 2, KCONTIG = KIND == 2;
  using TA = typename std::conditional<KIND == 0, float, T>::type;
  using TC = typename std::conditional<KIND == 2, float, T>::type;
  using P2 = typename Pair<T>::type;
  constexpr int BM = Cfg::BM, BN = Cfg::BN, NT = Cfg::NT, LA = Cfg::LA, LB = Cfg::LB, LDA = Cfg::LDA;
  constexpr int TM = Cfg::TM, TN = Cfg::TN, VA = Cfg::VA;
  extern __shared__ __align__(16) unsigned char mode_smem[];
  P2* const As = reinterpret_cast<P2*>(mode_smem);  // [2 buffers][BK][LDA]: (x+, x-), or (x-, x+) for a swapped pair
  P2* const Bs = As + 2 * kBK * LDA;                // [2 buffers][BK][BN]: (to the even, to the odd output half)

  const int tid = threadIdx.x;
  const int rank = SUM ? (int)(blockIdx.x % S.split) : 0;
  int tile = SUM ? blockIdx.x / S.split : blockIdx.x;
  const int tn = tile % S.tiles_n;
  tile /= S.tiles_n;
  const int job = tile % S.njobs;
  tile /= S.njobs;
  int k0 = 0, k1 = 1;
  if (SUM) {
    k0 = S.nodes * rank / S.split;
    k1 = S.nodes * (rank + 1) / S.split;
  } else {
    k0 = tile % S.nodes;
    tile /= S.nodes;
    k1 = k0 + 1;
  }
  const int row0 = tile * BM;
  const int col0 = tn * BN;
  const int npairs = S.npairs[job];
  const int nkb = (S.h + kBK - 1) / kBK;
  const int steps = (k1 - k0) * npairs * nkb;

  // The elements (index lk(i), row lr(i)) this thread loads per step: consecutive threads on consecutive
  // rows or, with the contraction index contiguous, on 8 indices of one row.
  constexpr int RP = KCONTIG ? LA : (BM > NT ? BM / NT : 1);  // different rows
  constexpr int KSTEP = BM > NT ? 1 : NT / BM;
  static_assert(KCONTIG || (BM > NT ? BM % NT == 0 : NT % BM == 0), "row mapping");
  auto lk = [&](int i) { return KCONTIG ? tid % kBK : (BM > NT ? i / RP : tid / BM + i * KSTEP); };
  auto lr = [&](int i) { return KCONTIG ? tid / kBK + i * (NT / kBK) : (BM > NT ? tid + (i % RP) * NT : tid % BM); };
  long rbase[RP];
  bool rok[RP];
#pragma unroll
  for (int i = 0; i < RP; ++i) {
    const int r = row0 + lr(i);
    rok[i] = r < S.rows;
    rbase[i] = row_offset<KIND>(S, r);
  }

  // raw entries x_j, x_{n-1-j} of the next operands: their sums are formed when they are stored, so
  // that no arithmetic waits for the loads while the current operands are used
  TA ax[LA], ay[LA];
  int ld_sw = 0;
  int ld_k = k0, ld_p = 0, ld_kb = 0;  // what the next load fetches
  auto load = [&](int buf) {
    const TA* A = reinterpret_cast<const TA*>(S.A) + ((long)ld_k * S.a_node + S.a_field[job][ld_p]) * S.N;
    const P2* B = reinterpret_cast<const P2*>(reinterpret_cast<const T*>(S.B) + (long)ld_k * S.b_node +
                                              S.b_off[job][ld_p]);
    ld_sw = S.swap[job][ld_p];
    const int j0 = ld_kb * kBK;
    const bool whole = j0 + kBK <= S.h;
    P2* b = Bs + buf * kBK * BN;
#pragma unroll
    for (int i = 0; i < (LB + NT - 1) / NT; ++i) {
      const int e = tid + i * NT, kk = e / (BN / VA), a = e % (BN / VA) * VA;
      if (LB % NT == 0 || e < LB) {
        const bool ok = (whole || j0 + kk < S.h) && col0 + a < S.ldh;
        copy16(b + kk * BN + a, ok ? B + (j0 + kk) * S.ldh + col0 + a : B, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (whole && row0 + BM <= S.rows) {  // no bounds: addresses advance by fixed strides
      const long d = KCONTIG ? (NT / kBK) * S.ostride : KSTEP * S.kstride;
      const long ox = (j0 + lk(0)) * S.kstride, oy = (S.n - 1 - j0 - lk(0)) * S.kstride;
#pragma unroll
      for (int i = 0; i < LA; ++i) {
        const TA* p = A + rbase[KCONTIG ? 0 : i % RP];
        const int t = KCONTIG ? i : i / RP;
        ax[i] = p[ox + t * d];
        ay[i] = p[KCONTIG ? oy + t * d : oy - t * d];
      }
    } else {
#pragma unroll
      for (int i = 0; i < LA; ++i) {
        const int ri = i % RP, j = j0 + lk(i);
        ax[i] = ay[i] = (TA)0;
        if (rok[ri] && j < S.h) {
          ax[i] = A[rbase[ri] + j * S.kstride];
          ay[i] = A[rbase[ri] + (S.n - 1 - j) * S.kstride];
        }
      }
    }
    if (++ld_kb == nkb) {
      ld_kb = 0;
      if (++ld_p == npairs) {
        ld_p = 0;
        ++ld_k;
      }
    }
  };
  auto store = [&](int buf) {
    P2* a = As + buf * kBK * LDA;
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const T x = (T)ax[i];
      P2 v;
      if constexpr (KIND == 0 && std::is_same<T, float>::value) {
        // half sums, which two values of any size have; the fields between the stages are half their
        // values, and the axis-1 factors make up for it
        const float y = 0.5f * ay[i], p = fmaf(0.5f, x, y), q = fmaf(0.5f, x, -y);
        v.x = ld_sw ? q : p;
        v.y = ld_sw ? p : q;
      } else {
        const T y = (T)ay[i];
        v.x = ld_sw ? x - y : x + y;
        v.y = ld_sw ? x + y : x - y;
      }
      a[lk(i) * LDA + lr(i)] = v;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  };

  const int warp = tid / 32, lane = tid % 32;
  const int wr = (warp % Cfg::WR) * (8 * TM) + (lane % 8) * VA;  // row of accumulator i: wr + (i / VA) 8 VA + i % VA
  const int wc = (warp / Cfg::WR) * (4 * TN) + (lane / 8) * TN;  // column of accumulator j: wc + j
  ModeAcc<Cfg, T> acc;
  acc.clear();
  if (steps > 0) {
    load(0);
    store(0);
  }
  __syncthreads();
  for (int s = 0; s < steps; ++s) {
    const int cur = s & 1;
    if (s + 1 < steps) load(cur ^ 1);
    const P2* a = As + cur * kBK * LDA + wr;
    const P2* b = Bs + cur * kBK * BN + wc;
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) acc.step(a + kk * LDA, b + kk * BN);
    if (s + 1 < steps) store(cur ^ 1);
    __syncthreads();
  }

  const T alpha = SUM ? (T)S.alpha : (T)1;
  if (SUM && S.split > 1) {
    // add the ranges' halves in rank order; block `rank` finishes its share of the columns
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    T* red = reinterpret_cast<T*>(mode_smem);  // [half][BN][BM], the operand buffers are done with
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int j = 0; j < TN; ++j)
#pragma unroll
        for (int i = 0; i < TM; ++i)
          red[((long)s * BN + wc + j) * BM + wr + (i / VA) * 8 * VA + i % VA] = acc.get(s, i, j);
    cluster.sync();
    const int c0 = BN * rank / S.split, c1 = BN * (rank + 1) / S.split;
    TC* C = reinterpret_cast<TC*>(S.C) + (long)job * S.N;
    for (int e = tid; e < (c1 - c0) * BM; e += NT) {
      // the contraction index is the fastest of the output too: consecutive threads on consecutive columns
      const int c = c0 + e % (c1 - c0), r = e / (c1 - c0);
      const int a = col0 + c;
      const int row = row0 + r;
      if (a >= S.h || row >= S.rows) continue;
      T p = (T)0, q = (T)0;
      for (int s = 0; s < S.split; ++s) {
        const T* o = cluster.map_shared_rank(red, s);
        p += o[(long)c * BM + r];
        q += o[(long)(BN + c) * BM + r];
      }
      const int a2 = S.n - 1 - a;
      C[row * S.ostride + a] = (TC)(alpha * (p + q));
      if (a2 != a) C[row * S.ostride + a2] = (TC)(alpha * (p - q));
    }
    cluster.sync();  // no block leaves while another still reads its halves
    return;
  }

  TC* C = reinterpret_cast<TC*>(S.C) + ((long)(SUM ? 0 : k0) * S.c_node + job) * S.N;
#pragma unroll
  for (int c = 0; c < TM / VA; ++c) {
    const int r = row0 + wr + c * 8 * VA;
    // rows r .. r + VA - 1: consecutive addresses from an aligned one when inner and kstride allow it
    const bool vec = !KCONTIG && S.inner % VA == 0 && S.kstride % VA == 0 && S.N % VA == 0 && r + VA <= S.rows;
    long o[VA];
#pragma unroll
    for (int v = 0; v < VA; ++v)
      o[v] = v && vec ? 0 : row_offset<KIND>(S, r + v);
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int a = col0 + wc + j;
      if (a >= S.h) continue;
      const int a2 = S.n - 1 - a;
      T hi[VA], lo[VA];
#pragma unroll
      for (int v = 0; v < VA; ++v) {
        const T p = acc.get(0, c * VA + v, j), q = acc.get(1, c * VA + v, j);
        hi[v] = alpha * (p + q);
        lo[v] = alpha * (p - q);
      }
      if constexpr (!KCONTIG && VA == 2) {
        if (vec) {
          *reinterpret_cast<float2*>(C + o[0] + a * S.kstride) = make_float2(hi[0], hi[1]);
          if (a2 != a) *reinterpret_cast<float2*>(C + o[0] + a2 * S.kstride) = make_float2(lo[0], lo[1]);
          continue;
        }
      }
#pragma unroll
      for (int v = 0; v < VA; ++v) {
        if (r + v >= S.rows) break;
        C[o[v] + a * S.kstride] = (TC)hi[v];
        if (a2 != a) C[o[v] + a2 * S.kstride] = (TC)lo[v];
      }
    }
  }
}

// ---------------------------------------------------------------- factor parts
//
// Per (node, type, axis) and part: h x ldh pairs [j][a] (a contiguous), the
// factors to the even and to the odd output half.  With
// j' = n-1-j, a' = n-1-a and T = gen[a - j]:
//   uniform grid (one part): (T[a][j] +- T[a][j'])/2, halved at j = j' where
//   x+ holds the entry twice; symmetric factors go x+ -> even, x- -> odd,
//   skew ones x- -> even, x+ -> odd;
//   non-uniform grid (two parts): the even / odd blocks of any matrix, part 0
//   (x+ -> even, x- -> odd), part 1 (x- -> even, x+ -> odd).
// Formed in FP64 and rounded once; the axis-1 factors carry c s omega_k, in FP32 twice that: the
// axis-3 stage takes x+-/2, since the sum of two values of more than half the type's maximum overflows.

struct ModeLayout {
  int h[3], ldh[3];
  int nparts;
  size_t off[3], part;  // offset of axis p inside one part, elements of one part (all axes)
};

static ModeLayout mode_layout(const demag_plan* P) {
  ModeLayout L;
  L.nparts = P->nonuniform ? 2 : 1;
  L.part = 0;
  for (int p = 0; p < 3; ++p) {
    L.h[p] = (P->n[p] + 1) / 2;
    L.ldh[p] = (L.h[p] + 1) / 2 * 2;  // 16-byte rows of pairs
    L.off[p] = L.part;
    L.part += (size_t)2 * L.h[p] * L.ldh[p];
  }
  return L;
}

static size_t factor_elems(const demag_plan* P) {
  const ModeLayout L = mode_layout(P);
  return (size_t)P->M * 2 * L.nparts * L.part;
}

struct FactorSource {
  int n[3], glen;
  const double* gen;    // [M][2][3][glen] (uniform grid)
  const double* fac;    // [M][2][tgroup] full matrices (non-uniform grid), else NULL
  size_t tgroup, toff[3];
  const double* scale;  // [M]
  int skew_e;           // type 0 is the skew factor (derivative generators)
  int transpose;
};

template <typename T>
__global__ void factor_parts_kernel(int M, ModeLayout L, FactorSource s, T* out) {
  const size_t total = (size_t)M * 2 * L.nparts * L.part;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const size_t e = idx % L.part;
    const size_t ktp = idx / L.part;
    const int part = (int)(ktp % L.nparts);
    const size_t kt = ktp / L.nparts;  // k * 2 + type
    const int p = e < L.off[1] ? 0 : (e < L.off[2] ? 1 : 2);
    const int n = s.n[p], h = L.h[p], ld = L.ldh[p];
    const size_t local = e - L.off[p];
    const int odd = (int)(local & 1);  // output half
    const int j = (int)(local / 2 / ld), a = (int)(local / 2 % ld);
    double v = 0.0;
    if (a < h) {
      const int j2 = n - 1 - j, a2 = n - 1 - a;
      auto entry = [&](int i, int jj) -> double {
        if (!s.fac) return s.gen[(kt * 3 + p) * s.glen + (i - jj + n - 1)];
        const double* f = s.fac + kt * s.tgroup + s.toff[p];
        return s.transpose ? f[(size_t)jj * n + i] : f[(size_t)i * n + jj];
      };
      const bool skew = s.fac ? part == 1 : ((int)(kt & 1) ^ s.skew_e);
      const double sj = (odd != 0) != skew ? -1.0 : 1.0;  // -1: this half is fed by x-
      v = 0.5 * (entry(a, j) + sj * entry(a, j2));
      if (s.fac) v = 0.5 * (v + (odd ? -0.5 : 0.5) * (entry(a2, j) + sj * entry(a2, j2)));
      if (j == j2) v *= 0.5;
      if (p == 0) v *= (std::is_same<T, float>::value ? 2.0 : 1.0) * s.scale[kt / 2];
    }
    out[idx] = (T)v;
  }
}

template <typename T>
static demag_status build_factor_parts(demag_plan* P, const double* gen, bool deriv, bool transpose, T* out,
                                       cudaStream_t st) {
  FactorSource s;
  for (int p = 0; p < 3; ++p) {
    s.n[p] = P->n[p];
    s.toff[p] = P->toff[p];
  }
  s.glen = P->glen;
  s.gen = gen;
  s.fac = P->nonuniform ? P->fac64 : nullptr;
  s.tgroup = P->tgroup;
  s.scale = P->scale;
  s.skew_e = deriv;
  s.transpose = transpose;
  const size_t total = factor_elems(P);
  int blocks = (int)((total + 255) / 256 > 152 * 64 ? 152 * 64 : (total + 255) / 256);
  DEMAG_LAUNCH(P, kFamSetup, st, factor_parts_kernel<T><<<blocks, 256, 0, st>>>(P->M, mode_layout(P), s, out));
  DEMAG_LAUNCHED(P, "factor_parts_kernel");
  return DEMAG_OK;
}

template <typename T>
static demag_status ensure_parts(demag_plan* P, T** out, const double* gen, bool deriv, bool transpose,
                                 cudaStream_t st) {
  if (*out) return DEMAG_OK;
  DEMAG_CUDA(P, cudaMalloc(out, sizeof(T) * factor_elems(P)));
  return build_factor_parts<T>(P, gen, deriv, transpose, *out, st);
}

demag_status ensure_dense_factors(demag_plan* P, demag_precision prec, cudaStream_t st) {
  return prec == DEMAG_FP64 ? ensure_parts<double>(P, &P->T64, P->gen64, false, false, st)
                            : ensure_parts<float>(P, &P->T32, P->gen64, false, false, st);
}

// Transposed factors of a non-uniform plan, for the adjoint on CUDA cores:
// (P^(q))^T = c sum_k omega_k U3^T (x) U2^T (x) U1^T.
static demag_status ensure_transposed_factors(demag_plan* P, demag_precision prec, cudaStream_t st) {
  return prec == DEMAG_FP64 ? ensure_parts<double>(P, &P->T64t, P->gen64, false, true, st)
                            : ensure_parts<float>(P, &P->T32t, P->gen64, false, true, st);
}

// ---------------------------------------------------------------- launches

// The factors used along each axis: the forward (or transposed) table, or the
// derivative table, whose even and odd factors change places.
template <typename T> struct ModeFactors {
  const T* base[3];
  bool deriv[3];
};

// Stage `kind` (0: axis 3, 1: axis 2, 2: axis 1 with the node sum) of nodes [k0, k0 + nodes)
template <typename T>
static ModeStage make_stage(const demag_plan* P, int kind, const ModeFactors<T>& F, int k0, int nodes, const void* A,
                            int a_node, void* C, int c_node) {
  const ModeLayout L = mode_layout(P);
  const int p = 2 - kind;
  ModeStage S;
  S.n = P->n[p];
  S.h = L.h[p];
  S.ldh = L.ldh[p];
  S.N = (long)field_size(P);
  S.rows = (int)(S.N / S.n);
  S.kstride = p == 0 ? 1 : p == 1 ? P->n[0] : (long)P->n[0] * P->n[1];
  S.inner = (int)S.kstride;
  S.ostride = S.kstride * S.n;
  S.inner_shift = 0;
  while ((1ull << S.inner_shift) < (unsigned long long)S.inner) ++S.inner_shift;
  S.inner_mul = (unsigned)(((1ull << 32) * ((1ull << S.inner_shift) - S.inner)) / S.inner + 1);
  S.A = A;
  S.b_node = (long)(2 * L.nparts * L.part);
  S.B = F.base[p] + (size_t)k0 * S.b_node + L.off[p];
  S.C = C;
  S.nodes = nodes;
  S.a_node = a_node;
  S.c_node = c_node;
  S.njobs = 0;
  S.npairs[0] = S.npairs[1] = S.npairs[2] = 0;
  S.split = 1;
  S.alpha = 1.f;
  return S;
}

// One more (field, factor type) pair of output `job`
template <typename T>
static void add_pair(const demag_plan* P, ModeStage& S, const ModeFactors<T>& F, int axis, int job, int field,
                     int type) {
  const ModeLayout L = mode_layout(P);
  if (job >= S.njobs) S.njobs = job + 1;
  for (int part = 0; part < L.nparts; ++part) {
    const int at = S.npairs[job]++;
    S.a_field[job][at] = field;
    S.b_off[job][at] = (long)((type * L.nparts + part) * L.part);
    S.swap[job][at] = L.nparts == 2 ? part : (type ^ (F.deriv[axis] ? 1 : 0));
  }
}

template <typename T, typename Cfg, int KIND>
static cudaError_t launch_mode_cfg(demag_plan* P, ModeStage S, int split, cudaStream_t st) {
  S.tiles_n = (S.h + Cfg::BN - 1) / Cfg::BN;
  S.split = split;
  const long tiles = ((long)S.rows + Cfg::BM - 1) / Cfg::BM * S.tiles_n * S.njobs * (KIND == 2 ? split : S.nodes);
  if (tiles > INT_MAX) return cudaErrorInvalidValue;
  const size_t smem = split > 1 && Cfg::reduce > Cfg::operands ? Cfg::reduce : Cfg::operands;
  if (Cfg::reduce > 48 * 1024 || Cfg::operands > 48 * 1024) {
    static unsigned long long done = 0;  // once per device: later launches, e.g. under capture, make no attribute calls
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(done & bit)) {
      const size_t most = Cfg::reduce > Cfg::operands ? Cfg::reduce : Cfg::operands;
      cudaError_t e = cudaFuncSetAttribute(mode_kernel<T, Cfg, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)most);
      if (e != cudaSuccess) return e;
      done |= bit;
    }
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3((unsigned)tiles);
  lc.blockDim = dim3(Cfg::NT);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)split;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = split > 1 ? 1 : 0;
  cudaError_t e = cudaSuccess;
  DEMAG_LAUNCH(P, kFamGemmSimt, st, e = cudaLaunchKernelEx(&lc, mode_kernel<T, Cfg, KIND>, S));
  return e;
}

// Time of a stage in a configuration, up to a factor: the tiles of the busiest
// SM, times their multiply-adds (contraction steps plus prologue and epilogue,
// and the exchange of a split sum), over the configuration's rate, which falls
// when fewer blocks are resident than fit.  The rates and overheads were fitted
// to the times of every configuration at 13 grids from 16^3 to 192^3 (R = 41):
// for the stages of axes 3 and 2 the choice is within 2% of the fastest on
// average (the split sum of axis 1 needs the terms below).  E.g. axis 3 of 128^3:
// 128 x 64 tiles 398 us, 256 x 32 413, 128 x 32 447, 256 x 16 493, 64 x 16 705;
// of 16^3: 10.2, 10.2, 11.0, 10.1, 7.0; axis 1 (the node sum) of 48^3: 128 x 64
// 129, split over 4 blocks 45, 64 x 16 over 8 blocks 26.5.
struct ModeShape {
  int bm, bn, occ;
  double rate, fill;  // at full occupancy; exponent of the resident share below it
};

// A split sum runs as clusters, and three things decide its time beside that:
// the longest node range (20 nodes over 6 or 7 blocks: 4 and 3); the share of the
// block slots that clusters of one size can fill (as
// cudaOccupancyMaxActiveClusters reports it: 266 of 304 for 7 blocks, 296 for 4);
// and, when there are few, that a cluster stays in one of eight groups of up to
// 20 SMs, which 3 clusters of 7 overfill while others idle.  With them, and its
// own rates, the sum's choice is 0.3% off the fastest split and tile on average
// over 14 FP32 grids (1.3% at most), where the model of whole SMs was 6% (18%)
// off: 128^3 1170 -> 1130 us, 112^3 823 -> 748, 64^3 146 -> 124, 128 x 40 x 60
// 220 -> 188 (the whole application).
static double cluster_share(int occ, int split) {
  static const double share[3][9] = {{1, 1, 1, .957, .974, .954, .908, .875, .947},   // 2 blocks per SM
                                     {1, 1, 1, .974, .965, .954, .974, .906, .895},   // 3
                                     {1, 1, 1, .970, .974, .966, .957, .938, .974}};  // 6 or 8
  return share[occ <= 2 ? 0 : occ <= 3 ? 1 : 2][split];
}

static double mode_cost(const ModeStage& S, bool sum, const ModeShape& c, int split) {
  double pairs = 0;
  for (int j = 0; j < S.njobs; ++j) pairs += S.npairs[j];
  pairs /= S.njobs;
  const double tiles = std::ceil((double)S.rows / c.bm) * ((S.h + c.bn - 1) / c.bn) * S.njobs * (sum ? split : S.nodes);
  const double steps = (double)((S.h + kBK - 1) / kBK * kBK) * pairs *
                       (sum ? 0.8 * ((S.nodes + split - 1) / split) + 0.2 * S.nodes / split : 1.0);
  double per_sm = std::ceil(tiles / (152.0 * cluster_share(c.occ, split)) - 1e-9);
  if (split > 1) per_sm = std::max(per_sm, std::ceil(std::ceil(tiles / split / 8) * split / 20));
  const double full = per_sm < c.occ ? std::pow(per_sm / c.occ, c.fill) : 1.0;
  return per_sm * (steps + 24 + (split > 1 ? 48 : 0)) * c.bm * c.bn / (c.rate * full);
}

template <typename T, int KIND>
static cudaError_t launch_mode(demag_plan* P, const ModeStage& S, cudaStream_t st) {
  constexpr bool SUM = KIND == 2;
  using Fn = cudaError_t (*)(demag_plan*, ModeStage, int, cudaStream_t);
  struct Choice {
    ModeShape shape;
    Fn run;
  } all[5];
  int count = 0;
  auto add = [&](auto cfg, double rate) {
    using Cfg = decltype(cfg);
    all[count++] = {{Cfg::BM, Cfg::BN, Cfg::OCC, rate, SUM && std::is_same<T, float>::value ? 0.7 : 0.3},
                    launch_mode_cfg<T, Cfg, KIND>};
  };
  if constexpr (std::is_same<T, float>::value) {
    add(ModeCfg<float, 128, 64, 8, 8, 2>{}, 1.0);
    add(ModeCfg<float, 256, 32, 8, 8, 2>{}, 0.95);
    add(ModeCfg<float, 128, 32, 8, 4, 3>{}, SUM ? 0.85 : 0.8);
    add(ModeCfg<float, 256, 16, 8, 4, 3>{}, SUM ? 0.85 : 0.8);
    add(ModeCfg<float, 64, 16, 4, 2, 8>{}, 0.6);
  } else {
    // FP64 multiply-adds run at 1/64 of the FP32 rate: any tile feeds them, and small ones balance the SMs
    add(ModeCfg<double, 64, 32, 4, 4, 3>{}, 1.0);
    add(ModeCfg<double, 32, 16, 2, 2, 6>{}, 0.9);
  }
  const int most = SUM ? std::min(S.nodes, 8) : 1;
  const Choice* pick = nullptr;
  int split = 1;
  double best = 0;
  for (int c = 0; c < count; ++c)
    for (int s = 1; s <= most; ++s) {
      const double t = mode_cost(S, SUM, all[c].shape, s);
      if (!pick || t < best) {
        best = t;
        pick = &all[c];
        split = s;
      }
    }
  // an FP32 sum goes to four blocks where the model sees little between them and fewer: shorter chains of
  // additions (128^3: error 5.7e-7 over 2 blocks, 3.0e-7 over 4, 1130 and 1127 us); where they fill the
  // chip worse they stay fewer (200 x 64 x 150: 1360 us against 1542)
  if (SUM && std::is_same<T, float>::value && split < 4 && most >= 4 &&
      mode_cost(S, true, pick->shape, 4) <= 1.06 * best)
    split = 4;
  return pick->run(P, S, split, st);
}

// ---------------------------------------------------------------- workspace

// Fields of the workspace: the axis-2 outputs of every node (2 M forward, 3 M
// adjoint) and the axis-3 outputs of a chunk of nodes (3 or 2 per node).  The
// chunk gets 3 fields, or as many as fit in 256 MiB: small grids run all their
// nodes in one launch per stage (their launches are what takes time), large
// ones fill the chip with a few nodes and keep the memory of one chunk.
static size_t chunk_nodes(const demag_plan* P, size_t elem) {
  const size_t per = 3 * field_size(P) * elem;
  size_t k = (size_t(256) << 20) / per;
  if (k < 1) k = 1;
  return k < (size_t)P->M ? k : (size_t)P->M;
}

size_t workspace_bytes(const demag_plan* P, demag_precision prec) {
  if (prec == DEMAG_TF32X3 || prec == DEMAG_BF16X3) return tc_workspace_bytes(P, prec);
  const size_t elem = prec == DEMAG_FP64 ? sizeof(double) : sizeof(float);
  return 3 * ((size_t)P->M + chunk_nodes(P, elem)) * field_size(P) * elem;
}

demag_status ensure_workspace(demag_plan* P, demag_precision prec) {
  if (prec == DEMAG_TF32X3 || prec == DEMAG_BF16X3) return tc_prepare(P, prec, 0);  // owns its buffers
  demag::Workspace& w = P->ws[prec];
  const size_t need = workspace_bytes(P, prec);
  if (w.base && w.bytes >= need) return DEMAG_OK;
  if (w.base) cudaFree(w.base);
  w.base = nullptr;
  w.bytes = 0;
  cudaError_t e = cudaMalloc(&w.base, need);
  if (e != cudaSuccess) return cuda_error(P, e, "workspace allocation");
  w.bytes = need;
  return DEMAG_OK;
}

// ---------------------------------------------------------------- forward and adjoint

// m (3 fields) -> phi = alpha P m; UV: 2 M fields, Y: 3 * chunk fields of type T
template <typename T>
static demag_status mode_forward(demag_plan* P, const float* m, float* phi, const ModeFactors<T>& F, T* UV, T* Y,
                                 int chunk, float alpha, cudaStream_t st) {
  const size_t N = field_size(P);
  const int M = P->M;
  chunk = (M + (M + chunk - 1) / chunk - 1) / ((M + chunk - 1) / chunk);  // the same number of launches, even chunks
  for (int k = 0; k < M; k += chunk) {
    const int nk = k + chunk < M ? chunk : M - k;
    ModeStage s3 = make_stage<T>(P, 0, F, k, nk, m, 0, Y, 3);
    for (int q = 0; q < 3; ++q) add_pair(P, s3, F, 2, q, q, q == 2 ? 1 : 0);
    cudaError_t e = launch_mode<T, 0>(P, s3, st);
    if (e != cudaSuccess) return cuda_error(P, e, "mode_kernel (axis 3)");
    ModeStage s2 = make_stage<T>(P, 1, F, k, nk, Y, 3, UV + (size_t)2 * k * N, 2);
    add_pair(P, s2, F, 1, 0, 1, 1);
    add_pair(P, s2, F, 1, 0, 2, 0);
    add_pair(P, s2, F, 1, 1, 0, 0);
    e = launch_mode<T, 1>(P, s2, st);
    if (e != cudaSuccess) return cuda_error(P, e, "mode_kernel (axis 2)");
  }
  ModeStage s1 = make_stage<T>(P, 2, F, 0, M, UV, 2, phi, 0);
  s1.alpha = alpha;
  add_pair(P, s1, F, 0, 0, 0, 0);
  add_pair(P, s1, F, 0, 0, 1, 1);
  cudaError_t e = launch_mode<T, 2>(P, s1, st);
  if (e != cudaSuccess) return cuda_error(P, e, "mode_kernel (axis 1)");
  return DEMAG_OK;
}

// y (1 field) -> g (3 fields).  Uniform grid: g^(q) = -P^(q) y with the forward
// factors (sign -1); non-uniform grid: the transposed factors and sign +1.
// Z: 3 M fields, Y: 2 * chunk fields
template <typename T>
static demag_status mode_adjoint(demag_plan* P, const float* y, float* g, const ModeFactors<T>& F, T* Z, T* Y,
                                 int chunk, float sign, cudaStream_t st) {
  const size_t N = field_size(P);
  const int M = P->M;
  chunk = (M + (M + chunk - 1) / chunk - 1) / ((M + chunk - 1) / chunk);
  for (int k = 0; k < M; k += chunk) {
    const int nk = k + chunk < M ? chunk : M - k;
    ModeStage s3 = make_stage<T>(P, 0, F, k, nk, y, 0, Y, 2);
    add_pair(P, s3, F, 2, 0, 0, 1);
    add_pair(P, s3, F, 2, 1, 0, 0);
    cudaError_t e = launch_mode<T, 0>(P, s3, st);
    if (e != cudaSuccess) return cuda_error(P, e, "mode_kernel (adjoint, axis 3)");
    ModeStage s2 = make_stage<T>(P, 1, F, k, nk, Y, 2, Z + (size_t)3 * k * N, 3);
    add_pair(P, s2, F, 1, 0, 1, 0);
    add_pair(P, s2, F, 1, 1, 1, 1);
    add_pair(P, s2, F, 1, 2, 0, 0);
    e = launch_mode<T, 1>(P, s2, st);
    if (e != cudaSuccess) return cuda_error(P, e, "mode_kernel (adjoint, axis 2)");
  }
  ModeStage s1 = make_stage<T>(P, 2, F, 0, M, Z, 3, g, 0);
  s1.alpha = sign;
  for (int q = 0; q < 3; ++q) add_pair(P, s1, F, 0, q, q, q == 0 ? 1 : 0);
  cudaError_t e = launch_mode<T, 2>(P, s1, st);
  if (e != cudaSuccess) return cuda_error(P, e, "mode_kernel (adjoint, axis 1)");
  return DEMAG_OK;
}

// The regions of the workspace and the chunk the axis-3 outputs have room for
template <typename T>
static demag_status run_forward(demag_plan* P, const float* m, float* phi, const ModeFactors<T>& F, float alpha,
                                demag_precision prec, cudaStream_t st) {
  const size_t N = field_size(P), M = P->M;
  T* UV = (T*)P->ws[prec].base;
  const size_t chunk = (M + 3 * chunk_nodes(P, sizeof(T))) / 3;
  return mode_forward<T>(P, m, phi, F, UV, UV + 2 * M * N, (int)(chunk < M ? chunk : M), alpha, st);
}
template <typename T>
static demag_status run_adjoint(demag_plan* P, const float* y, float* g, const ModeFactors<T>& F, float sign,
                                demag_precision prec, cudaStream_t st) {
  const size_t N = field_size(P), M = P->M;
  T* Z = (T*)P->ws[prec].base;
  const size_t chunk = 3 * chunk_nodes(P, sizeof(T)) / 2;
  return mode_adjoint<T>(P, y, g, F, Z, Z + 3 * M * N, (int)(chunk < M ? chunk : M), sign, st);
}

template <typename T> static ModeFactors<T> same_factors(const T* t) { return {{t, t, t}, {false, false, false}}; }

demag_status full_forward(demag_plan* P, const float* m, float* phi, demag_precision prec, cudaStream_t st) {
  if (prec == DEMAG_TF32X3 || prec == DEMAG_BF16X3) return tc_forward(P, m, phi, prec, st);
  demag_status s = ensure_dense_factors(P, prec, st);
  if (s != DEMAG_OK) return s;
  s = ensure_workspace(P, prec);
  if (s != DEMAG_OK) return s;
  if (prec == DEMAG_FP32) return run_forward<float>(P, m, phi, same_factors<float>(P->T32), 1.f, prec, st);
  return run_forward<double>(P, m, phi, same_factors<double>(P->T64), 1.f, prec, st);
}

// ---------------------------------------------------------------- analytic stray field (CUDA cores)

// h_d[p] = -dphi/dxi_p for p = 1..3: the forward chain with the axis-p factors
// replaced by the derivative ones (built from the derivative generators).
template <typename T>
static demag_status mode_field(demag_plan* P, const float* m, float* hd, const T* plain, T** deriv,
                               demag_precision prec, cudaStream_t st) {
  demag_status s = ensure_parts<T>(P, deriv, P->gend, true, false, st);
  for (int p = 0; p < 3 && s == DEMAG_OK; ++p) {
    ModeFactors<T> F = same_factors<T>(plain);
    F.base[p] = *deriv;
    F.deriv[p] = true;
    s = run_forward<T>(P, m, hd + p * field_size(P), F, -1.f, prec, st);
  }
  return s;
}

demag_status simt_field(demag_plan* P, const float* m, float* hd, demag_precision prec, cudaStream_t st) {
  demag_status s = ensure_dense_factors(P, prec, st);
  if (s == DEMAG_OK) s = ensure_workspace(P, prec);
  if (s == DEMAG_OK) s = ensure_field_generators(P, st);
  if (s != DEMAG_OK) return s;
  if (prec == DEMAG_FP32) return mode_field<float>(P, m, hd, P->T32, &P->T32d, prec, st);
  return mode_field<double>(P, m, hd, P->T64, &P->T64d, prec, st);
}

demag_status full_adjoint(demag_plan* P, const float* y, float* g, demag_precision prec, cudaStream_t st) {
  if (prec == DEMAG_TF32X3 || prec == DEMAG_BF16X3) {
    // the split-precision adjoint programs rely on P^T = -P (uniform grids)
    demag_status u = require_uniform(P, "demag_apply_adjoint in split precision");
    if (u != DEMAG_OK) return u;
    return tc_adjoint(P, y, g, prec, st);
  }
  demag_status s = P->nonuniform ? ensure_transposed_factors(P, prec, st) : ensure_dense_factors(P, prec, st);
  if (s != DEMAG_OK) return s;
  s = ensure_workspace(P, prec);
  if (s != DEMAG_OK) return s;
  const float sign = P->nonuniform ? 1.f : -1.f;
  if (prec == DEMAG_FP32)
    return run_adjoint<float>(P, y, g, same_factors<float>(P->nonuniform ? P->T32t : P->T32), sign, prec, st);
  return run_adjoint<double>(P, y, g, same_factors<double>(P->nonuniform ? P->T64t : P->T64), sign, prec, st);
}

static demag_status check_prec(demag_plan* P, demag_precision prec, const char* what) {
  if ((int)prec < 0 || (int)prec > 3) return set_error(P, DEMAG_EINVAL, "%s: unknown precision %d", what, (int)prec);
  return DEMAG_OK;
}

}  // namespace demag

using namespace demag;

extern "C" demag_status demag_reserve_workspace(demag_plan* P, demag_precision prec) {
  if (!P) return set_error(nullptr, DEMAG_EINVAL, "demag_reserve_workspace: plan is NULL");
  demag_status s = check_prec(P, prec, "demag_reserve_workspace");
  if (s != DEMAG_OK) return s;
  if (prec != DEMAG_TF32X3 && prec != DEMAG_BF16X3) {
    s = ensure_dense_factors(P, prec, 0);
    if (s != DEMAG_OK) return s;
  }
  s = ensure_workspace(P, prec);
  if (s != DEMAG_OK) return s;
  DEMAG_CUDA(P, cudaDeviceSynchronize());
  return DEMAG_OK;
}

extern "C" demag_status demag_apply_full(demag_plan* P, const float* m, float* phi, demag_precision prec,
                                         void* stream) {
  if (!P) return set_error(nullptr, DEMAG_EINVAL, "demag_apply_full: plan is NULL");
  demag_status s = check_prec(P, prec, "demag_apply_full");
  if (s != DEMAG_OK) return s;
  if (!m || !phi) return set_error(P, DEMAG_EINVAL, "demag_apply_full: NULL pointer");
  return full_forward(P, m, phi, prec, (cudaStream_t)stream);
}

extern "C" demag_status demag_apply_adjoint(demag_plan* P, const float* y, float* g, demag_precision prec,
                                            void* stream) {
  if (!P) return set_error(nullptr, DEMAG_EINVAL, "demag_apply_adjoint: plan is NULL");
  demag_status s = check_prec(P, prec, "demag_apply_adjoint");
  if (s != DEMAG_OK) return s;
  if (!y || !g) return set_error(P, DEMAG_EINVAL, "demag_apply_adjoint: NULL pointer");
  return full_adjoint(P, y, g, prec, (cudaStream_t)stream);
}

static demag_status check_batch(demag_plan* const* plans, const float* const* m, float* const* phi, int count,
                                demag_precision prec, const char* what) {
  if (count < 0 || (count > 0 && (!plans || !m || !phi)))
    return set_error(nullptr, DEMAG_EINVAL, "%s: bad arguments", what);
  if ((int)prec < 0 || (int)prec > (int)DEMAG_BF16X3)
    return set_error(nullptr, DEMAG_EINVAL, "%s: unknown precision %d", what, (int)prec);
  for (int i = 0; i < count; ++i) {
    if (!plans[i] || !m[i] || !phi[i]) return set_error(nullptr, DEMAG_EINVAL, "%s: NULL entry %d", what, i);
    const bool tc = prec == DEMAG_TF32X3 || prec == DEMAG_BF16X3;
    if (tc ? !tc_ready(plans[i], prec) : !plans[i]->ws[prec].base)
      return set_error(plans[i], DEMAG_EINVAL, "%s: plan %d has no workspace", what, i);
  }
  return DEMAG_OK;
}

extern "C" demag_status demag_apply_full_batched(demag_plan* const* plans, const float* const* m,
                                                 float* const* phi, int count, demag_precision prec,
                                                 void* stream) {
  demag_status cs = check_batch(plans, m, phi, count, prec, "demag_apply_full_batched");
  if (cs != DEMAG_OK) return cs;
  if (prec == DEMAG_TF32X3 || prec == DEMAG_BF16X3) {
    // each stage of a run of distinct plans is one grouped persistent launch;
    // a plan that repeats (it owns one set of intermediates) starts a new run
    int first = 0;
    for (int i = 1; i <= count; ++i) {
      bool repeat = false;
      for (int j = first; j < i && i < count; ++j) repeat = repeat || plans[j] == plans[i];
      if (i == count || repeat) {
        demag_status s = tc_forward_batched(plans + first, m + first, phi + first, i - first, prec,
                                            (cudaStream_t)stream);
        if (s != DEMAG_OK) return s;
        first = i;
      }
    }
    return DEMAG_OK;
  }
  for (int i = 0; i < count; ++i) {
    demag_status s = full_forward(plans[i], m[i], phi[i], prec, (cudaStream_t)stream);
    if (s != DEMAG_OK) return s;
  }
  return DEMAG_OK;
}

// ---------------------------------------------------------------- CUDA-graph form of the batched apply

struct demag_graph {
  std::vector<demag_plan*> plans;
  demag::TcBatch* batch = nullptr;  // grouped descriptors owned by this graph (tensor-core forms)
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  int kernels = 0;
};

extern "C" void demag_graph_destroy(demag_graph* g) {
  if (!g) return;
  if (g->exec) cudaGraphExecDestroy(g->exec);
  if (g->graph) cudaGraphDestroy(g->graph);
  tc_batch_destroy(g->batch);
  delete g;
}

extern "C" demag_status demag_graph_create_batched(demag_plan* const* plans, const float* const* m,
                                                   float* const* phi, int count, demag_precision prec,
                                                   demag_graph** out) {
  if (!out) return set_error(nullptr, DEMAG_EINVAL, "demag_graph_create_batched: out is NULL");
  *out = nullptr;
  demag_status s = check_batch(plans, m, phi, count, prec, "demag_graph_create_batched");
  if (s != DEMAG_OK) return s;
  if (count == 0) return set_error(nullptr, DEMAG_EINVAL, "demag_graph_create_batched: empty batch");
  for (int i = 0; i < count; ++i)
    for (int j = 0; j < i; ++j)
      if (plans[i] == plans[j])
        return set_error(plans[i], DEMAG_EINVAL, "demag_graph_create_batched: plan %d repeats plan %d", i, j);
  const bool tc = prec == DEMAG_TF32X3 || prec == DEMAG_BF16X3;
  demag_graph* g = new demag_graph();
  g->plans.assign(plans, plans + count);
  if (tc) {
    s = tc_batch_create(plans, count, prec, &g->batch);
    if (s != DEMAG_OK) {
      demag_graph_destroy(g);
      return s;
    }
  }
  cudaStream_t cs = nullptr;
  cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    demag_graph_destroy(g);
    return cuda_error(plans[0], e, "demag_graph_create_batched: stream");
  }
  // event timing would record into the graph: off while capturing
  std::vector<char> prof(count);
  std::vector<unsigned long long> before(count);
  for (int i = 0; i < count; ++i) {
    prof[i] = plans[i]->prof_on;
    plans[i]->prof_on = false;
    before[i] = plans[i]->launches;
  }
  e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    if (tc) {
      s = tc_batch_run(g->batch, m, phi, cs);
    } else {
      for (int i = 0; i < count && s == DEMAG_OK; ++i) s = full_forward(plans[i], m[i], phi[i], prec, cs);
    }
    cudaGraph_t graph = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(cs, &graph);
    g->graph = graph;
    if (s == DEMAG_OK && e2 != cudaSuccess) s = cuda_error(plans[0], e2, "demag_graph_create_batched: capture");
  } else {
    s = cuda_error(plans[0], e, "demag_graph_create_batched: begin capture");
  }
  // the capture launched nothing: move the recorded kernels out of the counters
  unsigned long long recorded = 0;
  for (int i = 0; i < count; ++i) {
    plans[i]->prof_on = prof[i];
    recorded += plans[i]->launches - before[i];
    plans[i]->launches = before[i];
  }
  g->kernels = (int)recorded;
  cudaStreamDestroy(cs);
  if (s == DEMAG_OK && g->graph) {
    e = cudaGraphInstantiate(&g->exec, g->graph, 0);
    if (e != cudaSuccess) s = cuda_error(plans[0], e, "demag_graph_create_batched: instantiate");
  }
  if (s != DEMAG_OK) {
    demag_graph_destroy(g);
    return s;
  }
  *out = g;
  return DEMAG_OK;
}

extern "C" demag_status demag_graph_launch(demag_graph* g, void* stream) {
  if (!g || !g->exec) return set_error(nullptr, DEMAG_EINVAL, "demag_graph_launch: graph is NULL");
  cudaError_t e = cudaGraphLaunch(g->exec, (cudaStream_t)stream);
  if (e != cudaSuccess) return cuda_error(g->plans[0], e, "demag_graph_launch");
  g->plans[0]->launches += (unsigned long long)g->kernels;
  return DEMAG_OK;
}

extern "C" int demag_graph_kernel_count(const demag_graph* g) { return g ? g->kernels : 0; }

// ---------------------------------------------------------------- allocation-free entry point
//
// demag_apply_full_noalloc serves callers that must not allocate device
// memory themselves or through this library: code that runs while a device
// memory pool owned by a host framework has reserved the GPU (a cudaMalloc
// from a library would fail or fragment it), latency-critical loops where
// an allocation would implicitly synchronise the device, and embedders whose
// plugin rules forbid allocation.  Everything this call needs beyond the
// caller's input and output (nodes, generators, factor parts and the
// intermediates of the mode-product chain) lives in one file-scope device
// array of fixed size, which every GPU that loads the library keeps until
// the process exits.  The arithmetic is that of demag_apply_full with
// DEMAG_FP32 (same kernels, same order).

namespace demag {

constexpr size_t kNoAllocBytes = size_t(32) << 20;  // 32 MiB of device scratch
constexpr int kNoAllocMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

static void* g_noalloc_addr[kNoAllocMaxDevices];
static std::mutex g_noalloc_mu;

// Device address of the scratch array on the current device.  Host code sees
// only a host-side stand-in for `g_noalloc_scratch`, so the address is asked
// from the runtime once per device (with that device current) and cached.
static demag_status noalloc_address(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(nullptr, e, "demag_apply_full_noalloc: cudaGetDevice");
  if (dev < 0 || dev >= kNoAllocMaxDevices)
    return set_error(nullptr, DEMAG_EUNSUPPORTED, "demag_apply_full_noalloc: device %d out of range", dev);
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_error(nullptr, e, "demag_apply_full_noalloc: cudaGetSymbolAddress");
    g_noalloc_addr[dev] = p;
  }
  *out = g_noalloc_addr[dev];
  return DEMAG_OK;
}

static size_t na_align(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace demag

extern "C" demag_status demag_apply_full_noalloc(const demag_grid_desc* d, const float* m, float* phi,
                                                 void* stream) {
  using namespace demag;
  if (!d || !m || !phi) return set_error(nullptr, DEMAG_EINVAL, "demag_apply_full_noalloc: NULL pointer");
  for (int p = 0; p < 3; ++p) {
    if (d->n[p] < 1) return set_error(nullptr, DEMAG_EINVAL, "n[%d] = %d must be >= 1", p, d->n[p]);
    if (!(d->h[p] > 0.0) || !std::isfinite(d->h[p]))
      return set_error(nullptr, DEMAG_EINVAL, "h[%d] must be positive and finite", p);
  }
  if (d->R < 5 || d->R % 2 == 0)
    return set_error(nullptr, DEMAG_EINVAL, "R = %d must be odd and >= 5 (R = 2M+1)", d->R);
  if ((d->R - 1) / 2 > kMaxTerms)
    return set_error(nullptr, DEMAG_EUNSUPPORTED, "R = %d exceeds 2*%d+1", d->R, kMaxTerms);
  if (!(d->c0 > 0.0) || !std::isfinite(d->c0))
    return set_error(nullptr, DEMAG_EINVAL, "c0 must be positive and finite");

  // the fields of a plan this call needs, kept on the host stack
  demag_plan P;
  snprintf(P.err, sizeof(P.err), "no error");
  P.R = d->R;
  P.M = (d->R - 1) / 2;
  P.c0 = d->c0;
  P.s = 0.0;
  P.nmax = 0;
  for (int p = 0; p < 3; ++p) {
    P.n[p] = d->n[p];
    P.h[p] = d->h[p];
    P.s = fmax(P.s, (double)d->n[p] * d->h[p]);
    P.nmax = d->n[p] > P.nmax ? d->n[p] : P.nmax;
  }
  P.tgroup = 0;
  for (int p = 0; p < 3; ++p) {
    P.hh[p] = P.h[p] / P.s;
    P.toff[p] = P.tgroup;
    P.tgroup += (size_t)P.n[p] * P.n[p];
  }
  P.glen = 2 * P.nmax - 1;
  const int M = P.M;
  const size_t N = (size_t)P.n[0] * P.n[1] * P.n[2];

  // scratch layout: nodes [3][M], scale [M], generators [M][2][3][glen] (FP64),
  // factor parts and the chain's fields Y (3) + U, V (2M) (FP32); the limit counts [M][2][sum n_p^2] entries
  // for the factors, about twice what their parts take
  const size_t b_nodes = na_align(sizeof(double) * 3 * M);
  const size_t b_scale = na_align(sizeof(double) * M);
  const size_t b_gen = na_align(sizeof(double) * (size_t)M * 6 * P.glen);
  const size_t b_fac = na_align(sizeof(float) * (size_t)M * 2 * P.tgroup);
  const size_t b_ws = na_align(sizeof(float) * (2 * (size_t)M + 3) * N);
  const size_t need = b_nodes + b_scale + b_gen + b_fac + b_ws;
  if (need > kNoAllocBytes)
    return set_error(nullptr, DEMAG_EUNSUPPORTED,
                     "demag_apply_full_noalloc: this grid needs %zu bytes of scratch, the fixed maximum is %zu "
                     "bytes (%d MiB); use demag_apply_full",
                     need, kNoAllocBytes, (int)(kNoAllocBytes >> 20));

  void* base = nullptr;
  demag_status s = noalloc_address(&base);
  if (s != DEMAG_OK) return s;
  unsigned char* at = static_cast<unsigned char*>(base);
  P.nodes = reinterpret_cast<double*>(at);
  P.scale = reinterpret_cast<double*>(at + b_nodes);
  P.gen64 = reinterpret_cast<double*>(at + b_nodes + b_scale);
  float* T = reinterpret_cast<float*>(at + b_nodes + b_scale + b_gen);
  // the factor parts take about half of the region of the limit above; on axes of at most three cells
  // their padding makes them larger than n_p^2, on grids far below the limit
  const size_t b_parts = na_align(sizeof(float) * factor_elems(&P));
  float* Y = reinterpret_cast<float*>(at + b_nodes + b_scale + b_gen + (b_parts > b_fac ? b_parts : b_fac));
  float* UV = Y + 3 * N;
  cudaStream_t st = (cudaStream_t)stream;

  // setup: every scratch region below is fully written before it is read,
  // so nothing has to be cleared between calls
  DEMAG_LAUNCH(&P, kFamSetup, st, nodes_kernel<<<(M + 63) / 64, 64, 0, st>>>(M, P.c0, kCPot * P.s, P.nodes, P.scale));
  DEMAG_LAUNCHED(&P, "nodes_kernel (allocation-free)");
  GridInfo g;
  for (int p = 0; p < 3; ++p) {
    g.n[p] = P.n[p];
    g.hh[p] = P.hh[p];
  }
  {
    long total = (long)M * 6 * P.glen;
    int blocks = (int)((total + 255) / 256);
    if (blocks > 152 * 32) blocks = 152 * 32;
    DEMAG_LAUNCH(&P, kFamSetup, st, generators_kernel<<<blocks, 256, 0, st>>>(M, P.glen, g, P.nodes, P.gen64));
    DEMAG_LAUNCHED(&P, "generators_kernel (allocation-free)");
  }
  s = build_factor_parts<float>(&P, P.gen64, false, false, T, st);
  if (s != DEMAG_OK) return s;

  // the mode-product chain of demag_apply_full (DEMAG_FP32), one node at a time
  return mode_forward<float>(&P, m, phi, same_factors<float>(T), UV, Y, 1, 1.f, st);
}
