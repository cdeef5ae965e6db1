// Batched dense kernels for the BDDC setup: a grouped GEMM (every batch
// item has its own sizes, offsets and leading dimensions) and the blocked
// Gauss-Jordan "sweep" over a leading range of pivots.
//
// Sweeping the pivots of the leading block A of [[A, B], [C, D]] yields
//   [[A^-1, A^-1 B], [-C A^-1, D - C A^-1 B]]
// in place.  With A = A_II this gives the Dirichlet inverse, the harmonic
// extension, the restriction operator and the Schur complement of
// Section 3.2 in one pass; sweeping a whole matrix inverts it.
//
// Pivot block k (rows/cols kk of width kb <= NB) is processed as
//   P = A_kk^-1 (a CTA or a cluster per matrix, Gauss-Jordan),
//   X = A[:, kk] with X[kk] = -I,   Y = P A[kk, :] with Y[:, kk] = P,
//   A[kk, :] = 0, A[:, kk] = 0,     A -= X Y   (grouped GEMM, K = kb),
// which is the rank-kb form of the sweep.  No pivoting: a pivot below
// tol * max|diag| (or non-finite) sets DEV_PIVOT in the status word.
#pragma once
#include <cooperative_groups.h>

#include <algorithm>
#include <memory>
#include <vector>

#include "common.h"
#include "oz_gemm.cuh"
#include "tc_gemm.cuh"

namespace cbddc {

struct GemmProb {
  int M, N, K;
  int lda, ldb, ldc;
  int64_t a, b, c;  // element offsets from the kernel's base pointers
  // FP64 products by integer slices: column k of op(A) is scaled by 2^(ks
  // kexp[ke + k]) and row k of op(B) by its inverse (0: no scaling)
  int ks = 0;
  int64_t ke = 0;
};

// FP32 setup GEMMs run on the tensor cores (tcgen05, split TF32) unless
// this is cleared (cbddc_set_tensor_cores).  FP64 lists run there as integer
// slices whatever it says (oz_gemm.cuh), but for the coarsest inverse under FP32
// level-2 operators, which has no digit scratch and uses the CUDA cores.
// tc_parts(sweep) is the number of TF32 parts per operand (2 or 3) for sweep
// updates and for the other products, read when a context is created.
bool tensor_cores_enabled();
bool tensor_cores_for(bool sweep);  // per kind of list (sweep updates / other products)
bool tc_sweep_ks1();                 // sweep updates accumulate one K-step per TMEM slice
bool tc_other_ks1();                 // the other products too
int tc_parts(bool sweep);

template <typename T> struct GemmCfg;
template <> struct GemmCfg<float> { static constexpr int BM = 128, BN = 128, BK = 16, TM = 8, TN = 8; };
template <> struct GemmCfg<double> { static constexpr int BM = 64, BN = 64, BK = 16, TM = 4, TN = 4; };

// C = alpha op(A) op(B) + beta C for every problem; one CTA per output
// tile, the tiles listed as {problem, tile row, tile column} (only tiles
// that exist, so problems of uneven size launch no empty CTAs).
// Row-major storage; op(A) = A^T reads A as K x M, op(B) = B^T reads B as N x K.
// A problem with K == 0 has no tiles and leaves C untouched (callers use
// beta = 1 there).
template <typename T, bool TA, bool TB>
__global__ void __launch_bounds__((GemmCfg<T>::BM / GemmCfg<T>::TM) * (GemmCfg<T>::BN / GemmCfg<T>::TN))
gemm_grouped_kernel(const int4* __restrict__ tiles, const GemmProb* __restrict__ probs, const T* __restrict__ A,
                    const T* __restrict__ B, T* __restrict__ C, T alpha, T beta) {
  constexpr int BM = GemmCfg<T>::BM, BN = GemmCfg<T>::BN, BK = GemmCfg<T>::BK;
  constexpr int TM = GemmCfg<T>::TM, TN = GemmCfg<T>::TN;
  constexpr int NT = (BM / TM) * (BN / TN);
  const int4 tl = tiles[blockIdx.x];
  const GemmProb p = probs[tl.x];
  const int m0 = tl.y * BM, n0 = tl.z * BN;
  if (m0 >= p.M || n0 >= p.N || p.K <= 0) return;
  __shared__ T As[BK][BM + 4];
  __shared__ T Bs[BK][BN + 4];
  const int tid = threadIdx.x;
  const int tx = tid % (BN / TN), ty = tid / (BN / TN);
  const T* Ab = A + p.a;
  const T* Bb = B + p.b;
  T acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
  for (int k0 = 0; k0 < p.K; k0 += BK) {
    // A tile (BM x BK) -> As[k][m]
#pragma unroll
    for (int t = tid; t < BM * BK; t += NT) {
      int m, k;
      if (TA) { k = t / BM; m = t % BM; } else { m = t / BK; k = t % BK; }
      const int gm = m0 + m, gk = k0 + k;
      T v = T(0);
      if (gm < p.M && gk < p.K) v = TA ? Ab[(int64_t)gk * p.lda + gm] : Ab[(int64_t)gm * p.lda + gk];
      As[k][m] = v;
    }
    // B tile (BK x BN) -> Bs[k][n]
#pragma unroll
    for (int t = tid; t < BN * BK; t += NT) {
      int n, k;
      if (TB) { n = t / BK; k = t % BK; } else { k = t / BN; n = t % BN; }
      const int gn = n0 + n, gk = k0 + k;
      T v = T(0);
      if (gn < p.N && gk < p.K) v = TB ? Bb[(int64_t)gn * p.ldb + gk] : Bb[(int64_t)gk * p.ldb + gn];
      Bs[k][n] = v;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      T a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[k][ty * TM + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[k][tx * TN + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  T* Cb = C + p.c;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int gm = m0 + ty * TM + i;
    if (gm >= p.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int gn = n0 + tx * TN + j;
      if (gn >= p.N) continue;
      T* cp = Cb + (int64_t)gm * p.ldc + gn;
      *cp = (beta == T(0)) ? alpha * acc[i][j] : alpha * acc[i][j] + beta * *cp;
    }
  }
}

// Fast path for C = alpha A B + beta C (both operands row-major, not
// transposed): tiles of (32 VEC) x (32 VEC) with VEC = 16 / sizeof(T) (128 x
// 128 for FP32, 64 x 64 for FP64), 256 threads, a 2 VEC x 2 VEC split
// micro-tile per thread.  K slices of 16 go global -> shared with 16-byte
// asynchronous copies (cp.async) through a 3-stage ring, so two slices are
// in flight while one is multiplied, with one barrier per slice.  Operands
// must start on 16-byte boundaries with leading dimensions that are
// multiples of VEC (checked on the host); copies past M, N or K read nothing
// and zero-fill.
template <typename T> struct VecT;
template <> struct VecT<float> { using V = float4; static constexpr int W = 4; };
template <> struct VecT<double> { using V = double2; static constexpr int W = 2; };

template <typename T>
__device__ inline void vstore4(T* dst, const typename VecT<T>::V& v);
template <>
__device__ inline void vstore4<float>(float* d, const float4& v) { d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w; }
template <>
__device__ inline void vstore4<double>(double* d, const double2& v) { d[0] = v.x; d[1] = v.y; }

template <typename T>
__device__ inline typename VecT<T>::V vmask(typename VecT<T>::V v, int valid);
template <>
__device__ inline float4 vmask<float>(float4 v, int valid) {
  if (valid < 4) v.w = 0.f;
  if (valid < 3) v.z = 0.f;
  if (valid < 2) v.y = 0.f;
  if (valid < 1) v.x = 0.f;
  return v;
}
template <>
__device__ inline double2 vmask<double>(double2 v, int valid) {
  if (valid < 2) v.y = 0.0;
  if (valid < 1) v.x = 0.0;
  return v;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, int src_bytes) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

template <typename T>
__global__ void __launch_bounds__(256, 2)
gemm_nn_kernel(const int4* __restrict__ tiles, const GemmProb* __restrict__ probs, const T* __restrict__ A,
               const T* __restrict__ B, T* __restrict__ C, T alpha, T beta) {
  using V = typename VecT<T>::V;
  constexpr int W = VecT<T>::W;
  constexpr int BM = 32 * W, BN = 32 * W, BK = 16, STAGES = 3;
  constexpr int HALF = BM / 2;
  constexpr int ACH = BK / W;            // 16-byte chunks per A row slice
  static_assert(BM * BK / W == 2 * 256 && BK * BN / W == 2 * 256, "two chunks of A and of B per thread");
  const int4 tl = tiles[blockIdx.x];
  const GemmProb p = probs[tl.x];
  const int m0 = tl.y * BM, n0 = tl.z * BN;
  if (m0 >= p.M || n0 >= p.N || p.K <= 0) return;
  __shared__ __align__(16) T As[STAGES][BM][BK + 4];   // [m][k]
  __shared__ __align__(16) T Bs[STAGES][BK][BN + 4];   // [k][n]
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const T* Ab = A + p.a;
  const T* Bb = B + p.b;
  // issue the copies of K slice kt into stage st (zero-fill outside M, N, K)
  auto load_slice = [&](int kt, int st) {
    const int k0 = kt * BK;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = tid + 256 * h;
      const int row = c / ACH, kq = (c % ACH) * W;
      const int gm = m0 + row, gk = k0 + kq;
      const int valid = (gm < p.M) ? max(0, min(W, p.K - gk)) : 0;
      const T* src = valid > 0 ? Ab + (int64_t)gm * p.lda + gk : Ab;
      cp_async16(&As[st][row][kq], src, valid * (int)sizeof(T));
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = tid + 256 * h;
      const int kr = c / (BN / W), nq = (c % (BN / W)) * W;
      const int gk = k0 + kr, gn = n0 + nq;
      const int valid = (gk < p.K) ? max(0, min(W, p.N - gn)) : 0;
      const T* src = valid > 0 ? Bb + (int64_t)gk * p.ldb + gn : Bb;
      cp_async16(&Bs[st][kr][nq], src, valid * (int)sizeof(T));
    }
  };
  const int kTiles = (p.K + BK - 1) / BK;
#pragma unroll
  for (int st = 0; st < STAGES - 1; ++st) {
    if (st < kTiles) load_slice(st, st);
    cp_async_commit();
  }
  // The C tile is prefetched into L2 now, so that the epilogue's reads of
  // C (beta != 0) do not wait on DRAM.
  T* Cb = C + p.c;
  const bool cvec = ((p.c % W) == 0) && ((p.ldc % W) == 0);
  if (beta != T(0)) {
#pragma unroll
    for (int i = 0; i < 2 * W; ++i) {
      const int gm = m0 + (i < W ? ty * W + i : HALF + ty * W + (i - W));
      if (gm < p.M && (tx & 7) == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int gn0 = n0 + h * HALF + tx * W;
          if (gn0 < p.N)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(Cb + (int64_t)gm * p.ldc + gn0));
        }
      }
    }
  }
  T acc[2 * W][2 * W];
#pragma unroll
  for (int i = 0; i < 2 * W; ++i)
#pragma unroll
    for (int j = 0; j < 2 * W; ++j) acc[i][j] = T(0);
  for (int kt = 0; kt < kTiles; ++kt) {
    cp_async_wait<STAGES - 2>();   // slice kt has landed (this thread's copies)
    __syncthreads();               // ... and everyone's; stage (kt-1)%S is free
    if (kt + STAGES - 1 < kTiles) load_slice(kt + STAGES - 1, (kt + STAGES - 1) % STAGES);
    cp_async_commit();
    const int st = kt % STAGES;
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      T a[2 * W], b[2 * W];
#pragma unroll
      for (int i = 0; i < W; ++i) {
        a[i] = As[st][ty * W + i][k];
        a[W + i] = As[st][HALF + ty * W + i][k];
      }
      vstore4<T>(b, *reinterpret_cast<const V*>(&Bs[st][k][tx * W]));
      vstore4<T>(b + W, *reinterpret_cast<const V*>(&Bs[st][k][HALF + tx * W]));
#pragma unroll
      for (int i = 0; i < 2 * W; ++i)
#pragma unroll
        for (int j = 0; j < 2 * W; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
  }
  cp_async_wait<0>();
#pragma unroll
  for (int i = 0; i < 2 * W; ++i) {
    const int gm = m0 + (i < W ? ty * W + i : HALF + ty * W + (i - W));
    if (gm >= p.M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gn0 = n0 + h * HALF + tx * W;
      T* cp = Cb + (int64_t)gm * p.ldc + gn0;
      if (cvec && gn0 + W <= p.N) {
        T v[W];
        if (beta != T(0)) vstore4<T>(v, *reinterpret_cast<const V*>(cp));
#pragma unroll
        for (int j = 0; j < W; ++j) v[j] = (beta == T(0)) ? alpha * acc[i][h * W + j] : alpha * acc[i][h * W + j] + beta * v[j];
        V o;
        if constexpr (W == 4) o = V{v[0], v[1], v[2], v[3]};
        else o = V{v[0], v[1]};
        *reinterpret_cast<V*>(cp) = o;
      } else {
#pragma unroll
        for (int j = 0; j < W; ++j) {
          if (gn0 + j >= p.N) break;
          const T v = alpha * acc[i][h * W + j];
          cp[j] = (beta == T(0)) ? v : v + beta * cp[j];
        }
      }
    }
  }
}

// Output tile edge of both GEMM kernels: 128 for FP32, 64 for FP64.
inline int gemm_tile(size_t esize) { return esize == 4 ? 128 : 64; }
static_assert(GemmCfg<float>::BM == 128 && GemmCfg<float>::BN == 128 && 32 * VecT<float>::W == 128, "tile");
static_assert(GemmCfg<double>::BM == 64 && GemmCfg<double>::BN == 64 && 32 * VecT<double>::W == 64, "tile");

// A list of grouped GEMM problems with its output tiles and host-side totals.
// FP32 lists also carry the plan of the tensor-core path: every problem's
// first row in the split operand arrays (op(A): M rows, op(B)^T: N rows, K
// padded to Kp), and, once bound to a scratch buffer, the four TMA maps.
struct GemmList {
  DVec<GemmProb> d;
  DVec<int4> tiles;  // {problem, tile row, tile column, 0}
  int n = 0, ntiles = 0;
  double flops = 0.0, bytes = 0.0;
  bool fast = true;  // every problem meets the vector-load alignment
  // tensor-core plan (FP32 only)
  bool tc_planned = false, tc_bound = false, presplit = false;
  int Kp = 0, maxM = 0, maxN = 0;
  int64_t rowsA = 0, rowsB = 0;
  DVec<tc::TcProb> tcp;
  DVec<tc::SplitProb> spa, spb;
  float* tc_base = nullptr;
  int* tc_status = nullptr;
  int np = 2;  // TF32 parts per operand
  tc::TcMaps maps;
  std::vector<GemmProb> h;  // host copy of the problems
  // integer-slice tensor-core plan (FP64)
  DVec<oz::Prob> ozp;
  DVec<oz::SplitProb> oza, ozb;
  DVec<int2> oz_ia, oz_ib;  // split work items
  DVec<int4> oz_tiles;
  std::vector<oz::Batch> oz_batches;
  unsigned char* oz_base = nullptr;
  int* oz_status = nullptr;
  const int* oz_kexp = nullptr;  // exponents along K
  std::unique_ptr<GemmList> panel;  // FP64 sweep step: Y = P A_kk as products of their own
  bool trans_a = false, trans_b = false;
  int tile_order = 0;
  // order 1: tiles of the largest problems (M N K) first, so that with
  // uneven subdomains the long tile runs of a persistent kernel start early
  void set(const std::vector<GemmProb>& v, size_t esize, bool ta = false, int order = 0, bool tb = false) {
    h = v;
    trans_a = ta;
    trans_b = tb;
    tile_order = order;
    n = (int)v.size();
    flops = bytes = 0.0;
    const int w = (int)(16 / esize);
    const int tile = gemm_tile(esize);
    fast = !ta;
    std::vector<int4> t;
    for (int i = 0; i < n; ++i) {
      const GemmProb& q = v[i];
      if (q.M <= 0 || q.N <= 0 || q.K <= 0) continue;
      flops += 2.0 * q.M * q.N * q.K;
      bytes += (double)esize * (2.0 * q.M * q.N + (double)q.K * (q.M + q.N));
      if (q.a % w || q.b % w || q.lda % w || q.ldb % w) fast = false;
      for (int tm = 0; tm < (int)cdiv(q.M, tile); ++tm)
        for (int tn = 0; tn < (int)cdiv(q.N, tile); ++tn) t.push_back(make_int4(i, tm, tn, 0));
    }
    if (order == 1) {
      auto work = [&](const int4& a) { return (double)v[a.x].M * v[a.x].N * v[a.x].K; };
      std::stable_sort(t.begin(), t.end(), [&](const int4& a, const int4& b) { return work(a) > work(b); });
    }
    ntiles = (int)t.size();
    d.upload(v);
    tiles.upload(t);
    tc_planned = tc_bound = false;
    if (esize == 4 && ntiles > 0 && n <= 65535) plan_tc(v);
    if (esize == 8 && ntiles > 0) plan_oz();
  }
  // FP64: batches of problems, or of blocks of whole tiles of a problem, whose
  // digits share a buffer of cap bytes (one tile row and column fit whatever the
  // cap), with the split work items (blocks of 32 rows) and the output tiles of
  // each
  void plan_oz(int64_t cap = oz::kBatchBytes) {
    std::vector<oz::Prob> pr;
    std::vector<oz::SplitProb> sa, sb;
    std::vector<int2> ia, ib;
    std::vector<int4> t;
    oz_batches.clear();
    auto work = [&](const int4& a) { return (double)pr[a.x].M * pr[a.x].N * pr[a.x].K; };
    auto close = [&] {
      if (oz_batches.empty()) return;
      oz::Batch& b = oz_batches.back();
      b.na = (int)ia.size() - b.a0;
      b.nb = (int)ib.size() - b.b0;
      b.nt = (int)t.size() - b.t0;
      if (tile_order == 1)
        std::stable_sort(t.begin() + b.t0, t.end(), [&](const int4& x, const int4& y) { return work(x) > work(y); });
    };
    for (const GemmProb& q : h) {
      if (q.M <= 0 || q.N <= 0 || q.K <= 0) continue;
      CB_CHECK(q.K <= 1 << 24, CBDDC_EINVAL, "dense product too long");
      const int Kp = (int)round_up(q.K, oz::BK);
      // rows of op(A) and columns of op(B) per block: all of them, or as many
      // rows as fit beside all columns, or half of the cap each
      const int64_t fit = cap / ((int64_t)oz::S * Kp * 2 + 8);
      int bm = q.M, bn = q.N;
      if (q.M + round_up(q.N, 16) > fit) {
        if (q.N > fit / 2) bn = (int)std::min<int64_t>(q.N, std::max<int64_t>(oz::BN, fit / 2 / oz::BN * oz::BN));
        bm = (int)std::min<int64_t>(q.M, std::max<int64_t>(oz::BM, (fit - round_up(bn, 16)) / oz::BM * oz::BM));
      }
      for (int m0 = 0; m0 < q.M; m0 += bm)
        for (int n0 = 0; n0 < q.N; n0 += bn) {
          const int M = std::min(bm, q.M - m0), N = std::min(bn, q.N - n0), i = (int)pr.size();
          bool fresh = oz_batches.empty();
          if (!fresh) {
            oz::Batch b = oz_batches.back();
            b.Kp = std::max(b.Kp, Kp);
            b.rowsA += M;
            b.rowsB += round_up(N, 16);
            fresh = b.bytes() > cap || b.rowsA >= INT32_MAX || b.rowsB >= INT32_MAX;
          }
          if (fresh) {
            close();
            oz::Batch b;
            b.a0 = (int)ia.size();
            b.b0 = (int)ib.size();
            b.t0 = (int)t.size();
            oz_batches.push_back(b);
          }
          oz::Batch& b = oz_batches.back();
          b.Kp = std::max(b.Kp, Kp);
          pr.push_back(oz::Prob{M, N, q.K, q.ldc, q.c + (int64_t)m0 * q.ldc + n0, (int)b.rowsA, (int)b.rowsB});
          sa.push_back(oz::SplitProb{M, M, q.K, q.lda, (int)b.rowsA, q.ks, q.a + (int64_t)m0 * (trans_a ? 1 : q.lda),
                                     q.ke});
          sb.push_back(oz::SplitProb{N, (int)round_up(N, 16), q.K, q.ldb, (int)b.rowsB, -q.ks,
                                     q.b + (int64_t)n0 * (trans_b ? q.ldb : 1), q.ke});
          b.rowsA += M;
          b.rowsB += round_up(N, 16);
          for (int k = 0; k < (int)cdiv(M, 32); ++k) ia.push_back(make_int2(i, k));
          for (int k = 0; k < (int)cdiv(N, 32); ++k) ib.push_back(make_int2(i, k));
          for (int tm = 0; tm < (int)cdiv(M, oz::BM); ++tm)
            for (int tn = 0; tn < (int)cdiv(N, oz::BN); ++tn) t.push_back(make_int4(i, tm, tn, 0));
        }
    }
    close();
    ozp.upload(pr);
    oza.upload(sa);
    ozb.upload(sb);
    oz_ia.upload(ia);
    oz_ib.upload(ib);
    oz_tiles.upload(t);
  }
  // device memory of the plan itself
  int64_t device_bytes() const {
    return (int64_t)(d.bytes() + tiles.bytes() + tcp.bytes() + spa.bytes() + spb.bytes() + ozp.bytes() + oza.bytes() +
                     ozb.bytes() + oz_ia.bytes() + oz_ib.bytes() + oz_tiles.bytes()) +
           (panel ? panel->device_bytes() : 0);
  }
  // bytes of digit scratch this list needs
  int64_t oz_bytes() const {
    int64_t m = 0;
    for (const auto& b : oz_batches) m = std::max(m, b.bytes());
    return m;
  }
  void bind_oz(unsigned char* base, int* status, const int* kexp = nullptr) {
    oz_base = base;
    oz_status = status;
    oz_kexp = kexp;
    for (auto& b : oz_batches) {
      b.maps.a = oz::encode_digits(reinterpret_cast<__half*>(base), b.rowsA, b.Kp, oz::BM);
      b.maps.b = oz::encode_digits(reinterpret_cast<__half*>(base + b.bytes_a()), b.rowsB, b.Kp, oz::BN);
    }
  }
  void plan_tc(const std::vector<GemmProb>& v) {
    std::vector<tc::TcProb> tp(n);
    std::vector<tc::SplitProb> sa(n), sb(n);
    int kmax = 0;
    rowsA = rowsB = 0;
    maxM = maxN = 0;
    for (int i = 0; i < n; ++i) {
      const GemmProb& q = v[i];
      const int M = std::max(q.M, 0), N = std::max(q.N, 0), K = std::max(q.K, 0);
      tp[i] = tc::TcProb{M, N, K, q.ldc, q.c, (int)rowsA, (int)rowsB};
      sa[i] = tc::SplitProb{K > 0 ? M : 0, K, q.lda, q.a, (int)rowsA};
      sb[i] = tc::SplitProb{K > 0 ? N : 0, K, q.ldb, q.b, (int)rowsB};
      rowsA += M;
      rowsB += N;
      kmax = std::max(kmax, K);
      maxM = std::max(maxM, M);
      maxN = std::max(maxN, N);
    }
    if (rowsA >= INT32_MAX || rowsB >= INT32_MAX) return;
    Kp = (int)round_up(std::max(kmax, 1), tc::BKC);
    tcp.upload(tp);
    spa.upload(sa);
    spb.upload(sb);
    tc_planned = true;
  }
  // floats of split operands this list needs
  int64_t tc_floats(int parts) const { return tc_planned ? parts * (rowsA + rowsB) * (int64_t)Kp : 0; }
  // Sweep updates whose operands the panel kernel writes already split:
  // op(A) = X at rows a / nb of the [rowsA][nb] hi/lo arrays, op(B)^T =
  // Y^T at rows b / nb of the [rowsB][nb] ones (panel offsets are multiples
  // of nb).
  void bind_presplit(int nb, int parts, float* const* Ap, int64_t rA, float* const* Bp, int64_t rB,
                     int* status) {
    if (ntiles == 0 || n > 65535) return;
    const std::vector<GemmProb>& v = h;
    std::vector<tc::TcProb> tp(n);
    for (int i = 0; i < n; ++i) {
      const GemmProb& q = v[i];
      tp[i] = tc::TcProb{std::max(q.M, 0), std::max(q.N, 0), std::max(q.K, 0), q.ldc, q.c, (int)(q.a / nb),
                         (int)(q.b / nb)};
    }
    tcp.upload(tp);
    Kp = nb;
    rowsA = rA;
    rowsB = rB;
    tc_status = status;
    np = parts;
    for (int q = 0; q < np; ++q) {
      maps.a[q] = tc::encode_kmajor(Ap[q], rA, nb);
      maps.b[q] = tc::encode_kmajor(Bp[q], rB, nb);
    }
    tc_planned = false;  // no split arrays in the shared scratch
    tc_bound = presplit = true;
  }
  // split arrays in the scratch: the parts of op(A) ([rowsA][Kp] each),
  // then those of op(B)^T ([rowsB][Kp] each)
  void bind_tc(float* base, int parts, int* status) {
    if (!tc_planned) return;
    tc_base = base;
    tc_status = status;
    np = parts;
    for (int q = 0; q < np; ++q) {
      maps.a[q] = tc::encode_kmajor(base + q * rowsA * Kp, rowsA, Kp);
      maps.b[q] = tc::encode_kmajor(base + np * rowsA * Kp + q * rowsB * Kp, rowsB, Kp);
    }
    tc_bound = true;
  }
};

// C = alpha op(A) op(B) + beta C for a bound FP32 list on the tensor cores:
// split both operands into the list's K-major hi/lo arrays, then one
// tcgen05 CTA per output tile.
template <bool TA, bool TB>
void launch_tc(const GemmList& g, const float* A, const float* B, float* C, float alpha, float beta,
               cudaStream_t s) {
  if (!g.presplit) {
    float* Ap = g.tc_base;
    float* Bp = Ap + g.np * g.rowsA * g.Kp;
    const dim3 ga(cdiv(g.maxM, 32) * (unsigned)(g.Kp / 32), g.n), gb(cdiv(g.maxN, 32) * (unsigned)(g.Kp / 32), g.n);
    // op(A) rows are A's rows unless TA; op(B)^T rows are B's rows when TB
    if (g.np == 3) {
      tc::tc_split_kernel<!TA, 3><<<ga, 256, 0, s>>>(g.spa.p, g.Kp, A, Ap, g.rowsA * g.Kp);
      CB_LAUNCH();
      tc::tc_split_kernel<TB, 3><<<gb, 256, 0, s>>>(g.spb.p, g.Kp, B, Bp, g.rowsB * g.Kp);
    } else {
      tc::tc_split_kernel<!TA, 2><<<ga, 256, 0, s>>>(g.spa.p, g.Kp, A, Ap, g.rowsA * g.Kp);
      CB_LAUNCH();
      tc::tc_split_kernel<TB, 2><<<gb, 256, 0, s>>>(g.spb.p, g.Kp, B, Bp, g.rowsB * g.Kp);
    }
    CB_LAUNCH();
  }
  // rank-64 sweep updates (two K chunks) are bound by C's traffic: one
  // operand stage and two C buffers; longer K: two stages and one C buffer
  // (three-part operands: one stage and two C buffers always)
  const int grid = tc::tc_grid(g.ntiles);
  // one K-step per TMEM slice (else a 32-wide K block per slice)
  const bool ks1 = g.presplit ? tc_sweep_ks1() : tc_other_ks1();
#define CB_TC_LAUNCH(NST, NCB, NP, KS)                                                              \
  tc::set_smem_attr<NST, NCB, NP, KS>(),                                                            \
  tc::tc_gemm_kernel<NST, NCB, NP, KS><<<grid, tc::TC_THREADS, tc::TcSmem<NST, NCB, NP>::bytes, s>>>( \
      g.tiles.p, g.ntiles, g.tcp.p, g.maps, C, alpha, beta, g.tc_status)
  if (g.np == 3) {
    if (ks1) CB_TC_LAUNCH(1, 2, 3, 1);
    else CB_TC_LAUNCH(1, 2, 3, 4);
  } else if (g.Kp <= 2 * tc::BKC) {
    if (ks1) CB_TC_LAUNCH(1, 2, 2, 1);
    else CB_TC_LAUNCH(1, 2, 2, 4);
  } else {
    if (ks1) CB_TC_LAUNCH(2, 1, 2, 1);
    else CB_TC_LAUNCH(2, 1, 2, 4);
  }
#undef CB_TC_LAUNCH
  CB_LAUNCH();
}

// C = sign op(A) op(B) (+ C) for a bound FP64 list: per batch, the digits of
// both operands, then one persistent tcgen05 kernel.
template <bool TA, bool TB>
void launch_oz(const GemmList& g, const double* A, const double* B, double* C, double alpha, double beta,
               cudaStream_t s) {
  CB_CHECK((alpha == 1.0 || alpha == -1.0) && (beta == 0.0 || beta == 1.0), CBDDC_EINVAL, "dense product factors");
  for (const oz::Batch& b : g.oz_batches) {
    __half* da = reinterpret_cast<__half*>(g.oz_base);
    __half* db = reinterpret_cast<__half*>(g.oz_base + b.bytes_a());
    int* ea = reinterpret_cast<int*>(g.oz_base + b.bytes_a() + b.bytes_b());
    int* eb = reinterpret_cast<int*>(g.oz_base + b.bytes_a() + b.bytes_b() + b.bytes_ea());
    oz::split_kernel<!TA><<<b.na, 256, 0, s>>>(g.oz_ia.p + b.a0, g.oza.p, b.Kp, A, g.oz_kexp, da, b.rowsA * b.Kp, ea);
    CB_LAUNCH();
    oz::split_kernel<TB><<<b.nb, 256, 0, s>>>(g.oz_ib.p + b.b0, g.ozb.p, b.Kp, B, g.oz_kexp, db, b.rowsB * b.Kp, eb);
    CB_LAUNCH();
    const int grid = tc::tc_grid(b.nt);
    if (beta == 0.0) oz::set_smem_attr<false>();
    else oz::set_smem_attr<true>();
    if (beta == 0.0)
      oz::gemm_kernel<false><<<grid, oz::THREADS, oz::SMEM, s>>>(g.oz_tiles.p + b.t0, b.nt, g.ozp.p, b.maps, ea, eb,
                                                                 C, alpha < 0.0, g.oz_status);
    else
      oz::gemm_kernel<true><<<grid, oz::THREADS, oz::SMEM, s>>>(g.oz_tiles.p + b.t0, b.nt, g.ozp.p, b.maps, ea, eb,
                                                                C, alpha < 0.0, g.oz_status);
    CB_LAUNCH();
  }
}

template <typename T, bool TA, bool TB>
void launch_gemm(const int4* tiles, int ntiles, const GemmProb* probs, const T* A, const T* B, T* C,
                 T alpha, T beta, cudaStream_t s, bool fast = false) {
  if (ntiles == 0) return;
  if (!TA && !TB && fast) {
    gemm_nn_kernel<T><<<ntiles, 256, 0, s>>>(tiles, probs, A, B, C, alpha, beta);
    CB_LAUNCH();
    return;
  }
  constexpr int BM = GemmCfg<T>::BM, BN = GemmCfg<T>::BN;
  constexpr int NT = (BM / GemmCfg<T>::TM) * (BN / GemmCfg<T>::TN);
  gemm_grouped_kernel<T, TA, TB><<<ntiles, NT, 0, s>>>(tiles, probs, A, B, C, alpha, beta);
  CB_LAUNCH();
}

// Launch of a whole list (timed as a setup GEMM when the timer follows
// them: FP32 lists in class SETUP_GEMM, FP64 ones in SETUP_GEMM_F64).
template <typename T, bool TA, bool TB>
void launch_list(const GemmList& g, const T* A, const T* B, T* C, T alpha, T beta, cudaStream_t s) {
  if (g.ntiles == 0) return;
  const int cls = sizeof(T) == 4 ? CBDDC_TIMER_SWEEP_GEMM : CBDDC_TIMER_SETUP_GEMM_F64;
  timer_begin(cls, s);
  if constexpr (sizeof(T) == 4) {
    if (g.tc_bound && tensor_cores_for(g.presplit)) {
      launch_tc<TA, TB>(g, A, B, C, alpha, beta, s);
      timer_end(cls, s, g.flops, g.bytes);
      return;
    }
  } else if (g.oz_base != nullptr) {
    launch_oz<TA, TB>(g, A, B, C, alpha, beta, s);
    timer_end(cls, s, g.flops, g.bytes);
    return;
  }
  // FP64 without digit scratch: a coarsest inverse (plain products only)
  if constexpr (sizeof(T) == 4 || (!TA && !TB))
    launch_gemm<T, TA, TB>(g.tiles.p, g.ntiles, g.d.p, A, B, C, alpha, beta, s, g.fast);
  else
    CB_CHECK(false, CBDDC_EINVAL, "transposed FP64 product without scratch");
  timer_end(cls, s, g.flops, g.bytes);
}

// --------------------------------------------------------------- sweeps
// Pivot block width of the sweeps: 64 (FP64 operators, and the FP32 default)
// or 128 (FP32; half the passes over each matrix for the same flops).
constexpr int SWEEP_NB = 64;
constexpr int SWEEP_NB_MAX = 128;

struct SweepDesc {
  int rows, cols, ld, p;  // matrix shape, leading dimension, pivots to sweep
  int64_t off;            // matrix offset
  int64_t offX;           // X panel offset (rows x NB, ld NB)
  int64_t offY;           // Y panel offset (NB x cols, ld ld)
  int64_t offP;           // diagonal inverse (NB x NB)
  int64_t ke = 0;         // FP64: first of its exponents (diag_exp_kernel)
};

// kexp[ke + i] = half the exponent of diagonal entry i: 2^kexp is the square
// root of the entry within a factor of two, the Jacobi scaling of row and
// column i (0 for entries that are zero or not finite).
static __global__ void diag_exp_kernel(const SweepDesc* __restrict__ desc, const double* __restrict__ mat,
                                       int* __restrict__ kexp) {
  const SweepDesc d = desc[blockIdx.y];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d.rows) return;
  const int e = oz::exp_key(mat[d.off + (int64_t)i * d.ld + i]);
  kexp[d.ke + i] = e == 0 || e == 2047 ? 0 : (e - 1023) >> 1;
}

// P = inverse of the kb x kb diagonal block of pivot step k, by Gauss-Jordan
// in the operator precision T: at pivot j
//   a[j][c] <- a[j][c] / p,  a[i][c] <- a[i][c] - a[i][j] a[j][c] / p (c != j),
//   a[i][j] <- -a[i][j] / p, a[j][j] <- 1 / p.
// Warp w keeps rows 8 w .. 8 w + 7 in registers, lane l their columns l, l +
// 32, ...  The warp that owns row j + 1 updates that row first, forms the
// reciprocal of its pivot and the scaled row, and publishes them (with the
// reciprocal in place of entry j + 1) in a double-buffered shared copy, as the
// owners of column j + 1 do with the column, while the other warps still
// update: one barrier per pivot, and one reciprocal instead of one per warp.
//
// One CTA per matrix, a chain of kb pivots.  FP64: bound by the FP64 pipe, 128
// warp instructions of 16 clocks per pivot of a 64-wide block (66 us at
// least); 95 us measured, 166 us when every warp formed the reciprocal behind
// the barrier.  FP32: bound by the chain (barrier, reciprocal, broadcast),
// 22 us against 39 us.
//
// CL > 1: the rows of one block go over a cluster of CL CTAs, RW rows per warp,
// and the owner of the next row writes it into every CTA's shared memory before
// the cluster barrier that takes the place of the CTA's.  The arithmetic of
// every entry is the same.  A single SM's FP64 pipe is then no longer the
// bound, but the chain of update, reciprocal and barrier: 79 us for FP64 blocks
// of 64 (one to a few matrices) against 95 us.  It pays while the matrices leave
// SMs idle (DIAG_CLUSTER * matrices <= 152); with 64 and 512 matrices both forms
// take the same time (99 and 94 us).
constexpr int DIAG_CLUSTER = 4;
template <int NB, int CL, int RW>
struct DiagThreads { static constexpr int value = 32 * NB / (RW * CL); };
template <typename T, int NB, int CL, int RW>
__global__ void __launch_bounds__(DiagThreads<NB, CL, RW>::value)
sweep_diag_kernel(const SweepDesc* __restrict__ desc, int k, T* __restrict__ mat, T* __restrict__ Pbuf,
                  int* __restrict__ status, double tol) {
  static_assert(RW % 2 == 0 && NB % (RW * CL) == 0, "rows per warp and CTA");
  constexpr int CW = NB / 32;  // columns per lane
  constexpr int WARPS = NB / (RW * CL);
  __shared__ __align__(16) T colb[2][NB];
  __shared__ T rowb[2][NB];
  const SweepDesc d = desc[blockIdx.x / CL];
  const int k0 = k * NB;
  if (k0 >= d.p) return;
  const int kb = min(NB, d.p - k0);
  // warp of the block's NB / RW, and its first row
  const int warp = (int)(blockIdx.x % CL) * WARPS + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int r0 = RW * warp;
  auto sync = [] {
    if constexpr (CL > 1) cooperative_groups::this_cluster().sync();
    else __syncthreads();
  };
  const T* A = mat + d.off + (int64_t)k0 * d.ld + k0;
  T a[RW][CW];
#pragma unroll
  for (int q = 0; q < RW; ++q)
#pragma unroll
    for (int v = 0; v < CW; ++v) {
      const int c = lane + 32 * v;
      a[q][v] = (r0 + q < kb && c < kb) ? A[(int64_t)(r0 + q) * d.ld + c] : T(0);
    }
  // scale of the pivots: largest |diagonal| of the block (every warp)
  double scale = 0.0;
  for (int i = lane; i < kb; i += 32) scale = fmax(scale, fabs((double)A[(int64_t)i * d.ld + i]));
  for (int o = 16; o > 0; o >>= 1) scale = fmax(scale, __shfl_xor_sync(0xffffffffu, scale, o));
  bool bad = false;
  // scaled row j (held by this warp in r) into buffer b
  auto publish_row = [&](const T* r, int j, int b) {
    T pv = T(0);
#pragma unroll
    for (int v = 0; v < CW; ++v)
      if (v == (j >> 5)) pv = r[v];
    pv = __shfl_sync(0xffffffffu, pv, j & 31);
    const T inv = T(1) / pv;
#pragma unroll
    for (int v = 0; v < CW; ++v) {
      const int c = lane + 32 * v;
      const T x = c == j ? inv : r[v] * inv;
      if constexpr (CL > 1) {
#pragma unroll
        for (int q = 0; q < CL; ++q) *cooperative_groups::this_cluster().map_shared_rank(&rowb[b][c], q) = x;
      } else {
        rowb[b][c] = x;
      }
    }
    if (!(fabs((double)pv) > tol * scale) || !isfinite((double)pv)) bad = true;
  };
  auto publish_col = [&](int j, int b) {
    if (lane == (j & 31)) {
#pragma unroll
      for (int v = 0; v < CW; ++v)
        if (v == (j >> 5)) {
#pragma unroll
          for (int q = 0; q < RW; ++q) colb[b][r0 + q] = a[q][v];
        }
    }
  };
  if constexpr (CL > 1) sync();  // every CTA of the cluster runs before its shared memory is written
  if (warp == 0) publish_row(a[0], 0, 0);
  publish_col(0, 0);
  for (int j0 = 0; j0 < kb; j0 += RW) {
#pragma unroll
    for (int u = 0; u < RW; ++u) {
      const int j = j0 + u;
      if (j >= kb) break;
      const int un = (u + 1) % RW;                  // row of j + 1 in its warp
      const int b = u & 1;
      const bool last = j + 1 >= kb;
      sync();
      T t[CW], col[RW];
      bool own[CW];                                 // this lane's column is j
#pragma unroll
      for (int v = 0; v < CW; ++v) {
        t[v] = rowb[b][lane + 32 * v];
        own[v] = lane + 32 * v == j;
      }
#pragma unroll
      for (int q = 0; q < RW; ++q) col[q] = colb[b][r0 + q];
      auto update = [&](int q) {
#pragma unroll
        for (int v = 0; v < CW; ++v) a[q][v] = (own[v] ? T(0) : a[q][v]) - col[q] * t[v];
      };
      if (warp == (j + 1) / RW && !last) {
        update(un);
        // (row j + 1 is never row j)
        publish_row(a[un], j + 1, b ^ 1);
#pragma unroll
        for (int q = 0; q < RW; ++q)
          if (q != un) update(q);
      } else {
#pragma unroll
        for (int q = 0; q < RW; ++q) update(q);
      }
      if (warp == j0 / RW) {
#pragma unroll
        for (int v = 0; v < CW; ++v) a[u][v] = t[v];
      }
      if (!last) publish_col(j + 1, b ^ 1);
    }
  }
  T* P = Pbuf + d.offP;
#pragma unroll
  for (int q = 0; q < RW; ++q)
#pragma unroll
    for (int v = 0; v < CW; ++v) {
      const int c = lane + 32 * v;
      if (c < kb && r0 + q < kb) P[(r0 + q) * NB + c] = a[q][v];
    }
  if (lane == 0 && bad) atomicOr(status, DEV_PIVOT);
}

// Builds X and Y panels and zeroes the pivot rows/columns, for indices
// [blockIdx.x*CH, +CH) of each matrix (as columns for Y, as rows for X).
// Reads and writes of different CTAs touch disjoint entries: the Y part reads
// pivot rows outside the pivot columns, the X part reads pivot columns outside
// the pivot rows (the pivot block itself is read only into Y entries that are
// replaced by P).  256 threads as 16 x 16; each forms NB / 16 rows of CH / 16
// columns of Y.  Shared memory (dynamic): P (NB x NB+1) and the chunk of pivot
// rows (NB x CH+4).
//
// Chunks of 64 read P once per 64 indices and give every P and pivot-row entry
// read from shared memory four uses; with chunks of 16, P (16 to 64 KB) was
// most of what a CTA read.  FP32, 64-wide blocks: 41 us per step against 50 us
// (48x48x12 slab), 121 us against 163 us (P2 ventricle, 582k unknowns).  Lists too
// short to fill the GPU with chunks of 64 (a single coarse matrix) keep 16, and
// so does FP64, which is bound by the FMAs of Y at 2 per SM and clock and ran
// slower in fewer, larger CTAs (262 us with 16, 359 us with 64, same slab).
template <typename T, int NB, int CH>
constexpr size_t panel_smem_bytes() {
  return sizeof(T) * ((size_t)NB * (NB + 1) + (size_t)NB * (CH + 4));
}

//
// NP > 0 (FP32 operators on the tensor cores): the panels are written as the
// K-major TF32 parts of the update GEMM's operands instead, X parts (rows x
// NB) at Xbuf, Xlo (, Xlo2) and Y^T parts (columns x NB) at Ybuf, Ylo (,
// Ylo2), with zeros beyond the kb pivots of a partial last block, so the
// update needs no separate split pass.
//
// NP < 0: Y's columns outside the pivots are already there (formed from the
// untouched pivot rows by a GEMM); the rest as above, without shared memory.
template <typename T, int NB, int NP, int CH>
__global__ void __launch_bounds__(256)
sweep_panel_kernel(const SweepDesc* __restrict__ desc, int k, T* __restrict__ mat,
                   const T* __restrict__ Pbuf, T* __restrict__ Xbuf, T* __restrict__ Ybuf,
                   T* __restrict__ Xlo, T* __restrict__ Ylo, T* __restrict__ Xlo2, T* __restrict__ Ylo2) {
  constexpr bool SPLIT = NP > 0, FORMED = NP < 0;
  constexpr int PER = NB * CH / 256, RY = NB / 16, CY = CH / 16, LDC = CH + 4;
  static_assert(NB % 16 == 0 && CH % 16 == 0, "16 x 16 threads");
  extern __shared__ __align__(16) unsigned char panel_smem[];
  T (*Ps)[NB + 1] = reinterpret_cast<T (*)[NB + 1]>(panel_smem);
  T (*col)[LDC] = reinterpret_cast<T (*)[LDC]>(panel_smem + sizeof(T) * NB * (NB + 1));
  const SweepDesc d = desc[blockIdx.y];
  const int k0 = k * NB;
  if (k0 >= d.p) return;
  const int kb = min(NB, d.p - k0);
  const int c0 = blockIdx.x * CH;
  if (c0 >= d.rows && c0 >= d.cols) return;
  const int cn = c0 < d.cols ? min(CH, d.cols - c0) : 0;   // columns in this chunk
  const int rn = c0 < d.rows ? min(CH, d.rows - c0) : 0;   // rows in this chunk
  const int tid = threadIdx.x;
  T* A = mat + d.off;
  const T* P = Pbuf + d.offP;
  T* X = Xbuf + d.offX;
  T* Y = Ybuf + d.offY;
  if (!FORMED && cn > 0) {
#pragma unroll 8
    for (int t = tid; t < NB * NB; t += 256) {
      const int r = t / NB, q = t % NB;
      Ps[r][q] = (r < kb && q < kb) ? P[r * NB + q] : T(0);
    }
    // pivot rows restricted to this column chunk (zero outside kb x cn)
#pragma unroll 8
    for (int t = tid; t < NB * CH; t += 256) {
      const int r = t / CH, cc = t % CH;
      col[r][cc] = (r < kb && cc < cn) ? A[(int64_t)(k0 + r) * d.ld + c0 + cc] : T(0);
    }
  }
  // X[i, :] = A[i, kk] (i outside kk), X[kk] = -I ; then A[i, kk] = 0
  if (rn > 0) {
    constexpr int XB = PER < 16 ? PER : 16;  // entries in flight per thread
#pragma unroll 1
    for (int u0 = 0; u0 < PER; u0 += XB) {
      T xv[XB];
#pragma unroll
      for (int u = 0; u < XB; ++u) {
        const int t = tid + 256 * (u0 + u), r = t / NB, q = t % NB, i = c0 + r;
        xv[u] = (r < rn && q < kb && !(i >= k0 && i < k0 + kb)) ? A[(int64_t)i * d.ld + k0 + q] : T(0);
      }
#pragma unroll
      for (int u = 0; u < XB; ++u) {
        const int t = tid + 256 * (u0 + u), r = t / NB, q = t % NB, i = c0 + r;
        if (SPLIT) {
          if (r < rn) {
            const bool piv = i >= k0 && i < k0 + kb;
            const T x = q < kb ? (piv ? ((i - k0 == q) ? T(-1) : T(0)) : xv[u]) : T(0);
            float parts[3];
            tc::split_tf32<NP == 3 ? 3 : 2>((float)x, parts);
            X[(int64_t)i * NB + q] = parts[0];
            Xlo[d.offX + (int64_t)i * NB + q] = parts[1];
            if (NP == 3) Xlo2[d.offX + (int64_t)i * NB + q] = parts[2];
            if (q < kb) A[(int64_t)i * d.ld + k0 + q] = T(0);
          }
        } else if (r < rn && q < kb) {
          const bool piv = i >= k0 && i < k0 + kb;
          X[(int64_t)i * NB + q] = piv ? ((i - k0 == q) ? T(-1) : T(0)) : xv[u];
          A[(int64_t)i * d.ld + k0 + q] = T(0);
        }
      }
    }
  }
  if (cn == 0) return;
  if constexpr (FORMED) {
    for (int t = tid; t < kb * CH; t += 256) {
      const int r = t / CH, c = t % CH, jg = c0 + c;
      if (c >= cn) continue;
      if (jg >= k0 && jg < k0 + kb) Y[(int64_t)r * d.ld + jg] = P[r * NB + jg - k0];
      A[(int64_t)(k0 + r) * d.ld + jg] = T(0);
    }
    return;
  }
  __syncthreads();
  // Y[r, j] = sum_q P[r][q] A[k0+q, j]  (j outside kk),  Y[:, kk] = P
  const int ty = tid / 16, tx = tid % 16;  // rows RY ty .., columns tx + 16 x
  T acc[RY][CY];
#pragma unroll
  for (int i = 0; i < RY; ++i)
#pragma unroll
    for (int x = 0; x < CY; ++x) acc[i][x] = T(0);
#pragma unroll 4
  for (int q = 0; q < kb; ++q) {
    T cq[CY];
#pragma unroll
    for (int x = 0; x < CY; ++x) cq[x] = col[q][tx + 16 * x];
#pragma unroll
    for (int i = 0; i < RY; ++i) {
      const T pq = Ps[RY * ty + i][q];
#pragma unroll
      for (int x = 0; x < CY; ++x) acc[i][x] = fma(pq, cq[x], acc[i][x]);
    }
  }
#pragma unroll
  for (int x = 0; x < CY; ++x) {
    const int c = tx + 16 * x;
    if (c >= cn) continue;
    const int jg = c0 + c;
    const bool pivc = jg >= k0 && jg < k0 + kb;
#pragma unroll
    for (int i = 0; i < RY; ++i) {
      const int r = RY * ty + i;
      if (SPLIT) {
        // Y^T row jg, K index r (zero beyond kb)
        const T y = r < kb ? (pivc ? Ps[r][jg - k0] : acc[i][x]) : T(0);
        float parts[3];
        tc::split_tf32<NP == 3 ? 3 : 2>((float)y, parts);
        Y[(int64_t)jg * NB + r] = parts[0];
        Ylo[d.offY + (int64_t)jg * NB + r] = parts[1];
        if (NP == 3) Ylo2[d.offY + (int64_t)jg * NB + r] = parts[2];
        if (r < kb) A[(int64_t)(k0 + r) * d.ld + jg] = T(0);
        continue;
      }
      if (r >= kb) continue;
      Y[(int64_t)r * d.ld + jg] = pivc ? Ps[r][jg - k0] : acc[i][x];
      A[(int64_t)(k0 + r) * d.ld + jg] = T(0);
    }
  }
}

}  // namespace cbddc
