// Grouped FP64 GEMM on the fifth-generation tensor cores, for the dense
// contractions of FP64 local operators and of the FP64 coarse inverse.
//
// FP64 FMAs run at about 2 per SM and clock on this part (1.2 TFLOP/s), so a
// product formed by them costs a thousand times what the FP16 tensor pipe
// needs per multiplication.  The products are therefore formed from exact
// integer slices (the error-free splitting of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication and its applications", Numer.
// Algorithms 59, 2012):
//
//   * column k of op(A) is multiplied by a power of two and row k of op(B)
//     divided by it (exact: exponents are integers here), chosen by the caller
//     from the diagonal of the matrix that k runs over;
//   * every row of op(A) and every column of op(B) then gets one exponent e
//     with |x| < 2^e, and x = 2^(e - 62) Q with an integer |Q| <= 2^62 (entries
//     at least 2^-10 of the row's largest are exact, the others round at
//     2^-63 of it);
//   * Q = sum_i d_i 512^(6 - i), i = 0..6, with balanced digits |d_i| <= 256,
//     which FP16 holds exactly;
//   * the product keeps the digit pairs with i + j <= 6 (28 of 49; the
//     dropped ones are below 2^-63 of the leading one).  The pairs of one
//     order i + j = k over a K block of 64 accumulate in one TMEM tile:
//     every sum is an integer below 2^22 (k + 1), so the FP32 accumulator is
//     exact up to order 3, and its truncation in the higher orders (only
//     possible if all digits are extremal) is below 2^-60;
//   * the epilogue adds the order sums of every K block in two 64-bit
//     integers (exact) and rounds once to FP64.
//
// Errors against extended precision of inverses by Gauss-Jordan sweeps of
// elasticity matrices (Q1 and Q2 slabs, P1 and P2 ventricles, 210 to 369 unknowns,
// root mean square over five states): 0.93, 0.57, 1.03 and 0.80 times those of the
// FP64 FMA kernel (single states: 0.4 to 1.4 times).  With six slices (54 bits)
// single states were 2.1, 2.4 and 1.1 times as far off (Q1, Q2, P1), which is why
// there are seven.
//
// The powers of two along K (Jacobi scaling) keep that so for graded matrices.
// FMAs do not see a diagonal scaling between the operands, but entries held
// relative to the largest of their row lose digits by it: a sweep multiplies
// columns of size d_i d_k by rows of size d_j / d_k.  Emulated on a Q1 slab
// tangent of 300 unknowns scaled on both sides by random factors from 1 to 10^3,
// 10^6 and 10^12, the errors of the inverse against extended precision are 1.3,
// 250 and 10^8 times an FP64 sweep's without these powers, and 0.8, 1.1 and 1.0
// times with them; those of E, S, Phi and S Phi up to 1.7 10^9 times without and
// at most 1.2 times with them.
//
// A row or column that holds an infinity or a NaN makes its whole row or
// column of the product NaN (an FMA chain gives NaN or an infinity there).
#pragma once
#include <cuda_fp16.h>

#include "tc_gemm.cuh"

namespace cbddc {
namespace oz {

constexpr int S = 7;               // slices
constexpr int DB = 9;              // bits per slice (balanced digits, |d| <= 256)
constexpr int BM = 128, BN = 64;   // output tile
constexpr int BK = 64;             // K block: one 128-byte swizzle row of FP16
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;
constexpr int EPI = 16;            // epilogue warps
constexpr int THREADS = 64 + 32 * EPI;  // producer, MMA issuer, epilogue
constexpr int SLOTS = 8;           // TMEM tiles of BN columns
constexpr int SMEM = S * (A_BYTES + B_BYTES) + 1024 /* alignment */ + 512 /* barriers */;
static_assert(SMEM <= 232448, "shared memory per CTA");
constexpr int EXP_NAN = 0x7fffff;  // row exponent of a row with a non-finite entry

// kind::f16 instruction descriptor: D = F32 (bits 4-5), A = B = F16 (0),
// both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28.
constexpr uint32_t kIdescF16 = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(kIdescF16), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(tc::smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(tc::smem_u32(bar))
      : "memory");
}

// 16 consecutive TMEM columns of this warp's 32 lanes (one row per thread),
// as integers (the order sums are integers).
__device__ __forceinline__ void tmem_ld16i(uint32_t taddr, int* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __float2int_rn(__uint_as_float(r[i]));
}

// ------------------------------------------------------------------- split
// One operand of a problem: output row r (< rows) holds op(X)(r, 0:K), and rows
// up to out_rows hold zeros.  (op(B) is padded to the epilogue's groups of 16
// columns, which are shifted together: with the next problem's rows there, the
// last bits of a product would depend on it.)
struct SplitProb {
  int rows, out_rows, K, ld;
  int r0;       // first output row
  int ks;       // op(X)(:, k) is scaled by 2^(ks kexp[ke + k]); 0: not scaled
  int64_t off, ke;
};

// Exponent key of an FP64 value: its biased exponent (1 for subnormal
// numbers, whose value is below 2^-1021), 0 for zero, 2047 for inf and NaN.
__device__ __forceinline__ int exp_key(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff, e = hi >> 20;
  return e > 0 ? e : (hi | __double2loint(x)) != 0 ? 1 : 0;
}
constexpr int KEY_NONE = -(1 << 20), KEY_NAN = 1 << 20;  // keys of rows that are all zero, or not finite

// The seven digits of x 2^shift relative to the row's largest key (|x
// 2^shift| < 2^(key - 1022)), by integer shifts: no FP64 instruction.
__device__ __forceinline__ void digits(double x, int shift, int key, short* d) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffLL;
  if (e) m |= 1LL << 52;
  const int s = m == 0 ? 64 : key - shift - (e > 1 ? e : 1);  // >= 0
  long long q;
  if (s <= 9) q = m << (9 - s);
  else if (s < 64) q = (m + (1LL << (s - 10))) >> (s - 9);
  else q = 0;
  if (b < 0) q = -q;
#pragma unroll
  for (int i = S - 1; i > 0; --i) {
    const int low = (int)(((unsigned)q + 256u) & 511u) - 256;
    d[i] = (short)low;
    q = (q - low) >> DB;
  }
  d[0] = (short)q;
}

// Eight consecutive K entries of a row as FP16 digits, 16 bytes per slice.
__device__ __forceinline__ void store_digits8(const double* v, const int* shift, int key, __half* out,
                                              int64_t slice_stride) {
  uint32_t w[S][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    short a[S], b[S];
    digits(v[2 * p], shift[2 * p], key, a);
    digits(v[2 * p + 1], shift[2 * p + 1], key, b);
#pragma unroll
    for (int i = 0; i < S; ++i) {
      const __half2 h = __halves2half2(__short2half_rn(a[i]), __short2half_rn(b[i]));
      w[i][p] = *reinterpret_cast<const uint32_t*>(&h);
    }
  }
#pragma unroll
  for (int i = 0; i < S; ++i)
    *reinterpret_cast<uint4*>(out + i * slice_stride) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// Split of one operand into K-major digit arrays [slice][row][Kp] (FP16) and
// row exponents.  Work items {problem, block of 32 rows}; 256 threads.
// KMAJ: op(X)(r, k) = X[off + r ld + k]: eight threads per row, each eight
// consecutive k.  Otherwise X[off + k ld + r]: the 32 rows of the block run
// along the lanes (coalesced reads), each warp takes eight k, and the block goes
// through shared memory to the same eight threads per row, so that the digits
// of a row leave as 128 consecutive bytes (written by the reading threads, 16
// bytes per row and warp, they took 47 us per step of the 48x48x12 slab, now
// 31 us).  Two passes over the rows (largest exponent, digits); with K <= 64
// the entries stay in registers.  Bound by its memory traffic: 8 bytes read and
// 14 written per entry.
template <bool KMAJ>
__global__ void __launch_bounds__(256)
split_kernel(const int2* __restrict__ items, const SplitProb* __restrict__ probs, int Kp,
             const double* __restrict__ X, const int* __restrict__ kexp, __half* __restrict__ out,
             int64_t slice_stride, int* __restrict__ exps) {
  __shared__ int keys[8][32];
  __shared__ double block[KMAJ ? 1 : 32][65];
  const int2 it = items[blockIdx.x];
  const SplitProb q = probs[it.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = (int)(threadIdx.x >> 3), grp = (int)(threadIdx.x & 7);  // as written
  const int rl = KMAJ ? row : lane;   // row of the block, as read
  const int kg = KMAJ ? grp : warp;   // group of eight k, as read
  const int r = it.y * 32 + rl;
  const bool in = r < q.rows;
  const double* src = X + q.off + (KMAJ ? (int64_t)r * q.ld : (int64_t)r);
  const int64_t ks = KMAJ ? 1 : q.ld;
  double v[8];
  int sh[8];  // powers of two of eight k from group g on
  auto shifts = [&](int k0, int g) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + 8 * g + u;
      sh[u] = q.ks != 0 && k < q.K ? q.ks * __ldg(kexp + q.ke + k) : 0;
    }
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + 8 * kg + u;
      v[u] = (in && k < q.K) ? __ldg(src + k * ks) : 0.0;
    }
  };
  int key = KEY_NONE;
  for (int k0 = 0; k0 < q.K; k0 += 64) {
    load(k0);
    shifts(k0, kg);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = exp_key(v[u]);
      key = max(key, e == 0 ? KEY_NONE : e == 2047 ? KEY_NAN : e + sh[u]);
    }
  }
  if (KMAJ) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
  } else {
    keys[warp][lane] = key;
    __syncthreads();
    key = KEY_NONE;
#pragma unroll
    for (int w = 0; w < 8; ++w) key = max(key, keys[w][row]);
  }
  const int rw = it.y * 32 + row;  // row written
  const bool out_in = rw < q.out_rows;
  // (a row of zeros takes any exponent)
  if (out_in && grp == 0) exps[q.r0 + rw] = key == KEY_NAN ? EXP_NAN : key == KEY_NONE ? 0 : key - 1022;
  __half* dst = out + (int64_t)(q.r0 + rw) * Kp + 8 * grp;
  for (int k0 = 0; k0 < Kp; k0 += 64) {
    if (q.K > 64) load(k0);
    else if (k0 > 0) {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = 0.0;
    }
    if (!KMAJ) {
      if (k0 > 0) __syncthreads();  // the block of the last pass is read
#pragma unroll
      for (int u = 0; u < 8; ++u) block[lane][8 * warp + u] = v[u];
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = block[row][8 * grp + u];
    }
    if (q.K > 64 || !KMAJ) shifts(k0, grp);
    if (out_in) store_digits8(v, sh, key, dst + k0, slice_stride);
  }
}

// (hi 2^27 + lo) 2^(e - sh) with e outside the range of the exponent field
// arithmetic, a NaN row or column, or more than 2^27 blocks' worth of shift:
// kept out of the unrolled epilogue.
static __device__ __noinline__ double slow_value(long long hi, long long lo, int sh, int e, int negate) {
  if (e > EXP_NAN / 2) return __longlong_as_double(0x7ff8000000000000LL);
  const long long v = (sh > 27 ? hi >> (sh - 27) : hi << (27 - sh)) + (lo >> sh);
  return scalbn((double)(negate ? -v : v), e);
}

// -------------------------------------------------------------------- GEMM
struct Prob {
  int M, N, K, ldc;
  int64_t c;
  int ar, br;  // first rows in the digit arrays of op(A) and op(B)^T
};

struct Maps {
  CUtensorMap a, b;
};

// Persistent grouped GEMM: CTA b takes the tiles b, b + gridDim.x, ... of the
// list ({problem, tile row, tile column}), each C = sign A B (+ C).
//
// Warp roles as in the TF32 kernel: warp 0 streams the digit tiles of a K
// block (seven of A, seven of B, 168 KB, one stage, a barrier per slice);
// warp 1 issues 28 x 4 MMAs (M = 128, N = 64, K = 16) per K block, one TMEM
// tile per order out of a ring of eight; warps 2-17 (warp w: TMEM lanes 32 (w
// mod 4).., columns 16 ((w - 2) / 4)..) add the order sums into 64-bit integers
// and free the tile.  At the end of an output tile each thread converts the
// 16 columns of its row to FP64 and adds them to C in whole 32-byte sectors
// (the row was brought into the L2 while the MMAs ran).  The orders run from
// the highest down, so that slice k of both operands is free for the next K
// block after order k and most of its loads hide behind the remaining MMAs.
//
// Cost of a tile of a rank-64 update: 112 MMAs of about 70 clocks (4.1 us),
// and beside them in the epilogue 7 float to integer conversions (16 per
// clock) and two FP64 instructions per entry (2 per clock).  Measured: 6.3 us
// per tile on 8192^2 x 64 (338 us, 25 TFLOP/s, 3.2 TB/s of C; the FP64 FMA
// kernel ran at 1.1 TFLOP/s), 4.3 us per K block on 2048^2 x 768 (31 TFLOP/s).
// A C whose leading dimension is no multiple of four goes entry by entry
// (1390 us on 8192^2 x 64).  Eight
// epilogue warps of 32 columns took 11 us per tile (two warps per scheduler do
// not cover the latencies), and adding to C by bulk reductions in the L2 12 us
// (they queue in front of the operand loads).
template <bool ADD>
__global__ void __launch_bounds__(THREADS, 1)
gemm_kernel(const int4* __restrict__ tiles, int ntiles, const Prob* __restrict__ probs,
            const __grid_constant__ Maps maps, const int* __restrict__ expA, const int* __restrict__ expB,
            double* __restrict__ C, int negate, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = tc::smem_u32(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (base & 1023u)) & 1023u);
  uint8_t* sA = smem;
  uint8_t* sB = smem + S * A_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * (A_BYTES + B_BYTES));  // [S]
  uint64_t* empty = full + S;        // [S]
  uint64_t* sfull = empty + S;       // [SLOTS]
  uint64_t* sempty = sfull + SLOTS;  // [SLOTS]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sempty + SLOTS);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  // the warp number is the same in every lane, and the shuffle says so: the
  // MMA warp's loop below then keeps its descriptors in uniform registers
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int ntl = ntiles > (int)blockIdx.x ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < SLOTS; ++i) {
      tc::mbar_init(&sfull[i], 1);
      tc::mbar_init(&sempty[i], EPI);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tmem_slot)),
                 "r"(SLOTS * BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  int issued = 0;  // slice copies the producer issued
  if (warp == 0) {
    if (lane == 0) {
      int b = 0;
      bool ok = true;
      for (int i = 0; i < ntl && ok && !*(volatile int*)abort_flag; ++i) {
        const int4 tl = tiles[blockIdx.x + i * gridDim.x];
        const Prob p = probs[tl.x];
        const int nk = (p.K + BK - 1) / BK;
        const int ya = p.ar + tl.y * BM, yb = p.br + tl.z * BN;
        for (int c = 0; c < nk; ++c, ++b) {
          // slices in the order in which the MMAs free them
          for (int q = S - 1; q >= 0; --q) {
            if (b > 0 && !tc::mbar_wait(&empty[q], (b - 1) & 1)) {
              atomicExch(abort_flag, 1);
              ok = false;
              break;
            }
            tc::mbar_expect_tx(&full[q], A_BYTES + B_BYTES);
            tma_load_3d(sA + q * A_BYTES, &maps.a, c * BK, ya, q, &full[q]);
            tma_load_3d(sB + q * B_BYTES, &maps.b, c * BK, yb, q, &full[q]);
            ++issued;
          }
          if (!ok) break;
        }
      }
    }
  } else if (warp == 1) {
    // The whole warp walks the loop and one lane issues: with the loop under
    // a single lane the operands of every MMA pass through vector registers,
    // which cost about 100 clocks per MMA whatever its N.
    int b = 0, g = 0;  // K blocks and TMEM tiles of this CTA so far
    bool ok = true;
    const uint64_t da0 = tc::sw128_desc(tc::smem_u32(sA)), db0 = tc::sw128_desc(tc::smem_u32(sB));
    for (int i = 0; i < ntl && ok && !tc::warp_aborted(abort_flag); ++i) {
      const int4 tl = tiles[blockIdx.x + i * gridDim.x];
      const int nk = (probs[tl.x].K + BK - 1) / BK;
      for (int c = 0; c < nk && ok; ++c, ++b) {
        for (int q = S - 1; q >= 0 && ok; --q) ok = tc::warp_wait(&full[q], b & 1);
        // orders from the highest down: slice k is free after order k
#pragma unroll
        for (int k = S - 1; k >= 0; --k, ++g) {
          const int a = g % SLOTS;
          if (!ok) break;
          if (g >= SLOTS && !tc::warp_wait(&sempty[a], (g / SLOTS - 1) & 1)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t acc = tmem + (uint32_t)(a * BN);
          if (tc::elect_one()) {
            // descriptors differ in their address field only (16-byte units)
#pragma unroll
            for (int x = 0; x <= k; ++x) {
#pragma unroll
              for (int kk = 0; kk < BK / 16; ++kk)
                mma_f16(acc, da0 + (uint32_t)(x * (A_BYTES / 16) + 2 * kk),
                        db0 + (uint32_t)((k - x) * (B_BYTES / 16) + 2 * kk), (x | kk) ? 1u : 0u);
            }
            tc::mma_commit(&sfull[a]);
            tc::mma_commit(&empty[k]);
          }
          __syncwarp();
        }
      }
    }
    if (!ok && lane == 0) atomicExch(abort_flag, 1);
  } else {
    const int wq = warp & 3, quarter = (warp - 2) >> 2;
    const int wrow0 = 32 * wq, col0 = 16 * quarter;
    int g = 0;
    bool ok = true;
    for (int i = 0; i < ntl && ok; ++i) {
      const int4 tl = tiles[blockIdx.x + i * gridDim.x];
      const Prob p = probs[tl.x];
      const int m0 = tl.y * BM + wrow0, n0 = tl.z * BN + col0;
      const int nk = (p.K + BK - 1) / BK;
      const bool row_in = m0 + lane < p.M;
      double* crow = C + p.c + (int64_t)(m0 + lane) * p.ldc + n0;
      // this row's 128 bytes of C into L2 while the MMAs run
      if (ADD && row_in && n0 < p.N) asm volatile("prefetch.global.L2 [%0];" ::"l"(crow));
      // exact sums over the K blocks: orders 0..3 in units of 512^-3, orders
      // 4..6 in units of 512^-6 of the leading digit product (below 2^52 and
      // 2^44 per block)
      long long hi[16], lo[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) hi[q] = lo[q] = 0;
      for (int c = 0; c < nk && ok; ++c) {
#pragma unroll
        for (int k = S - 1; k >= 0; --k, ++g) {
          const int a = g % SLOTS;
          if (!tc::warp_wait(&sfull[a], (g / SLOTS) & 1) || tc::warp_aborted(abort_flag)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t tcol = tmem + (uint32_t)(a * BN) + ((uint32_t)wrow0 << 16) + (uint32_t)col0;
          int v[16];
          tmem_ld16i(tcol, v);
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            if (k < 4) hi[q] += (long long)v[q] * (1 << (DB * (3 - k)));
            else lo[q] += (long long)v[q] * (1 << (DB * (6 - k)));
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&sempty[a])) : "memory");
        }
      }
      if (!ok) {
        atomicExch(abort_flag, 1);
        break;
      }
      // Each sum hi 2^27 + lo becomes one 64-bit integer, shifted right by
      // sh so that the row's largest keeps 62 bits (FP64 keeps 53), and then
      // one FP64 number, whose exponent field takes the rest of the scaling.
      const int eA = m0 + lane < p.M ? __ldg(expA + p.ar + m0 + lane) : 0;
      const int eB = lane < 16 && n0 + lane < p.N ? __ldg(expB + p.br + n0 + lane) : 0;
      int top = 0;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int h = (int)(hi[q] >> 32);
        top |= h ^ (h >> 31);
      }
      const int sh = max(0, 64 - 35 - __clz(top));
      const int e0 = eA + sh - 70;
      // the exponent field stays in the normal range for every column
      const bool plain =
          __all_sync(0xffffffffu, eA > -400 && eA < 400 && eB > -400 && eB < 400 && sh <= 27);
      const int sgn = negate ? (int)0x80000000 : 0;
      // rows of C in whole 32-byte sectors, one per load and store, half of the
      // columns at a time with the loads ahead of the conversions
      const bool vec = row_in && ((p.c | p.ldc) & 3) == 0 && n0 + 16 <= p.N;
      auto store = [&](auto value) {
#pragma unroll
        for (int h = 0; h < 16; h += 8) {
          double4_32a* c4 = reinterpret_cast<double4_32a*>(crow + h);
          double4_32a o0 = double4_32a{0.0, 0.0, 0.0, 0.0}, o1 = o0;
          if (ADD && vec) {
            o0 = c4[0];
            o1 = c4[1];
          }
          double w[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) w[q] = value(h + q, e0 + __shfl_sync(0xffffffffu, eB, h + q));
          if (vec) {
            if (ADD) {
              c4[0] = double4_32a{w[0] + o0.x, w[1] + o0.y, w[2] + o0.z, w[3] + o0.w};
              c4[1] = double4_32a{w[4] + o1.x, w[5] + o1.y, w[6] + o1.z, w[7] + o1.w};
            } else {
              c4[0] = double4_32a{w[0], w[1], w[2], w[3]};
              c4[1] = double4_32a{w[4], w[5], w[6], w[7]};
            }
          } else if (row_in) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (n0 + h + q < p.N) crow[h + q] = ADD ? crow[h + q] + w[q] : w[q];
          }
        }
      };
      if (plain)
        store([&](int cc, int e) -> double {
          const double x = (double)((hi[cc] << (27 - sh)) + (lo[cc] >> sh));
          const int xh = __double2hiint(x);
          return __hiloint2double(xh != 0 ? (xh + (e << 20)) ^ sgn : 0, __double2loint(x));
        });
      else
        store([&](int cc, int e) -> double { return slow_value(hi[cc], lo[cc], sh, e, negate); });
    }
  }
  __syncwarp();
  if (*(volatile int*)abort_flag != 0) {
    if (threadIdx.x == 0) atomicOr(status, DEV_TIMEOUT);
    // the last copy of every slice may be in flight: wait (bounded) before the
    // shared memory is released
    if (warp == 0 && lane == 0)
      for (int t = max(0, issued - S); t < issued; ++t)
        (void)tc::mbar_wait(&full[S - 1 - t % S], (t / S) & 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SLOTS * BN) : "memory");
  }
}

// ------------------------------------------------------------------ host
// 3-D map {Kp, rows, S} of a digit array: boxes of BK x box_rows x 1,
// 128-byte swizzle, zero fill outside.
inline CUtensorMap encode_digits(const __half* base, int64_t rows, int Kp, int box_rows) {
  CB_CHECK(Kp % BK == 0 && Kp > 0 && rows > 0, CBDDC_EINVAL, "tensor map: bad digit array shape");
  CB_CHECK(((uintptr_t)base & 15) == 0, CBDDC_EINVAL, "tensor map: base not 16-byte aligned");
  CUtensorMap m;
  const cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)rows, (cuuint64_t)S};
  const cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)Kp * 2 * (cuuint64_t)rows};
  const cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = tc::encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(base), dims,
                                     strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  CB_CHECK(r == CUDA_SUCCESS, CBDDC_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return m;
}

// Digit arrays of one batch of problems: A digits, B digits, exponents of
// both, each part starting on a 256-byte boundary.
struct Batch {
  int a0 = 0, na = 0, b0 = 0, nb = 0;  // split work items of op(A) and op(B)
  int t0 = 0, nt = 0;                  // output tiles
  int Kp = 64;
  int64_t rowsA = 0, rowsB = 0;
  Maps maps;
  int64_t bytes_a() const { return round_up((int64_t)S * rowsA * Kp * 2, 256); }
  int64_t bytes_b() const { return round_up((int64_t)S * rowsB * Kp * 2, 256); }
  int64_t bytes_ea() const { return round_up(rowsA * 4, 256); }
  int64_t bytes() const { return bytes_a() + bytes_b() + bytes_ea() + round_up(rowsB * 4, 256); }
};

// Digits of one batch, at most: problems share a batch while they fit, and
// a larger one is cut into blocks of whole tiles.  A context keeps one buffer of
// this size, or less where its products need less or the memory is short (a
// sixteenth of what is free, down to the second figure).  Each batch costs three launches and a last wave of
// tiles: the FP64 Newton step of the 48x48x12 slab (60 ms), whose E and S take 2.3
// and 2.4 GB of digits, takes 1% longer with 1 GiB than with 2 GiB, and 2% longer
// with 512 MiB.
constexpr int64_t kBatchBytes = (int64_t)1 << 30, kMinBatchBytes = (int64_t)8 << 20;

template <bool ADD>
static void set_smem_attr() {
  static PerDevice<bool> done;
  allow_smem(done, gemm_kernel<ADD>, SMEM);
}

}  // namespace oz
}  // namespace cbddc
