// Flexible GMRES (FP64) preconditioned by BDDC, and the Newton iteration of
// Eq. (tangent problem): d^{n,k} = d^{n,k-1} + delta, DF(d) delta = -F(d).
//
// GMRES: Arnoldi basis V (column j contiguous), preconditioned vectors
// Z_j = M^-1 v_j, classical Gram-Schmidt applied twice (two passes of
// h = V^T w, w -= V h), Givens rotations and the least-squares residual
// |g_{j+1}| kept on the device; restart after m steps with the true
// residual recomputed.
#include <algorithm>
#include <cmath>
#include <cstring>

#include <cooperative_groups.h>

#include "bddc.h"
#include "fem.h"
#include "krylov.h"

namespace cbddc {

namespace cg = cooperative_groups;

namespace {

constexpr int DOT_THREADS = 256;
constexpr int64_t kCoopMaxN = 1000000;  // longest vector for the cooperative orthogonalisation
// Longest vector whose orthogonalisation keeps a chunk of w per CTA; above, it
// goes in tiles.  Mean Arnoldi step over 100 vectors, chunks against tiles:
// 117 and 159 us at n = 126k, 208 and 231 us at 259k, 224 and 224 us at 304k,
// 388 and 341 us at 608k.
constexpr int64_t kChunkMaxN = 300000;
constexpr int MAXV = 128;       // Krylov vectors of the cooperative orthogonalisation
constexpr int MAXT = 256;       // Krylov vectors of its tiled form
constexpr int MAXR = 1024;      // Krylov vectors per cycle (restart <= MAXR - 1)

__device__ inline double wsum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block dot products with a last-block reduction.  Each CTA owns a tile of
// 256 * RPT consecutive rows: it first forms its rows of w (optionally
// w -= V hin, which fuses the update of one Gram-Schmidt pass with the dots
// of the next), keeps them in shared memory, then every warp takes whole
// columns of V and reads the tile's rows of that column with all 32 lanes
// (coalesced, 8 * RPT independent loads per lane), so the reduction costs
// one warp sum per column and CTA.  The CTA that finishes last (atomic
// ticket) sums the per-CTA partials in CTA order, so results do not depend
// on scheduling.
struct DotArgs {
  const double* V;      // nvec columns of length n, stride ldv
  int64_t ldv;
  int nvec;
  double* w;            // [n]
  int64_t n;
  const double* hin;    // if non-null: w -= V hin before the dots
  int self_norm;        // dots of w with itself instead of with V
  double* partial;      // [gridDim.x][pstride]
  int pstride;          // row stride of partial (>= nvec)
  unsigned* ticket;     // zero on entry, reset by the last CTA
  double* out;          // [nvec] (or [1] for the norm)
  const int* done;      // skip everything once GMRES has converged
  const int* gate;      // if non-null: skip unless *gate != 0
  int also_norm;        // dots with V plus out[nvec] = ||w||^2 (before any update)
};

__device__ inline void last_block_sum(const DotArgs& a, int nout) {
  __shared__ bool last;
  __shared__ double half[MAXV];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(a.ticket, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!last) return;
  // two threads per output: CTAs [0, G/2) and [G/2, G), four accumulators
  // each in a fixed order, then the halves added in a fixed order; outputs
  // in chunks of 128
  const int jl = threadIdx.x & (MAXV - 1), side = threadIdx.x >> 7;
  const unsigned G = gridDim.x, mid = G / 2;
  const unsigned c0 = side ? mid : 0u, c1 = side ? G : mid;
  for (int j0 = 0; j0 < nout; j0 += MAXV) {
    const int j = j0 + jl;
    double s4[4] = {0.0, 0.0, 0.0, 0.0};
    if (j < nout) {
      unsigned c = c0;
      for (; c + 4 <= c1; c += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) s4[q] += __ldcg(a.partial + (int64_t)(c + q) * a.pstride + j);
      }
      for (; c < c1; ++c) s4[0] += __ldcg(a.partial + (int64_t)c * a.pstride + j);
    }
    const double sum = (s4[0] + s4[1]) + (s4[2] + s4[3]);
    if (side == 1 && j < nout) half[jl] = sum;
    __syncthreads();
    if (side == 0 && j < nout) a.out[j] = sum + half[jl];
    __syncthreads();
  }
  if (threadIdx.x == 0) *a.ticket = 0u;
  __threadfence();
}

template <int RPT>
__global__ void __launch_bounds__(DOT_THREADS) fused_dots_kernel(DotArgs a) {
  if (a.done && *a.done) return;
  if (a.gate && !*a.gate) return;
  constexpr int TILE = DOT_THREADS * RPT;
  __shared__ double ws[TILE];
  __shared__ double hs[MAXR];
  __shared__ double red[DOT_THREADS / 32];
  const int64_t r0 = (int64_t)blockIdx.x * TILE;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows = (int)min((int64_t)TILE, a.n - r0);
  // rows of w (updated when hin is given)
  double x[RPT];
#pragma unroll
  for (int t = 0; t < RPT; ++t) {
    const int q = tid + DOT_THREADS * t;
    x[t] = q < rows ? a.w[r0 + q] : 0.0;
  }
  if (a.hin) {
    for (int j = tid; j < a.nvec; j += DOT_THREADS) hs[j] = a.hin[j];
    __syncthreads();
    for (int j = 0; j < a.nvec; ++j) {
      const double hj = hs[j];
      const double* Vj = a.V + (int64_t)j * a.ldv + r0;
#pragma unroll
      for (int t = 0; t < RPT; ++t) {
        const int q = tid + DOT_THREADS * t;
        if (q < rows) x[t] -= Vj[q] * hj;
      }
    }
#pragma unroll
    for (int t = 0; t < RPT; ++t) {
      const int q = tid + DOT_THREADS * t;
      if (q < rows) a.w[r0 + q] = x[t];
    }
  }
  const int nout = a.self_norm ? 1 : a.nvec + (a.also_norm ? 1 : 0);
  if (a.also_norm && !a.self_norm) {
    double acc = 0.0;
#pragma unroll
    for (int t = 0; t < RPT; ++t) acc += x[t] * x[t];
    acc = wsum(acc);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
      double sm = 0.0;
      for (int q = 0; q < DOT_THREADS / 32; ++q) sm += red[q];
      a.partial[(int64_t)blockIdx.x * a.pstride + a.nvec] = sm;
    }
  }
  if (a.self_norm) {
    double acc = 0.0;
#pragma unroll
    for (int t = 0; t < RPT; ++t) acc += x[t] * x[t];
    acc = wsum(acc);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (tid == 0) {
      double sm = 0.0;
      for (int q = 0; q < DOT_THREADS / 32; ++q) sm += red[q];
      a.partial[(int64_t)blockIdx.x * a.pstride] = sm;
    }
  } else {
#pragma unroll
    for (int t = 0; t < RPT; ++t) ws[tid + DOT_THREADS * t] = x[t];
    __syncthreads();
    for (int j = warp; j < a.nvec; j += DOT_THREADS / 32) {
      const double* Vj = a.V + (int64_t)j * a.ldv + r0;
      double acc = 0.0;
#pragma unroll 8
      for (int q = lane; q < TILE; q += 32)
        if (q < rows) acc += Vj[q] * ws[q];
      acc = wsum(acc);
      if (lane == 0) a.partial[(int64_t)blockIdx.x * a.pstride + j] = acc;
    }
  }
  last_block_sum(a, nout);
}

// Column j of the Hessenberg matrix from h1 + h2 (the two CGS passes) and
// ||w||^2, previous rotations, the new rotation and the residual estimate.
// scal[0] = |g_{j+1}| / ||b||, scal[1] = 1 / h_{j+1,j}, scal[2] = ||b||.
// Run by a whole CTA: the column and the rotations come into shared memory
// (sm: 3 (j + 1) doubles) first, because the chain over the j rotations is
// serial, and on global memory each link cost an L2 round trip (0.35 us; 9 us
// of a 100 us Arnoldi step at j = 25).
__device__ void givens_update(int j, int m, double* __restrict__ H, double* __restrict__ cs,
                              double* __restrict__ sn, double* __restrict__ g, const double* h1,
                              const double* h2, double wn2, double* __restrict__ scal, double rtol,
                              int* __restrict__ done, int* __restrict__ iters, double* sm) {
  double* col = sm;
  double* c = sm + (j + 1);
  double* s = sm + 2 * (j + 1);
  for (int i = threadIdx.x; i <= j; i += blockDim.x) {
    col[i] = h2 ? h1[i] + h2[i] : h1[i];
    if (i < j) {
      c[i] = cs[i];
      s[i] = sn[i];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double hn = sqrt(fmax(wn2, 0.0));
    scal[1] = hn > 0.0 ? 1.0 / hn : 0.0;
    double cur = col[0];
    for (int i = 0; i < j; ++i) {
      const double nxt = col[i + 1];
      const double t = c[i] * cur + s[i] * nxt;
      cur = -s[i] * cur + c[i] * nxt;
      col[i] = t;
    }
    const double den = hypot(cur, hn);
    cs[j] = den > 0.0 ? cur / den : 1.0;
    sn[j] = den > 0.0 ? hn / den : 0.0;
    col[j] = den;
    g[j + 1] = -sn[j] * g[j];
    g[j] = cs[j] * g[j];
    const double res = fabs(g[j + 1]) / scal[2];
    scal[0] = res;
    *iters += 1;
    if (res <= rtol || hn == 0.0) *done = 1;
  }
  __syncthreads();
  double* out = H + (int64_t)j * (m + 1);
  for (int i = threadIdx.x; i <= j + 1; i += blockDim.x) out[i] = i <= j ? col[i] : 0.0;
}

__global__ void givens_kernel(int j, int m, double* __restrict__ H, double* __restrict__ cs,
                              double* __restrict__ sn, double* __restrict__ g,
                              const double* __restrict__ h1, const double* __restrict__ h2,
                              const double* __restrict__ wn2, double* __restrict__ scal, double rtol,
                              int* __restrict__ done, int* __restrict__ iters) {
  __shared__ double sm[3 * MAXR];
  if (*done) return;
  __syncthreads();  // every thread has read the flag
  givens_update(j, m, H, cs, sn, g, h1, h2, wn2[0], scal, rtol, done, iters, sm);
}

// The whole orthogonalisation of one Arnoldi step in one cooperative launch
// (all CTAs resident, grid-wide barriers): h1 = V^T w; w -= V h1, h2 = V^T w;
// w -= V h2, ||w||^2; the Givens update (CTA 0) and v_{j+1} = w / ||w||.
//
// Every CTA keeps a contiguous chunk of w in shared memory through the whole
// step.  FP64 issue is the limit (4 (j + 1) n FMAs at 2 per SM and clock), so
// the work is spread over all SMs and all warps at any basis size and little
// is issued beside the FMAs: dots take eight columns per warp and a segment of
// the rows, and reduce the eight sums together at the end of the chunk (9
// additions instead of 40); updates take 32 rows and a part of the columns per
// warp, two to four parts so that the 16 warps have about 64 of these shares (a
// chunk has at most 1024 rows on 152 SMs), added at the end.  After each barrier
// every CTA sums all CTAs' partials in CTA order (identical on every CTA,
// independent of scheduling).
// Mean Arnoldi step of a solve: 60 us at n = 86k and 59 vectors (100 us with
// 256-row tiles dealt to half of the SMs, one column per warp and a Givens
// chain on global memory), 51 us at n = 27k and 90 vectors (114 us).
constexpr int CGS_THREADS = 512;
constexpr int CGS_WARPS = CGS_THREADS / 32;
constexpr int CGS_JS = 4;  // column parts of the update, at most (two at least)
struct CgsArgs {
  const double* V;   // nvec columns of length n (stride n)
  int64_t n;
  int nvec;          // j + 1
  int rows;          // rows per CTA
  int js;            // column parts of the update
  double* w;
  double* vnext;     // column j + 1
  double* part;      // [3][gridDim.x][MAXV]
  int j, m;
  double *H, *cs, *sn, *g, *scal;
  double rtol;
  int *done, *iters;
};

// This warp's share of V^T ws: columns c0 .. c0 + 7 over the rows of segment
// seg (32-row blocks seg, seg + nseg, ...); at most one share per warp.
struct CgsDots {
  int c0, seg, nseg;
  bool active;
  double s[8];
  __device__ CgsDots(int nvec) {
    const int warp = threadIdx.x >> 5;
    const int ng = (nvec + 7) / 8;                    // groups of eight columns
    nseg = max(1, CGS_WARPS / ng);                    // row segments
    c0 = 8 * (warp % ng);
    seg = warp / ng;
    active = seg < nseg;
#pragma unroll
    for (int q = 0; q < 8; ++q) s[q] = 0.0;
  }
  // the rows of the chunk
  __device__ void add(const CgsArgs& a, const double* __restrict__ ws, int64_t r0, int rows) {
    if (!active) return;
    const int lane = threadIdx.x & 31;
    const double* p[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) p[q] = a.V + (int64_t)min(c0 + q, a.nvec - 1) * a.n + r0;
#pragma unroll 2
    for (int r = 32 * seg + lane; r < rows; r += 32 * nseg) {
      const double x = ws[r];
#pragma unroll
      for (int q = 0; q < 8; ++q) s[q] = fma(__ldg(p[q] + r), x, s[q]);
    }
  }
  // part[0:nvec] = the CTA's sums; psum: [CGS_WARPS][MAXV] shared
  __device__ void finish(const CgsArgs& a, double* psum, double* __restrict__ part) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (active) {
#pragma unroll
      for (int w = 4; w > 0; w >>= 1) {
        const bool up = (lane & (4 * w)) != 0;
#pragma unroll
        for (int q = 0; q < w; ++q) {
          const double keep = up ? s[q + w] : s[q], give = up ? s[q] : s[q + w];
          s[q] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * w);
        }
      }
      s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
      s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
      if ((lane & 3) == 0) psum[seg * MAXV + c0 + (lane >> 2)] = s[0];
    }
    __syncthreads();
    for (int c = threadIdx.x; c < a.nvec; c += CGS_THREADS) {
      double t = psum[c];
      for (int q = 1; q < nseg; ++q) t += psum[q * MAXV + c];
      part[c] = t;
    }
  }
};

// ws -= V h over the chunk; upd: [js][a.rows] shared, the sums of js column
// parts.  Ends with a barrier.
__device__ void cgs_update(const CgsArgs& a, double* __restrict__ ws, double* __restrict__ upd, int64_t r0, int rows,
                           const double* __restrict__ h) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rb = (rows + 31) / 32;
  for (int it = warp; it < rb * a.js; it += CGS_WARPS) {
    const int r = 32 * (it % rb) + lane, part = it / rb;
    if (r < rows) {
      const double* p = a.V + r0 + r;
      double s = 0.0;
#pragma unroll 8
      for (int c = part; c < a.nvec; c += a.js) s = fma(__ldg(p + (int64_t)c * a.n), h[c], s);
      upd[part * a.rows + r] = s;
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < rows; r += CGS_THREADS) {
    double t = upd[r];
    for (int q = 1; q < a.js; ++q) t += upd[q * a.rows + r];
    ws[r] -= t;
  }
  __syncthreads();
}

// sums of every CTA's partials into out[0:nout] (shared memory): every warp
// 32 columns over every WARPS-th CTA, combined in a fixed order (identical
// on every CTA, independent of scheduling)
template <int WARPS, int NV>
__device__ void cgs_reduce(const double* part, int nout, double* psum, double* out) {
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  for (int j0 = 0; j0 < nout; j0 += 32) {
    const int j = j0 + lane;
    double s = 0.0;
    if (j < nout) {
#pragma unroll 4
      for (unsigned c = grp; c < gridDim.x; c += WARPS) s += __ldcg(part + (int64_t)c * NV + j);
    }
    psum[grp * 33 + lane] = s;
    __syncthreads();
    if (grp == 0 && j < nout) {
      double t = psum[lane];
      for (int q = 1; q < WARPS; ++q) t += psum[q * 33 + lane];
      out[j] = t;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(CGS_THREADS, 2) cgs2_coop_kernel(CgsArgs a) {
  cg::grid_group grid = cg::this_grid();
  if (*a.done) return;  // read by every CTA before any barrier: uniform
  extern __shared__ double cgs_smem[];
  __shared__ double psum[CGS_WARPS * MAXV];
  __shared__ double h1[MAXV], h2[MAXV], wn2s[1];
  double* ws = cgs_smem;               // [a.rows]
  double* upd = cgs_smem + a.rows;     // [js][a.rows]
  const int64_t r0 = (int64_t)blockIdx.x * a.rows;
  const int rows = (int)max((int64_t)0, min((int64_t)a.rows, a.n - r0));
  const int64_t stride = (int64_t)gridDim.x * MAXV;
  double* part = a.part + (int64_t)blockIdx.x * MAXV;
  for (int r = threadIdx.x; r < rows; r += CGS_THREADS) ws[r] = a.w[r0 + r];
  __syncthreads();
  {
    CgsDots d(a.nvec);
    d.add(a, ws, r0, rows);
    d.finish(a, psum, part);
  }
  grid.sync();
  cgs_reduce<CGS_WARPS, MAXV>(a.part, a.nvec, psum, h1);
  cgs_update(a, ws, upd, r0, rows, h1);
  {
    CgsDots d(a.nvec);
    d.add(a, ws, r0, rows);
    d.finish(a, psum, part + stride);
  }
  grid.sync();
  cgs_reduce<CGS_WARPS, MAXV>(a.part + stride, a.nvec, psum, h2);
  cgs_update(a, ws, upd, r0, rows, h2);
  {
    double s = 0.0;
    for (int r = threadIdx.x; r < rows; r += CGS_THREADS) s = fma(ws[r], ws[r], s);
    s = wsum(s);
    if ((threadIdx.x & 31) == 0) psum[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = psum[0];
      for (int q = 1; q < CGS_WARPS; ++q) t += psum[q];
      part[2 * stride] = t;
    }
  }
  grid.sync();
  cgs_reduce<CGS_WARPS, MAXV>(a.part + 2 * stride, 1, psum, wn2s);
  if (blockIdx.x == 0)
    givens_update(a.j, a.m, a.H, a.cs, a.sn, a.g, h1, h2, wn2s[0], a.scal, a.rtol, a.done, a.iters, psum);
  // v_{j+1} = w / ||w|| (the same value on every CTA)
  const double hn = sqrt(fmax(wn2s[0], 0.0));
  const double inv = hn > 0.0 ? 1.0 / hn : 0.0;
  for (int r = threadIdx.x; r < rows; r += CGS_THREADS) a.vnext[r0 + r] = ws[r] * inv;
}

// The same step for vectors above kChunkMaxN unknowns, where V streams from
// HBM, and for bases of MAXV to MAXT vectors: 256-row tiles dealt round-robin, w in global memory, a row per thread in
// the updates and whole columns per warp in the dots.  Neighbouring CTAs then
// read neighbouring tiles of the same column, which HBM serves better than the
// chunks' 304 distant streams, and the FMAs hide behind it.  Past MAXV vectors
// it replaces modified Gram-Schmidt, whose grid-wide barrier per vector cost
// more than the second pass: 924 us against 1100 us at n = 582k and 147 vectors,
// 397 us against 1404 us at n = 27k and 192 vectors.
template <int NV>
__device__ void tiles_phase(const CgsArgs& a, const double* hin, bool norm, double* ws, double* part) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int CPW = NV / (DOT_THREADS / 32);  // columns per warp
  double acc[CPW];
#pragma unroll
  for (int q = 0; q < CPW; ++q) acc[q] = 0.0;
  double nacc = 0.0;
  const int64_t ntiles = (a.n + DOT_THREADS - 1) / DOT_THREADS;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t r0 = t * DOT_THREADS;
    const int rows = (int)min((int64_t)DOT_THREADS, a.n - r0);
    double x = tid < rows ? a.w[r0 + tid] : 0.0;
    if (hin && tid < rows) {
      for (int j = 0; j < a.nvec; ++j) x -= a.V[(int64_t)j * a.n + r0 + tid] * hin[j];
      a.w[r0 + tid] = x;
    }
    if (norm) {
      nacc += x * x;
    } else {
      __syncthreads();   // the previous tile's readers of ws are done
      ws[tid] = x;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < CPW; ++q) {
        const int j = warp + (DOT_THREADS / 32) * q;
        if (j < a.nvec) {
          const double* Vj = a.V + (int64_t)j * a.n + r0;
          for (int rr = lane; rr < rows; rr += 32) acc[q] += Vj[rr] * ws[rr];
        }
      }
    }
  }
  __shared__ double red[DOT_THREADS / 32];
  if (norm) {
    nacc = wsum(nacc);
    if (lane == 0) red[warp] = nacc;
    __syncthreads();
    if (tid == 0) {
      double sm = 0.0;
      for (int q = 0; q < DOT_THREADS / 32; ++q) sm += red[q];
      part[(int64_t)blockIdx.x * NV] = sm;
    }
  } else {
#pragma unroll
    for (int q = 0; q < CPW; ++q) {
      const int j = warp + (DOT_THREADS / 32) * q;
      const double v = wsum(acc[q]);
      if (lane == 0 && j < a.nvec) part[(int64_t)blockIdx.x * NV + j] = v;
    }
  }
}

template <int NV>
__global__ void __launch_bounds__(DOT_THREADS, 2) cgs2_tiles_kernel(CgsArgs a) {
  cg::grid_group grid = cg::this_grid();
  if (*a.done) return;  // read by every CTA before any barrier: uniform
  __shared__ double ws[DOT_THREADS], psum[3 * NV];
  static_assert(3 * NV >= DOT_THREADS / 32 * 33, "reduction scratch");
  __shared__ double h1[NV], h2[NV], wn2s[1];
  const int64_t stride = (int64_t)gridDim.x * NV;
  tiles_phase<NV>(a, nullptr, false, ws, a.part);
  grid.sync();
  cgs_reduce<DOT_THREADS / 32, NV>(a.part, a.nvec, psum, h1);
  tiles_phase<NV>(a, h1, false, ws, a.part + stride);
  grid.sync();
  cgs_reduce<DOT_THREADS / 32, NV>(a.part + stride, a.nvec, psum, h2);
  tiles_phase<NV>(a, h2, true, ws, a.part + 2 * stride);
  grid.sync();
  cgs_reduce<DOT_THREADS / 32, NV>(a.part + 2 * stride, 1, psum, wn2s);
  if (blockIdx.x == 0)
    givens_update(a.j, a.m, a.H, a.cs, a.sn, a.g, h1, h2, wn2s[0], a.scal, a.rtol, a.done, a.iters, psum);
  // v_{j+1} = w / ||w|| (the same value on every CTA)
  const double hn = sqrt(fmax(wn2s[0], 0.0));
  const double inv = hn > 0.0 ? 1.0 / hn : 0.0;
  const int64_t ntiles = (a.n + DOT_THREADS - 1) / DOT_THREADS;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t r = t * DOT_THREADS + threadIdx.x;
    if (r < a.n) a.vnext[r] = a.w[r] * inv;
  }
}

// The Arnoldi step for long vectors or long bases in one cooperative
// launch, by modified Gram-Schmidt (backward stable for GMRES without a
// second pass, and the oracle's orthogonalisation): each thread keeps
// RPT rows of w in registers (32-row slices of its warp's segment); for
// i = 0..j: h_i = v_i . w (block sums, one grid-wide barrier, every CTA
// adds the CTA partials in CTA order), w -= h_i v_i; then ||w||, the
// Givens update (CTA 0) and v_{j+1} = w / ||w||.  V is read once per step
// (the update re-reads the rows of v_i that the thread has just read), and
// every FP64 FMA of the step is one of the 2 (j + 1) n of MGS.
constexpr int MGS_THREADS = 640;
struct MgsArgs {
  const double* V;   // j + 1 columns of length n (stride n)
  int64_t n;
  double* w;
  double* vnext;
  double* part;      // [2][gridDim.x]
  double* hcol;      // [m + 1]: this step's Hessenberg column
  int j, m;
  double *H, *cs, *sn, *g, *scal;
  double rtol;
  int *done, *iters;
};

template <int RPT>
__global__ void __launch_bounds__(MGS_THREADS, 1) mgs_coop_kernel(MgsArgs a) {
  cg::grid_group grid = cg::this_grid();
  if (*a.done) return;  // read by every CTA before any barrier: uniform
  __shared__ double red[MGS_THREADS / 32];
  __shared__ double hsh;
  __shared__ double gsm[3 * MAXR];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = gridDim.x;
  // warp-contiguous rows: the warp's segment of 32 RPT rows, lane + 32 k
  // (coalesced, and the offsets of the k loop are constants)
  const int64_t base = ((int64_t)blockIdx.x * (MGS_THREADS / 32) + warp) * (32 * RPT) + lane;
  const int64_t lim = a.n - base;  // row k exists iff 32 k < lim
  double x[RPT];
  {
    const double* wp = a.w + base;
#pragma unroll
    for (int k = 0; k < RPT; ++k) x[k] = 32 * k < lim ? wp[32 * k] : 0.0;
  }
  // grid-wide sum of one value per thread (deterministic), into hsh
  auto grid_sum = [&](double v, int buf) -> double {
    v = wsum(v);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int q = 0; q < MGS_THREADS / 32; ++q) t += red[q];
      a.part[(int64_t)buf * G + blockIdx.x] = t;
    }
    grid.sync();
    if (warp == 0) {
      double t = 0.0;
      for (int b = lane; b < G; b += 32) t += __ldcg(a.part + (int64_t)buf * G + b);
      t = wsum(t);
      if (lane == 0) hsh = t;
    }
    __syncthreads();
    const double out = hsh;
    __syncthreads();
    return out;
  };
  for (int i = 0; i <= a.j; ++i) {
    const double* vp = a.V + (int64_t)i * a.n + base;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < RPT; ++k)
      if (32 * k < lim) acc = fma(vp[32 * k], x[k], acc);
    const double h = grid_sum(acc, i & 1);
    if (blockIdx.x == 0 && threadIdx.x == 0) a.hcol[i] = h;
#pragma unroll
    for (int k = 0; k < RPT; ++k)
      if (32 * k < lim) x[k] = fma(-h, vp[32 * k], x[k]);
  }
  double nacc = 0.0;
#pragma unroll
  for (int k = 0; k < RPT; ++k) nacc = fma(x[k], x[k], nacc);
  const double wn2 = grid_sum(nacc, (a.j + 1) & 1);
  // (thread 0 of CTA 0 wrote hcol; the barriers since then order it)
  if (blockIdx.x == 0)
    givens_update(a.j, a.m, a.H, a.cs, a.sn, a.g, a.hcol, nullptr, wn2, a.scal, a.rtol, a.done, a.iters, gsm);
  const double hn = sqrt(fmax(wn2, 0.0));
  const double inv = hn > 0.0 ? 1.0 / hn : 0.0;
  double* op = a.vnext + base;
#pragma unroll
  for (int k = 0; k < RPT; ++k)
    if (32 * k < lim) op[32 * k] = x[k] * inv;
}

__global__ void scale_kernel(const double* __restrict__ w, double* __restrict__ v, int64_t n,
                             const double* __restrict__ scal, int idx, const int* __restrict__ done) {
  if (done && *done) return;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) v[i] = w[i] * scal[idx];
}

// y = R^-1 g (upper triangular, k columns), one CTA: column-oriented back
// substitution, y_i = s_i / R_ii and then s_r -= R_ri y_i for all r < i in
// parallel (one barrier per column)
__global__ void __launch_bounds__(256)
backsolve_kernel(const double* __restrict__ H, int m, const int* __restrict__ kp,
                 const double* __restrict__ g, double* __restrict__ y) {
  __shared__ double sv[MAXR];
  __shared__ double yi;
  const int k = *kp;
  for (int i = threadIdx.x; i < k; i += blockDim.x) sv[i] = g[i];
  __syncthreads();
  for (int i = k - 1; i >= 0; --i) {
    const double* col = H + (int64_t)i * (m + 1);
    if (threadIdx.x == 0) {
      yi = sv[i] / col[i];
      y[i] = yi;
    }
    __syncthreads();
    const double v = yi;
    for (int r = threadIdx.x; r < i; r += blockDim.x) sv[r] -= col[r] * v;
    __syncthreads();
  }
}

// Second Gram-Schmidt pass needed?  reorth = (||w - V h1||^2 < ||w||^2 / 2)
// with ||w||^2 in h1[nvec]; without it h2 = 0.  count[0] counts the passes.
__global__ void dgks_kernel(const double* __restrict__ h1, int nvec, const double* __restrict__ wn2,
                            double* __restrict__ h2, int* __restrict__ reorth, int* __restrict__ count,
                            const int* __restrict__ done) {
  if (*done) return;
  const bool again = !(wn2[0] >= 0.5 * h1[nvec]);
  if (!again)
    for (int i = threadIdx.x; i < nvec; i += blockDim.x) h2[i] = 0.0;
  if (threadIdx.x == 0) {
    *reorth = again ? 1 : 0;
    if (again) *count += 1;
  }
}

// x += Z y  (k = number of columns)
__global__ void combine_kernel(const double* __restrict__ Z, int64_t ldz, const int* __restrict__ kp,
                               const double* __restrict__ y, double* __restrict__ x, int64_t n) {
  __shared__ double ys[MAXR];
  const int k = *kp;
  for (int j = threadIdx.x; j < k; j += blockDim.x) ys[j] = y[j];
  __syncthreads();
  const int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (row >= n) return;
  double acc = x[row];
  for (int j = 0; j < k; ++j) acc += Z[(int64_t)j * ldz + row] * ys[j];
  x[row] = acc;
}

__global__ void axpby_kernel(double a, const double* __restrict__ x, double b, const double* __restrict__ y,
                             double* __restrict__ out, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) out[i] = a * x[i] + b * y[i];
}

// start of a cycle: beta = ||r|| -> g = (beta, 0, ...), scal[1] = 1/beta;
// the first cycle also records ||b||.
__global__ void cycle_start_kernel(const double* __restrict__ rn2, double* __restrict__ g, int m,
                                   double* __restrict__ scal, int first, double rtol,
                                   int* __restrict__ done, int* __restrict__ kcount) {
  const double beta = sqrt(fmax(rn2[0], 0.0));
  if (first) scal[2] = beta;
  for (int i = 0; i <= m; ++i) g[i] = 0.0;
  g[0] = beta;
  scal[1] = beta > 0.0 ? 1.0 / beta : 0.0;
  scal[0] = scal[2] > 0.0 ? beta / scal[2] : 0.0;
  *kcount = 0;
  *done = (beta <= rtol * scal[2]) ? 1 : 0;
}

}  // namespace

void Gmres::ensure_small(int64_t n_) {
  if (partial.p && nchunks == (int)cdiv(n_, DOT_THREADS)) return;
  nchunks = (int)cdiv(n_, DOT_THREADS);   // CTAs at one row per thread (the most)
  pstride = MAXV;
  partial.alloc((size_t)nchunks * pstride);
  ticket.alloc(1);
  CB_CUDA(cudaMemset(ticket.p, 0, sizeof(unsigned)));
  hstride = MAXV;
  h.alloc(3 * hstride);
  scal.alloc(10);
  CB_CUDA(cudaMemset(scal.p, 0, scal.bytes()));
  if (!host_scal) CB_CUDA(cudaMallocHost(&host_scal, 32 * sizeof(double)));
  for (auto& e : step_done)
    if (!e) CB_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
}

void Gmres::ensure(int64_t n_, int m_) {
  ensure_small(n_);
  if (n == n_ && m == m_) return;
  // cooperative orthogonalisation; 0 when the device cannot launch
  // cooperatively
  {
    int dev = 0, coop = 0, sms = 0, per_sm = 0;
    CB_CUDA(cudaGetDevice(&dev));
    CB_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    CB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    coop_grid = tile_grid = 0;
    if (coop && n_ <= kChunkMaxN) {
      // two CTAs per SM, fewer for short vectors: the FMAs shrink with the
      // grid and the sums of its partials grow with it
      const int64_t g = std::max<int64_t>(1, (int64_t)std::sqrt(2.0 * (double)n_));
      coop_grid = (int)std::min<int64_t>((n_ >= 1024 * (int64_t)sms ? 2 : 1) * sms, g);
      cgs_rows = (int)round_up(cdiv(n_, coop_grid), 32);
      coop_grid = (int)cdiv(n_, cgs_rows);
      cgs_js = (int)std::min<int64_t>(CGS_JS, std::max<int64_t>(2, 4 * CGS_WARPS / (cgs_rows / 32)));
      cgs_smem = (size_t)cgs_rows * (1 + cgs_js) * sizeof(double);
      CB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cgs2_coop_kernel, CGS_THREADS, cgs_smem));
      if (coop_grid > per_sm * sms) coop_grid = 0;
    }
    if (coop && n_ <= kCoopMaxN) {
      // at most two CTAs per SM, about four row tiles per CTA
      CB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cgs2_tiles_kernel<MAXT>, DOT_THREADS, 0));
      tile_grid = (int)std::min<int64_t>(std::min(per_sm, 2) * (int64_t)sms,
                                         std::max<int64_t>(1, cdiv(n_, DOT_THREADS) / 4));
    }
    if (coop_grid + tile_grid > 0)
      cpart.alloc(3 * std::max((size_t)coop_grid * MAXV, (size_t)tile_grid * MAXT));
    // MGS cooperative launch: one CTA of MGS_THREADS per SM, rows per
    // thread rounded up to 8, 16, 24 or 32 (n up to 3.1M on 152 SMs; 0:
    // the multi-launch path)
    mgs_grid = 0;
    mgs_rpt = 0;
    if (coop) {
      const int64_t T = (int64_t)sms * MGS_THREADS;
      const int64_t need = (n_ + T - 1) / T;
      const int rpt = need <= 8 ? 8 : need <= 16 ? 16 : need <= 24 ? 24 : need <= 32 ? 32 : 0;
      int per = 0;
      if (rpt == 8) CB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mgs_coop_kernel<8>, MGS_THREADS, 0));
      if (rpt == 16) CB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mgs_coop_kernel<16>, MGS_THREADS, 0));
      if (rpt == 24) CB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mgs_coop_kernel<24>, MGS_THREADS, 0));
      if (rpt == 32) CB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mgs_coop_kernel<32>, MGS_THREADS, 0));
      if (rpt > 0 && per >= 1) {
        mgs_grid = sms;
        mgs_rpt = rpt;
        mpart.alloc((size_t)2 * sms);
      }
    }
  }
  CB_CHECK(m_ >= 1 && m_ < MAXR, CBDDC_EINVAL, "restart must be in [1, 1023]");
  n = n_;
  m = m_;
  // partial sums and Hessenberg columns for up to m + 1 Krylov vectors
  if (m + 1 > pstride) {
    pstride = (int)round_up(m + 1, 32);
    partial.alloc((size_t)nchunks * pstride);
  }
  if (m + 1 > hstride) {
    hstride = (int)round_up(m + 1, 32);
    h.alloc(3 * (size_t)hstride);
  }
  V.alloc((size_t)(m + 1) * n);
  Zb.alloc((size_t)m * n);
  w.alloc(n);
  r.alloc(n);
  H.alloc((size_t)(m + 1) * m);
  cs.alloc(m);
  sn.alloc(m);
  g.alloc(m + 1);
  y.alloc(m);
}

Gmres::~Gmres() {
  if (host_scal) cudaFreeHost(host_scal);
  for (auto& e : step_done)
    if (e) cudaEventDestroy(e);
}

// out = V^T w over nvec columns (stride ldv), optionally after w -= V hin,
// or out[0] = ||w||^2 with self_norm; one launch with a last-block reduction.
static void fused_dots(Gmres& G, const double* V, int64_t ldv, int nvec, double* w, int64_t n,
                       const double* hin, int self_norm, double* out, const int* done, cudaStream_t s,
                       const int* gate = nullptr, int also_norm = 0) {
  DotArgs a{V, ldv, nvec, w, n, hin, self_norm, G.partial.p, G.pstride, G.ticket.p, out, done, gate, also_norm};
  // rows per thread: the largest of 16, 8, 4, 2, 1 that still gives two
  // CTAs per SM (fewer CTAs also shorten the last CTA's reduction)
  const int64_t sms2 = 2 * 152;
  if (n >= 16 * DOT_THREADS * sms2) {
    fused_dots_kernel<16><<<(unsigned)cdiv(n, 16 * DOT_THREADS), DOT_THREADS, 0, s>>>(a);
  } else if (n >= 8 * DOT_THREADS * sms2) {
    fused_dots_kernel<8><<<(unsigned)cdiv(n, 8 * DOT_THREADS), DOT_THREADS, 0, s>>>(a);
  } else if (n >= 4 * DOT_THREADS * sms2) {
    fused_dots_kernel<4><<<(unsigned)cdiv(n, 4 * DOT_THREADS), DOT_THREADS, 0, s>>>(a);
  } else if (n >= 2 * DOT_THREADS * sms2) {
    fused_dots_kernel<2><<<(unsigned)cdiv(n, 2 * DOT_THREADS), DOT_THREADS, 0, s>>>(a);
  } else {
    fused_dots_kernel<1><<<(unsigned)cdiv(n, DOT_THREADS), DOT_THREADS, 0, s>>>(a);
  }
  CB_LAUNCH();
}

int gmres_run(fem_problem* P, bddc_ctx* C, Gmres& G, const double* b, double* x, int restart,
              int max_iters, double rtol, int* iters_out, double* relres_out, cudaStream_t s) {
  const int64_t n = P->n_free;
  G.ensure(n, restart);
  const int m = restart;
  const unsigned nb = cdiv(n, 256);
  int* done = G.flags();
  int* kcount = G.flags() + 1;
  CB_CUDA(cudaMemsetAsync(x, 0, n * sizeof(double), s));
  int total = 0;
  bool first = true;
  CB_CUDA(cudaMemsetAsync(G.flags() + 3, 0, sizeof(int), s));  // second Gram-Schmidt passes
  bool converged = false;
  int flags[4] = {0, 0, 0, 0};  // the device's, as last read
  // scalars and flags of the device into a pinned slot
  auto fetch = [&](int slot) {
    CB_CUDA(cudaMemcpyAsync(G.host_scal + 10 * slot, G.scal.p, 10 * sizeof(double), cudaMemcpyDeviceToHost, s));
    CB_CUDA(cudaEventRecord(G.step_done[slot], s));
  };
  // Arnoldi step j of a cycle: v_j -> z_j = M^-1 v_j, w = K z_j, and w made
  // orthonormal to the basis
  auto arnoldi_step = [&](int j) {
    double* vj = G.V.p + (int64_t)j * n;
    double* zj = G.Zb.p + (int64_t)j * n;
    bddc_run_apply(C, vj, zj, s);
    bsr_spmv(P, zj, G.w.p, s);
    double* h1 = G.h.p;
    double* h2 = G.h.p + G.hstride;
    double* wn2 = G.h.p + 2 * G.hstride;
    timer_begin(CBDDC_TIMER_ORTH, s);
    const bool chunks = G.coop_grid > 0 && j + 1 <= MAXV;
    if (chunks || (G.tile_grid > 0 && j + 1 <= MAXT)) {
      // CGS2 in one cooperative launch
      CgsArgs ca{G.V.p, n, j + 1, G.cgs_rows, G.cgs_js, G.w.p, G.V.p + (int64_t)(j + 1) * n, G.cpart.p, j, m,
                 G.H.p, G.cs.p, G.sn.p, G.g.p, G.scal.p, rtol, done, kcount};
      void* args[] = {&ca};
      const void* fn = chunks          ? (const void*)cgs2_coop_kernel
                       : j + 1 <= MAXV ? (const void*)cgs2_tiles_kernel<MAXV>
                                       : (const void*)cgs2_tiles_kernel<MAXT>;
      CB_CUDA(cudaLaunchCooperativeKernel(fn, dim3(chunks ? G.coop_grid : G.tile_grid),
                                          dim3(chunks ? CGS_THREADS : DOT_THREADS), args, chunks ? G.cgs_smem : 0, s));
      CB_LAUNCH();
    } else if (G.mgs_grid > 0) {
      MgsArgs ma{G.V.p, n, G.w.p, G.V.p + (int64_t)(j + 1) * n, G.mpart.p, G.h.p, j, m,
                 G.H.p, G.cs.p, G.sn.p, G.g.p, G.scal.p, rtol, done, kcount};
      void* args[] = {&ma};
      const void* fn = G.mgs_rpt == 8    ? (const void*)mgs_coop_kernel<8>
                       : G.mgs_rpt == 16 ? (const void*)mgs_coop_kernel<16>
                       : G.mgs_rpt == 24 ? (const void*)mgs_coop_kernel<24>
                                         : (const void*)mgs_coop_kernel<32>;
      CB_CUDA(cudaLaunchCooperativeKernel(fn, dim3(G.mgs_grid), dim3(MGS_THREADS), args, 0, s));
      CB_LAUNCH();
    } else {
      // classical Gram-Schmidt with a second pass only where the first
      // one lost more than half of ||w||^2 (Daniel-Gragg-Kaufman-Stewart
      // criterion, eta = 1/sqrt(2)): h1 = V^T w with ||w||^2; w -= V h1
      // with the new ||w||^2; then, gated on the device, h2 = V^T w and
      // w -= V h2 with its norm
      int* reorth = G.flags() + 2;
      fused_dots(G, G.V.p, n, j + 1, G.w.p, n, nullptr, 0, h1, done, s, nullptr, 1);
      fused_dots(G, G.V.p, n, j + 1, G.w.p, n, h1, 1, wn2, done, s);
      dgks_kernel<<<1, 256, 0, s>>>(h1, j + 1, wn2, h2, reorth, G.flags() + 3, done);
      CB_LAUNCH();
      fused_dots(G, G.V.p, n, j + 1, G.w.p, n, nullptr, 0, h2, done, s, reorth);
      fused_dots(G, G.V.p, n, j + 1, G.w.p, n, h2, 1, wn2, done, s, reorth);
      givens_kernel<<<1, 256, 0, s>>>(j, m, G.H.p, G.cs.p, G.sn.p, G.g.p, h1, h2, wn2, G.scal.p, rtol, done,
                                      kcount);
      CB_LAUNCH();
      scale_kernel<<<nb, 256, 0, s>>>(G.w.p, G.V.p + (int64_t)(j + 1) * n, n, G.scal.p, 1, done);
      CB_LAUNCH();
    }
    // algorithmic traffic of one Gram-Schmidt pass (the second pass, when
    // taken, is not counted): V read twice (dots, update), w read twice
    // and written once, v_{j+1} written
    timer_end(CBDDC_TIMER_ORTH, s, 4.0 * (j + 1) * (double)n, 8.0 * (double)n * (2.0 * (j + 1) + 4.0));
    fetch(j & 1);
  };
  while (true) {
    // r = b - K x
    if (first) {
      CB_CUDA(cudaMemcpyAsync(G.r.p, b, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
    } else {
      bsr_spmv(P, x, G.w.p, s);
      axpby_kernel<<<nb, 256, 0, s>>>(1.0, b, -1.0, G.w.p, G.r.p, n);
      CB_LAUNCH();
    }
    fused_dots(G, G.r.p, n, 1, G.r.p, n, nullptr, 1, G.h.p, nullptr, s);
    cycle_start_kernel<<<1, 1, 0, s>>>(G.h.p, G.g.p, m, G.scal.p, first ? 1 : 0, rtol, done, kcount);
    CB_LAUNCH();
    scale_kernel<<<nb, 256, 0, s>>>(G.r.p, G.V.p, n, G.scal.p, 1, nullptr);
    CB_LAUNCH();
    fetch(0);
    CB_CUDA(cudaStreamSynchronize(s));
    first = false;
    std::memcpy(flags, G.host_scal + 8, sizeof flags);
    double res = G.host_scal[0];  // residual estimate of the last step known here
    *relres_out = res;
    if (flags[0]) { converged = true; break; }
    if (total >= max_iters) break;
    // The host reads the residual of every step.  Waiting for it before the
    // next step is launched left the GPU idle for the copy, the wake-up and the
    // first launches (4 to 6 us of each 170 to 440 us step of 27k unknowns), so
    // one further step is launched before step j's residual is known,
    // unless that residual can be expected to end the solve (one step gains
    // less than a factor of five): a step launched too many is skipped by the
    // Gram-Schmidt kernels, at the price of its apply and product.
    const int steps = std::min(m, max_iters - total);
    int launched = 0;
    for (int j = 0; j < steps; ++j) {
      while (launched < steps && (launched <= j || (launched == j + 1 && res > 5.0 * rtol))) arnoldi_step(launched++);
      CB_CUDA(cudaEventSynchronize(G.step_done[j & 1]));
      const double* slot = G.host_scal + 10 * (j & 1);
      std::memcpy(flags, slot + 8, sizeof flags);
      res = slot[0];
      ++total;
      if (flags[0]) {
        // (its product and preconditioner ran, its Gram-Schmidt step did not)
        if (launched > j + 1) timer_drop(CBDDC_TIMER_ORTH);
        break;
      }
    }
    // x += Z y over the columns built in this cycle
    backsolve_kernel<<<1, 256, 0, s>>>(G.H.p, m, kcount, G.g.p, G.y.p);
    CB_LAUNCH();
    combine_kernel<<<nb, 256, 0, s>>>(G.Zb.p, n, kcount, G.y.p, x, n);
    CB_LAUNCH();
    if (total >= max_iters && !flags[0]) {
      // final true residual
      bsr_spmv(P, x, G.w.p, s);
      axpby_kernel<<<nb, 256, 0, s>>>(1.0, b, -1.0, G.w.p, G.r.p, n);
      CB_LAUNCH();
      fused_dots(G, G.r.p, n, 1, G.r.p, n, nullptr, 1, G.h.p, nullptr, s);
      CB_CUDA(cudaMemcpyAsync(G.host_scal + 20, G.h.p, sizeof(double), cudaMemcpyDeviceToHost, s));
      CB_CUDA(cudaMemcpyAsync(G.host_scal, G.scal.p, 3 * sizeof(double), cudaMemcpyDeviceToHost, s));
      CB_CUDA(cudaStreamSynchronize(s));
      *relres_out = G.host_scal[2] > 0 ? std::sqrt(G.host_scal[20]) / G.host_scal[2] : 0.0;
      break;
    }
    // next cycle (or final check) recomputes the true residual
  }
  *iters_out = total;
  G.reorth = flags[3];
  return converged ? CBDDC_OK : CBDDC_ENOCONV;
}

double device_norm(fem_problem* P, Gmres& G, const double* v, cudaStream_t s) {
  G.ensure_small(P->n_free);
  fused_dots(G, v, P->n_free, 1, const_cast<double*>(v), P->n_free, nullptr, 1, G.h.p, nullptr, s);
  CB_CUDA(cudaMemcpyAsync(G.host_scal + 20, G.h.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  CB_CUDA(cudaStreamSynchronize(s));
  return std::sqrt(G.host_scal[20]);
}

void axpby(double a, const double* x, double b, const double* y, double* out, int64_t n, cudaStream_t s) {
  axpby_kernel<<<cdiv(n, 256), 256, 0, s>>>(a, x, b, y, out, n);
  CB_LAUNCH();
}

}  // namespace cbddc
