// Batched gather-GEMV used by the spaND apply sweeps (Sec. 2.2.1: the
// preconditioner is the product of the stored elimination, scaling and
// orthogonal operators).  Every operator application is
//     y[yidx[i]] = base[bidx[i]] + alpha * sum_t (op(M_t) x_t)[i]
// with x_t[j] = src[xidx[j]] - xsub[j]; M null means the identity.  Matrices
// are column-major; tri marks a stored lower (1) / upper (2) triangle so the
// kernel skips the zero half.  The sweeps alternate two vectors so no launch
// reads what another CTA of the same launch writes.
//
// Bound: HBM (each matrix entry is read once per sweep), but a sweep is a chain
// of launches and on the upper levels each holds a few hundred rows, so what
// counts is how much of a tile is in flight at once.  One CTA takes 32 output
// rows; the 32-column chunks of all the task's terms are dealt round-robin to
// its warps.  A warp gathers a chunk's x values into registers (one per lane)
// and needs no barrier until the final sum over the warps, so every warp keeps
// 16 coalesced matrix loads in flight and terms do not wait for one another.
//   op(M) = M:   lane = output row, a load per column of the chunk;
//   op(M) = M^T: lane = column of the chunk, a load per output row (32 running
//                sums per lane, transposed over the warp once at the end).
// The sum over the warps has a fixed order: results do not vary between runs.
//
// A separator's cluster next to many boxes collects tens of thousands of columns
// (31 boxes of 1,400 unknowns at 192 x 96 p=3) where an ordinary tile has a few
// thousand, so long tiles are cut into pieces for several CTAs; the last one to
// finish adds the pieces in their order.
#pragma once
#include <cuda_runtime.h>

namespace spand {

template <typename T>
struct GvTerm {
  const T* M;
  const T* x;
  const int* xidx;
  const T* xsub;
  int ld, k, trans, tri;
};

template <typename T>
struct GvTask {
  T* y;
  const int* yidx;
  const T* base;
  const int* bidx;
  T* y2;
  T alpha;
  int m, t0, t1;
};

// chunks [c0, c1) of the task's flattened (term, chunk) sequence for the rows from
// r0 on; a tile cut in nseg pieces has partial sums at slot, slot + 1, ... and its
// counter at `slot`
struct GvTile {
  int task, r0, c0, c1, slot, seg, nseg;
};

constexpr int GV_ROWS = 32;
constexpr int GV_WARPS_MAX = 16;
constexpr int GV_MANY = 2432;                     // 32-row tiles that fill the GPU: 16 per SM
// chunks (of 32 columns) of a piece at least: 32, 64, 128 and no pieces take 109.6,
// 111.3, 111.9 and 111.9 ms in a solve of 192 x 96 p=3, 88.9, 87.1, 87.1 and 87.1 in
// one of 75 x 33 p=3
constexpr int GV_PIECE = 64;

// columns [jlo, jhi) of a term with possibly non-zero entries for the rows from r0
// on, and their 32-column chunks (1 for an identity)
template <int R, typename T>
__host__ __device__ inline int gv_chunks(const GvTerm<T>& tm, int r0, int& jlo, int& jhi) {
  jlo = 0;
  jhi = tm.k;
  if (!tm.M) return 1;
  if (tm.tri) {
    if ((tm.tri == 1) != (tm.trans != 0)) jhi = tm.k < r0 + GV_ROWS * R ? tm.k : r0 + GV_ROWS * R;
    else jlo = tm.k < r0 ? tm.k : r0;
  }
  return (jhi - jlo + 31) / 32;
}

// lane l: the sum over the warp of x[l] (halving exchanges: 31 shuffles)
template <typename T>
__device__ inline T gv_transpose_sum(T (&x)[32], int lane) {
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) {
    const bool hi = lane & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const T send = hi ? x[i] : x[i + h];
      x[i] = (hi ? x[i + h] : x[i]) + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  return x[0];
}

// TR: the phase's matrices are applied transposed (a phase never mixes the two;
// identity terms may join either)
// R: 32-row groups per tile (2 in phases of many tiles, where half the gathers
// per matrix entry count for more than tiles to spread; 1 with TR)
template <typename T, bool TR, int R>
__global__ void __launch_bounds__(32 * GV_WARPS_MAX) k_gemv(const GvTask<T>* tasks, const GvTerm<T>* terms,
                                                            const GvTile* tiles, T* partial, int* done) {
  static_assert(R == 1 || !TR, "transposed tiles have 32 rows");
  __shared__ T part[GV_WARPS_MAX][GV_ROWS * R];
  constexpr int U = (TR && sizeof(T) == 8 ? 8 : 16) / R;   // steps per batch of matrix loads (R U in flight per lane)
  const GvTile tl = tiles[blockIdx.x];
  const GvTask<T> tk = tasks[tl.task];
  const int r0 = tl.r0, rows = min(GV_ROWS * R, tk.m - r0);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T acc[R];                                       // lane = output row
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = 0;
  T run[TR ? 32 : 1];
#pragma unroll
  for (int r = 0; r < (TR ? 32 : 1); ++r) run[r] = 0;
  int base = 0;                                   // chunks of the terms before t
  for (int t = tk.t0; t < tk.t1 && base < tl.c1; ++t) {
    const GvTerm<T> tm = terms[t];
    int jlo, jhi;
    const int nch = gv_chunks<R>(tm, r0, jlo, jhi);
    // the warp's chunks: indices w (mod nw) of the flattened sequence
    int c = max(tl.c0, base);
    c += (w - c % nw + nw) % nw;
    const int ce = min(tl.c1, base + nch);
    if (!tm.M) {
      if (c < ce)
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (lane + 32 * r < rows) {
            const int j = r0 + lane + 32 * r;
            T v = tm.xidx ? tm.x[tm.xidx[j]] : tm.x[j];
            if (tm.xsub) v -= tm.xsub[j];
            acc[r] += v;
          }
      base += nch;
      continue;
    }
    for (; c < ce; c += nw) {
      const int j0 = jlo + 32 * (c - base), nj = min(32, jhi - j0), j = j0 + lane;
      const int xi = lane < nj ? (tm.xidx ? tm.xidx[j] : j) : 0;
      // op(M) = M: lane = row, the chunk's columns one by one; M^T: lane = column,
      // the tile's rows one by one.  The matrix loads are issued before the gather
      // waits for its index.
      const T* Mp = TR ? tm.M + j + (size_t)r0 * tm.ld : tm.M + (r0 + lane) + (size_t)j0 * tm.ld;
      const int nl = TR ? nj : rows, ns = TR ? rows : nj;   // lanes and steps in use
      T xv = 0;
#pragma unroll
      for (int u0 = 0; u0 < 32; u0 += U) {
        T m[R][U];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int r = 0; r < R; ++r)
            m[r][u] = (lane + 32 * r < nl && u0 + u < ns) ? Mp[(size_t)(u0 + u) * tm.ld + 32 * r] : (T)0;
        if (u0 == 0 && lane < nj) {
          xv = tm.x[xi];
          if (tm.xsub) xv -= tm.xsub[j];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (TR) {
            run[u0 + u] += m[0][u] * xv;
          } else {
            const T xu = __shfl_sync(0xffffffffu, xv, u0 + u);
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] += m[r][u] * xu;
          }
        }
      }
    }
    base += nch;
  }
  if constexpr (TR) acc[0] += gv_transpose_sum<T>(run, lane);
#pragma unroll
  for (int r = 0; r < R; ++r) part[w][lane + 32 * r] = acc[r];
  __syncthreads();
  const int i = r0 + threadIdx.x;
  T s = 0;
  if ((int)threadIdx.x < rows)
    for (int q = 0; q < nw; ++q) s += part[q][threadIdx.x];
  if (tl.nseg > 1) {
    __shared__ int last;
    if ((int)threadIdx.x < rows) partial[(size_t)(tl.slot + tl.seg) * 64 + threadIdx.x] = s;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      last = atomicAdd(done + tl.slot, 1) == tl.nseg - 1;
      if (last) done[tl.slot] = 0;                // for the next launch
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    s = 0;
    if ((int)threadIdx.x < rows)
      for (int q = 0; q < tl.nseg; ++q) s += __ldcg(partial + (size_t)(tl.slot + q) * 64 + threadIdx.x);
  }
  if ((int)threadIdx.x < rows) {
    T v = tk.alpha * s;
    if (tk.base) v += tk.bidx ? tk.base[tk.bidx[i]] : tk.base[i];
    if (tk.yidx) tk.y[tk.yidx[i]] = v;
    else tk.y[i] = v;
    if (tk.y2) tk.y2[i] = v;
  }
}

}  // namespace spand
