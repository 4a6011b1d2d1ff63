// Column-pivoted Householder QR truncated at |R_kk| <= eps |R_00| (the RRQR of
// Eq. 12) of W = [A_sn A_ns^T] (n x c, c ~ 10-30 n), with W in L2 / HBM and
// every column brought up to date only when it can be the next pivot.
//
// The pivot of step k is the column with the largest residual norm.  A residual
// norm never grows, so the norm a column had when it was last touched bounds
// its norm now.  The factorization therefore runs in bands: with m the largest
// bound of the remaining columns, the columns whose bound is at least m / f are
// brought up to date (the reflectors they have missed are applied in blocks of
// QRS_NB while the column stays in shared memory, and its norm is recomputed); those
// still at or above m / f are the band's active columns.  Pivot steps then
// touch the active columns alone, until the largest active norm falls below
// m / f: until then no other column can be the pivot.  A column that falls
// below m / f goes back to the waiting list with its norm as its new bound, and
// a column whose norm has fallen to eps |R_00| is dropped for good (the
// factorization stops before it could be chosen).  The pivots, the rank and Q
// are those of the plain column-pivoted QR; every column sees the same
// reflectors in the same order.
//
// What bounds it.  Updating every live column at every step moved 885 GB at the
// leaf level of the 256 x 128 p=3 grid (193 ms) and 1.27 TB in all (392 ms).  On W
// of that discretisation the band form touches 3 to 7 % of those column-steps at
// f = 1.5 to 2 and 1.4 % more for the bring-ups.  What is left is the arithmetic
// of the bring-ups (4 flops per element and missed reflector) and the latency of
// the r sequential pivot steps: 90 ms at the leaf level, 223 ms in all (64 x 32
// p=2: 11.3 ms before, 9.0 ms now; FP64 there 64 and 38 ms).
//
// Layout and work split.  W is column-major (column j at W + j*ldw, ldw a
// multiple of 16 bytes), V has its columns on 128-byte lines (ldv), so no line
// of a reflector is read before the whole reflector has been written.  The CTAs
// of a group own the columns j = q (mod G), interleaved so that strong and weak
// neighbour blocks spread evenly over the group.  In a pivot step a warp keeps CB
// whole columns in registers (16-byte loads, NV vectors per lane and column, all
// in flight at once); the bring-ups go through shared memory (qrs_band_pass).
//
// A pivot step of a group: every CTA publishes its best active column, or the
// largest bound of its waiting columns when it has none; when no CTA has an
// active column the same exchange starts the next band.  Every CTA then reads
// the winner's column from W (its owner wrote it before the exchange and never
// touches it again) and builds the same reflector; the owner writes it to V.
#pragma once
#include <algorithm>
#include <type_traits>

#include "dense.cuh"

namespace spand {

template <typename T>
struct QrStreamTask {
  T* W;              // n x c column-major, leading dimension ldw; overwritten
  T* V;              // reflector k in column k (ld ldv), rows k..n-1 (v_k[k] = 1), zero elsewhere
  T* tau;            // min(n, c)
  int n, c, ldw, ldv;
  int* rank;         // output
  unsigned long long* work;   // column elements the passes read and wrote
  int* li;           // column lists: QRS_LISTS int arrays and QRS_VALS T arrays of G * ceil(c / G) entries
  T* lv;
  T* gram;           // per CTA: min(n, c) x NB inner products of the reflectors of a block
};

// warps of a CTA: 16 where it has an SM to itself, 8 where two share one
__host__ __device__ constexpr int qrs_warps(bool wide) { return wide ? 16 : 8; }
// per CTA: ids and number of reflectors seen of the waiting columns (two
// buffers) and of the columns to bring up, the ids of the active ones; the
// waiting columns' norms^2 (two buffers)
constexpr int QRS_LISTS = 7, QRS_VALS = 2;

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  using V = float4;
  static constexpr int W = 4;
  __device__ static inline V load(const float* p) { return *reinterpret_cast<const float4*>(p); }
  __device__ static inline void store(float* p, const V& v) { *reinterpret_cast<float4*>(p) = v; }
  __device__ static inline float get(const V& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
  __device__ static inline void set(V& v, int i, float a) {
    if (i == 0) v.x = a;
    else if (i == 1) v.y = a;
    else if (i == 2) v.z = a;
    else v.w = a;
  }
};
template <>
struct Vec16<double> {
  using V = double2;
  static constexpr int W = 2;
  __device__ static inline V load(const double* p) { return *reinterpret_cast<const double2*>(p); }
  __device__ static inline void store(double* p, const V& v) { *reinterpret_cast<double2*>(p) = v; }
  __device__ static inline double get(const V& v, int i) { return i == 0 ? v.x : v.y; }
  __device__ static inline void set(V& v, int i, double a) {
    if (i == 0) v.x = a;
    else v.y = a;
  }
};

constexpr int QRS_NB = 8;                     // reflectors per block of the band pass

// One column pass at step k: y = tau (v^T w); w -= y v; returns the residual
// norm^2 over rows k+1..n-1.  Rows [kb, n) are processed (kb = k rounded down to
// a vector boundary; v is zero on rows < k, so those rows are unchanged), and
// read twice: for columns taller than a warp's registers hold.
template <typename T>
__device__ inline T qrs_column_tall(T* __restrict__ col, const T* __restrict__ v, T tau, int k, int kb, int n,
                                    int lane) {
  using VT = Vec16<T>;
  constexpr int VW = VT::W;
  T d = 0;
  for (int i0 = kb + lane * VW; i0 < n; i0 += 32 * VW) {
    const typename VT::V a = VT::load(col + i0), vv = VT::load(v + i0);
#pragma unroll
    for (int e = 0; e < VW; ++e) d += VT::get(vv, e) * VT::get(a, e);
  }
  d = warp_sum(d) * tau;
  T s = 0;
  for (int i0 = kb + lane * VW; i0 < n; i0 += 32 * VW) {
    typename VT::V a = VT::load(col + i0);
    const typename VT::V vv = VT::load(v + i0);
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      const T x = VT::get(a, e) - d * VT::get(vv, e);
      VT::set(a, e, x);
      if (i0 + e > k) s += x * x;
    }
    VT::store(col + i0, a);
  }
  return warp_sum(s);
}

// The same for CB columns at once held in registers (n - kb <= 32 NV VW), one
// read and one write: all their loads are in flight together, so a warp keeps
// CB x NV 16-byte loads per lane outstanding.  act[b] = false skips column b.  sres[b]: residual norm^2.
template <typename T, int NV, int CB>
__device__ inline void qrs_columns(T* const (&col)[CB], const bool (&act)[CB], const T* __restrict__ v, T tau,
                                   int k, int kb, int n, int lane, T (&sres)[CB]) {
  using VT = Vec16<T>;
  constexpr int VW = VT::W;
  typename VT::V r[CB][NV];
#pragma unroll
  for (int b = 0; b < CB; ++b)
#pragma unroll
    for (int t = 0; t < NV; ++t) {
      const int i0 = kb + (lane + 32 * t) * VW;
      if (act[b] && i0 < n) r[b][t] = VT::load(col[b] + i0);
    }
  T d[CB];
#pragma unroll
  for (int b = 0; b < CB; ++b) d[b] = 0;
#pragma unroll
  for (int t = 0; t < NV; ++t) {
    const int i0 = kb + (lane + 32 * t) * VW;
    if (i0 < n) {
      const typename VT::V vv = VT::load(v + i0);
#pragma unroll
      for (int b = 0; b < CB; ++b)
        if (act[b])
#pragma unroll
          for (int e = 0; e < VW; ++e) d[b] += VT::get(vv, e) * VT::get(r[b][t], e);
    }
  }
#pragma unroll
  for (int b = 0; b < CB; ++b) d[b] = warp_sum(d[b]) * tau;
  T sq[CB];
#pragma unroll
  for (int b = 0; b < CB; ++b) sq[b] = 0;
#pragma unroll
  for (int t = 0; t < NV; ++t) {
    const int i0 = kb + (lane + 32 * t) * VW;
    if (i0 < n) {
      const typename VT::V vv = VT::load(v + i0);
#pragma unroll
      for (int b = 0; b < CB; ++b)
        if (act[b]) {
#pragma unroll
          for (int e = 0; e < VW; ++e) {
            const T a = VT::get(r[b][t], e) - d[b] * VT::get(vv, e);
            VT::set(r[b][t], e, a);
            if (i0 + e > k) sq[b] += a * a;
          }
          VT::store(col[b] + i0, r[b][t]);
        }
    }
  }
#pragma unroll
  for (int b = 0; b < CB; ++b) sres[b] = warp_sum(sq[b]);
}

// FP32 groups exchange their proposals in one word per CTA and exchange: the
// proposal's norm^2 (float bits, high half) and column index (bits 8..31, all
// ones for a bound of waiting columns) with the exchange's tag (its number mod
// 256, bits 0..7).  A CTA makes its column updates visible, then stores its
// word; the others poll every word of the group until all carry this tag, which
// is the barrier and the proposals' gather in one L2 round trip.  Words are
// double-buffered by parity (a CTA is at most one exchange ahead of the
// slowest).
__device__ inline unsigned long long qrs_pack(float v, int i, int k) {
  return ((unsigned long long)__float_as_uint(v) << 32) | ((unsigned long long)(unsigned)i << 8) |
         (unsigned long long)(k & 255);
}

// NB consecutive reflectors are applied in one go (the compact WY form): with
// d = V_b^T w, the factors of the reflectors are
//   y_j = tau_j (d_j - sum_{i<j} (v_j^T v_i) y_i),      w -= V_b y.
// Applied one at a time, each reflector costs a load, a reduction over the warp
// and an update in sequence (about a microsecond); the reflectors a late column
// has missed then take longer than the pivot steps themselves (leaf level of
// 256 x 128 p=3: 255 ms against 193 ms for the plain streaming form).

// Sums of NB values (8 or 16) over the warp by halving exchanges: lane l holds
// the sum of x[l / (32 / NB)].
template <typename T, int NB>
__device__ inline T qrs_sum_many(T (&x)[NB], int lane) {
  int o = 16;
#pragma unroll
  for (int h = NB / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool hi = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const T send = hi ? x[i] : x[i + h];
      x[i] = (hi ? x[i + h] : x[i]) + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
#pragma unroll
  for (int q = 16 / NB; q >= 1; q >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], q);
  return x[0];
}

// Inner products of the reflectors [k0, k) with those before them in their
// block (blocks of NB from `base` on): gram[j NB + i] = v_j^T v_{q0 + i}; a warp
// per reflector.  Every CTA of a group fills its own copy (a few hundred dot
// products per band), which needs no exchange.
template <typename T, int NB, int NW>
__device__ inline void qrs_gram(const T* V, int ldv, T* gram, int base, int k0, int k, int n) {
  using VT = Vec16<T>;
  constexpr int VW = VT::W;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll 1
  for (int j = k0 + wid; j < k; j += NW) {
    const int q0 = base + (j - base) / NB * NB;
    const T* w = V + (size_t)j * ldv;
    T d[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) d[i] = 0;
#pragma unroll 1
    for (int i0 = (j & ~(VW - 1)) + lane * VW; i0 < n; i0 += 32 * VW) {
      const typename VT::V a = VT::load(w + i0);
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const typename VT::V b = VT::load(V + (size_t)min(q0 + i, j) * ldv + i0);
#pragma unroll
        for (int e = 0; e < VW; ++e) d[i] += VT::get(a, e) * VT::get(b, e);
      }
    }
    const T g = qrs_sum_many<T, NB>(d, lane);
    if (lane % (32 / NB) == 0) gram[(size_t)j * NB + lane / (32 / NB)] = g;
  }
}

// Appends up to 32 entries (one per lane with put) to a list of the CTA; the
// order of a list never changes a result (columns are independent, ties go to
// the lowest index).
__device__ inline int qrs_append(int* count, bool put, int lane) {
  const unsigned m = __ballot_sync(0xffffffffu, put);
  if (!m) return -1;
  int base = 0;
  if (lane == 0) base = atomicAdd(count, __popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  return put ? base + __popc(m & ((1u << lane) - 1)) : -1;
}

// A CTA's column lists (QRS_LISTS int and QRS_VALS T arrays, one every `stride`)
// and the state the passes below share with the pivot loop.
template <typename T>
struct QrsState {
  int* li;
  T* lv;
  size_t stride;
  int* cnt;                   // shared: entries of waiting buffers 0 and 1, to bring up, active
  int cur;                    // the waiting buffer in use
  T tau2, cut2;               // band threshold, drop threshold (norm^2)
  T best, wmax;               // the warp's best active column and largest waiting bound
  int bi;
  unsigned long long work;
  __device__ int& w_id(int buf, int t) { return li[buf * stride + t]; }
  __device__ int& w_last(int buf, int t) { return li[(2 + buf) * stride + t]; }
  __device__ int& b_id(int t) { return li[4 * stride + t]; }
  __device__ int& b_last(int t) { return li[5 * stride + t]; }
  __device__ int& a_id(int t) { return li[6 * stride + t]; }
  __device__ T& w_s(int buf, int t) { return lv[buf * stride + t]; }
  // a column of norm^2 s belongs to the band (a NaN cut, from a non-finite W with eps = 0, excludes nothing)
  __device__ bool in_band(T s) const { return s >= tau2 && (s > cut2 || !(cut2 == cut2)); }
  // lane 0: column j back to the waiting list, with k reflectors seen and norm^2 s
  __device__ void wait(int j, int k, T s, int lane) {
    if (lane == 0) {
      const int at = atomicAdd(cnt + cur, 1);
      w_id(cur, at) = j;
      w_last(cur, at) = k;
      w_s(cur, at) = s;
    }
    if (s > wmax) wmax = s;
  }
};

// Dynamic shared memory: the reflector (ldw values), then the band pass's: one
// or two buffers of NB reflectors, and per column of a pass the column itself,
// the partial d and norm^2 of every row group, y, id and reflectors seen.
constexpr int QRS_MB = 64;                    // columns per pass at most
template <typename T, int NB, int NW>
struct QrsRoom {
  int nbuf, mb;                               // reflector buffers, columns per pass; mb = 0: nothing fits
  __host__ __device__ static constexpr int per_col(int ldw) { return ldw + NW * (NB + 1) + NB + 4; }
  // `vals` values of T: two buffers when a pass then still has 16 columns
  __host__ __device__ static QrsRoom of(long long vals, int ldw) {
    QrsRoom r{2, 0};
    long long m = (vals - 2ll * NB * ldw) / per_col(ldw);
    if (m < 16) {
      r.nbuf = 1;
      m = (vals - (long long)NB * ldw) / per_col(ldw);
    }
    r.mb = m < 1 ? 0 : m > QRS_MB ? QRS_MB : m >= 4 ? (int)m / 4 * 4 : (int)m;
    return r;
  }
  // Bytes a CTA asks for: room for a pass of QRS_MB columns, or what fits the
  // budget (an SM to itself, or half of one).  Columns too tall for it are
  // worked on in global memory (partial d and y of a pass of 16 columns on chip).
  static size_t bytes(int ldw, bool wide) {
    const size_t least = (size_t)ldw + 16 * (size_t)per_col(0);
    const size_t most = (size_t)ldw + 2 * (size_t)NB * ldw + QRS_MB * (size_t)per_col(ldw);
    const size_t budget = (wide ? 220 : 110) * 1024 / sizeof(T);
    return std::max(least, std::min(budget, most)) * sizeof(T);
  }
};
template <typename T>
inline size_t qrcp_stream_smem(int ldw, bool wide) {
  return wide ? QrsRoom<T, QRS_NB, qrs_warps(true)>::bytes(ldw, true)
              : QrsRoom<T, QRS_NB, qrs_warps(false)>::bytes(ldw, false);
}

// Sums over the 8 lanes l & 7 of a quarter warp, by halving exchanges: of the M
// values, lane l ends with the sums of x[(l & 7) M / 8 + i], i < M / 8, in x[i].
template <typename T, int M>
__device__ inline void qrs_sum8(T (&x)[M], int lane) {
  int o = 4;
#pragma unroll
  for (int h = M / 2; h >= M / 8; h >>= 1, o >>= 1) {
    const bool hi = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const T send = hi ? x[i] : x[i + h];
      x[i] = (hi ? x[i + h] : x[i]) + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
}

// The columns to bring up (nb of them, each having seen at least the reflectors
// below `base`): through the reflectors up to k - 1, then put among the active
// or the waiting columns, or dropped.  A pass takes as many columns as shared
// memory holds (at most QRS_MB), reads them once (rows from the first missed
// reflector on), applies every missed reflector to them NB at a time, and writes
// rows k..n-1 back (R is never needed, only V).  The reflectors come through
// shared memory too, the next block's copied while this one is applied: read
// from L2 by each warp, a block of 8 took 20,000 cycles.  The whole CTA works on one
// block of reflectors: warps are split RS x CS over the rows and the columns
// (whichever split leaves the longest warp shortest), so that few columns (a late
// band has a handful per CTA) still use every warp and a block's latency is two
// passes over a warp's rows and three barriers.  In a warp the 32 lanes are 8
// row lanes x 4 column lanes, and a lane accumulates NB x CB products over all its
// rows before one reduction over the row lanes.  (With 32 row lanes the reduction
// after every slice of 128 rows cost several times the multiply-adds: 7 % of the
// kernel's instructions were FFMA.)  Reflectors a column has seen, and those past
// k - 1 (never read), get y = 0.  Not inlined: its registers then do not compete
// with the pivot loop's state.
template <typename T, int NB, int CB, int NW>
__device__ __noinline__ void qrs_band_pass(const QrStreamTask<T>& tk, QrsState<T>& S, const T* gram, int nb, int base,
                                           int k, T* sm, int room) {
  using VT = Vec16<T>;
  constexpr int VW = VT::W, RW = 8 * VW, BW = 4 * CB;   // rows per step, columns per batch
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, rl = lane & 7, cl = lane >> 3;
  const int n = tk.n, ldv = tk.ldv, ldw = tk.ldw;
  const T* const V = tk.V;
  T* const W = tk.W;
  const QrsRoom<T, NB, NW> R = QrsRoom<T, NB, NW>::of(room, ldw);
  const bool on_chip = R.mb > 0;
  const int mb = on_chip ? R.mb : 16;
  T* const sv = sm;                           // [nbuf][NB][ldw]
  T* const sw = sv + (on_chip ? (size_t)R.nbuf * NB * ldw : 0);   // [mb][ldw]
  T* const sy = sw + (on_chip ? (size_t)mb * ldw : 0);            // [mb][NB]
  T* const sd = sy + (size_t)mb * NB;         // [RS][mb][NB]
  T* const ss = sd + (size_t)NW * mb * NB;    // [RS][mb]
  int* const sid = reinterpret_cast<int*>(ss + (size_t)NW * mb);
  int* const sla = sid + mb;
  // reflectors [q0, min(q0 + NB, k)) into buffer `buf`, rows from the first step's on
  auto fetch = [&](int q0, int buf) {
    for (int j = wid; j < min(NB, k - q0); j += NW) {
      const T* src = V + (size_t)(q0 + j) * ldv;
      T* dst = sv + ((size_t)buf * NB + j) * ldw;
      for (int i0 = q0 / RW * RW + lane * VW; i0 < n; i0 += 32 * VW)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                         (unsigned)__cvta_generic_to_shared(dst + i0)),
                     "l"(src + i0)
                     : "memory");
    }
  };
#pragma unroll 1
  for (int p0 = 0; p0 < nb; p0 += mb) {
    const int mc = min(mb, nb - p0);
    for (int t = threadIdx.x; t < mc; t += 32 * NW) {
      sid[t] = S.b_id(p0 + t);
      sla[t] = S.b_last(p0 + t);
    }
    __syncthreads();
    int lo = k;                               // the pass's first missed reflector
    for (int t = lane; t < mc; t += 32) lo = min(lo, sla[t]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    const int qlo = base + (lo - base) / NB * NB;
    if (on_chip) {
      // every column's rows from the first block's on, all copies in flight
      for (int c = wid; c < mc; c += NW) {
        const T* src = W + (size_t)sid[c] * ldw;
        for (int i0 = qlo / RW * RW + lane * VW; i0 < n; i0 += 32 * VW) {
          const unsigned dst = (unsigned)__cvta_generic_to_shared(sw + (size_t)c * ldw + i0);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src + i0) : "memory");
        }
      }
      fetch(qlo, 0);
      cp_async_commit();
    }
    int RS = 1, buf = 0;
#pragma unroll 1
    for (int q0 = qlo; q0 < k; q0 += NB) {
      const int r0 = q0 / RW * RW;            // the rows above are left alone by the block
      // (the split follows nb, not this pass's count: which pass a column falls
      // into varies with the order of the lists, its sums must not)
      const int nst = (n - r0 + RW - 1) / RW, nbt = (min(nb, mb) + BW - 1) / BW;
      RS = NW;
      for (int cs = 2; cs <= NW; cs *= 2)     // fewest (row step, batch) pairs in the longest warp
        if (((nbt + cs - 1) / cs) * ((nst * cs + NW - 1) / NW) <
            ((nbt + NW / RS - 1) / (NW / RS)) * ((nst + RS - 1) / RS))
          RS = NW / cs;
      const int CS = NW / RS, rg = wid / CS, cg = wid % CS;
      const bool fin = q0 + NB >= k;
      const int vstep = min(NB, k - q0) - 1;  // reflectors past k - 1 are read as the last one (y = 0)
      if (on_chip) {
        cp_async_wait<0>();
        __syncthreads();
        if (R.nbuf == 2 && !fin) {
          fetch(q0 + NB, buf ^ 1);
          cp_async_commit();
        }
      }
      const T* const vb = on_chip ? sv + (size_t)buf * NB * ldw : V + (size_t)q0 * ldv;
      const int ldb = on_chip ? ldw : ldv;
      // tau and the Gram row of this lane's y, loaded before they are needed
      const int me = q0 + lane;
      const bool mine = lane < NB && me < k;
      const T tl = mine ? __ldcg(tk.tau + me) : (T)0;
      T g[NB];
#pragma unroll
      for (int i = 0; i < NB; ++i) g[i] = (mine && lane > i) ? gram[(size_t)me * NB + i] : (T)0;
      // ---- d = V_b^T w
#pragma unroll 1
      for (int c0 = cg * BW; c0 < mc; c0 += CS * BW) {
        T d[CB * NB];
        const T* col[CB];
#pragma unroll
        for (int b = 0; b < CB; ++b) {
          const int c = min(c0 + cl * CB + b, mc - 1);
          col[b] = on_chip ? sw + (size_t)c * ldw : W + (size_t)sid[c] * ldw;
#pragma unroll
          for (int j = 0; j < NB; ++j) d[b * NB + j] = 0;
        }
#pragma unroll 1
        for (int st = rg; st < nst; st += RS) {
          const int i0 = r0 + st * RW + rl * VW;
          if (i0 >= n) continue;
          const T* vp = vb + i0;
          typename VT::V w[CB], v[NB];
#pragma unroll
          for (int j = 0; j < NB; ++j) v[j] = VT::load(vp + min(j, vstep) * ldb);
#pragma unroll
          for (int b = 0; b < CB; ++b) w[b] = VT::load(col[b] + i0);
#pragma unroll
          for (int j = 0; j < NB; ++j)
#pragma unroll
            for (int b = 0; b < CB; ++b)
#pragma unroll
              for (int e = 0; e < VW; ++e) d[b * NB + j] += VT::get(v[j], e) * VT::get(w[b], e);
        }
        __syncwarp();
        qrs_sum8<T, CB * NB>(d, lane);
        constexpr int PER = CB * NB / 8;      // sums a lane holds: column rl PER / NB of its four
        const int c = c0 + cl * CB + rl * PER / NB;
        if (c < mc)
#pragma unroll
          for (int i = 0; i < PER; ++i) sd[((size_t)rg * mb + c) * NB + (rl * PER) % NB + i] = d[i];
      }
      __syncthreads();
      // ---- y, a warp per column (four at a time), lane j on y_j
      {
#pragma unroll 1
        for (int c0 = wid * 4; c0 < mc; c0 += NW * 4) {
          T y[4], tb[4];
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const int c = min(c0 + b, mc - 1);
            y[b] = 0;
            if (lane < NB)
              for (int r = 0; r < RS; ++r) y[b] += sd[((size_t)r * mb + c) * NB + lane];
            tb[b] = me >= sla[c] ? tl : (T)0;
          }
#pragma unroll
          for (int i = 0; i < NB - 1; ++i)
#pragma unroll
            for (int b = 0; b < 4; ++b) y[b] -= g[i] * __shfl_sync(0xffffffffu, tb[b] * y[b], i);
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (lane < NB && c0 + b < mc) sy[(size_t)(c0 + b) * NB + lane] = tb[b] * y[b];
        }
      }
      __syncthreads();
      // ---- w -= V_b y; the last block writes W and sums the norms^2 of rows k..n-1
#pragma unroll 1
      for (int c0 = cg * BW; c0 < mc; c0 += CS * BW) {
        T y[CB * NB], sq[CB];
        T *col[CB], *out[CB];
        bool in[CB];
#pragma unroll
        for (int b = 0; b < CB; ++b) {
          const int c = min(c0 + cl * CB + b, mc - 1);
          in[b] = c0 + cl * CB + b < mc;
          out[b] = W + (size_t)sid[c] * ldw;
          col[b] = on_chip ? sw + (size_t)c * ldw : out[b];
          if (!fin) out[b] = col[b];
          sq[b] = 0;
#pragma unroll
          for (int j = 0; j < NB; j += VW) {
            const typename VT::V yv = VT::load(sy + (size_t)c * NB + j);
#pragma unroll
            for (int u = 0; u < VW; ++u) y[b * NB + j + u] = VT::get(yv, u);
          }
        }
#pragma unroll 1
        for (int st = rg; st < nst; st += RS) {
          const int i0 = r0 + st * RW + rl * VW;
          if (i0 >= n) continue;
          const T* vp = vb + i0;
          typename VT::V w[CB], v[NB];
#pragma unroll
          for (int j = 0; j < NB; ++j) v[j] = VT::load(vp + min(j, vstep) * ldb);
#pragma unroll
          for (int b = 0; b < CB; ++b) w[b] = VT::load(col[b] + i0);
#pragma unroll
          for (int j = 0; j < NB; ++j)
#pragma unroll
            for (int b = 0; b < CB; ++b)
#pragma unroll
              for (int e = 0; e < VW; ++e)
                VT::set(w[b], e, VT::get(w[b], e) - y[b * NB + j] * VT::get(v[j], e));
#pragma unroll
          for (int b = 0; b < CB; ++b) {
#pragma unroll
            for (int e = 0; e < VW; ++e)
              if (i0 + e >= k) sq[b] += VT::get(w[b], e) * VT::get(w[b], e);
            if (in[b]) VT::store(out[b] + i0, w[b]);
          }
        }
        __syncwarp();
        if (fin)
#pragma unroll
          for (int b = 0; b < CB; ++b) {
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) sq[b] += __shfl_xor_sync(0xffffffffu, sq[b], o);
            if (rl == 0 && in[b]) ss[(size_t)rg * mb + c0 + cl * CB + b] = sq[b];
          }
      }
      __syncthreads();                        // the next block deals rows and columns anew
      if (on_chip && !fin) {
        if (R.nbuf == 1) {
          fetch(q0 + NB, 0);
          cp_async_commit();
        } else {
          buf ^= 1;
        }
      }
    }
    // ---- where each column goes now (warps 0 and 1, a lane per column)
    if (wid * 32 < mc) {
      const int t = wid * 32 + lane;
      const bool in = t < mc;
      const int id = in ? sid[t] : 0;
      T s = 0;
      for (int r = 0; r < RS; ++r) s += in ? ss[(size_t)r * mb + t] : (T)0;
      int el = in ? n - sla[t] : 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) el += __shfl_xor_sync(0xffffffffu, el, o);
      S.work += (unsigned long long)el;
      const bool act = in && S.in_band(s), wait = in && !act && s > S.cut2;
      int at = qrs_append(S.cnt + 3, act, lane);
      if (act) {
        S.a_id(at) = id;
        argmax_pair(S.best, S.bi, s, id);
      }
      at = qrs_append(S.cnt + S.cur, wait, lane);
      if (wait) {
        S.w_id(S.cur, at) = id;
        S.w_last(S.cur, at) = k;
        S.w_s(S.cur, at) = s;
        if (s > S.wmax) S.wmax = s;
      }
    }
    __syncthreads();
  }
  warp_argmax(S.best, S.bi);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S.wmax = fmax(S.wmax, __shfl_xor_sync(0xffffffffu, S.wmax, o));
}

// Step k: the reflector (v, tau) on every active column of this warp (cnt of
// them, groups of CB entries wid, wid + NW, ...) but the pivot column p;
// exact norms; keep, put back or drop.  Returns how many the warp keeps.
template <typename T, int NV, int CB, int NW>
__device__ __forceinline__ int qrs_step_pass(const QrStreamTask<T>& tk, QrsState<T>& S, const T* v, T tau, int p, int k,
                                          int cnt) {
  constexpr int VW = Vec16<T>::W;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, n = tk.n, kb = k & ~(VW - 1);
  auto place = [&](int t) { return ((t / CB) * NW + wid) * CB + t % CB; };
  int kept = 0;
#pragma unroll 1
  for (int t = 0; t < cnt; t += CB) {
    int js[CB];
    bool act[CB];
    T* cols[CB];
    T sres[CB];
#pragma unroll
    for (int b = 0; b < CB; ++b) {
      js[b] = (t + b < cnt) ? S.a_id(place(t + b)) : -1;
      act[b] = js[b] >= 0 && js[b] != p;      // the pivot column is done (warp-uniform)
      cols[b] = tk.W + (size_t)(act[b] ? js[b] : 0) * tk.ldw;
    }
    __syncwarp();
    if (n - kb <= 32 * VW * NV) {
      qrs_columns<T, NV, CB>(cols, act, v, tau, k, kb, n, lane, sres);
    } else {
#pragma unroll
      for (int b = 0; b < CB; ++b)
        sres[b] = act[b] ? qrs_column_tall<T>(cols[b], v, tau, k, kb, n, lane) : (T)-1;
    }
#pragma unroll
    for (int b = 0; b < CB; ++b)
      if (act[b]) {
        S.work += (unsigned long long)(n - k);
        if (S.in_band(sres[b])) {
          if (lane == 0) S.a_id(place(kept)) = js[b];   // kept <= the entry's own index: compacted in place
          ++kept;
          argmax_pair(S.best, S.bi, sres[b], js[b]);
        } else if (sres[b] > S.cut2) {
          S.wait(js[b], k + 1, sres[b], lane);
        }
      }
    __syncwarp();
  }
  return kept;
}

// Once this many reflectors have been built since the last time, a band brings
// up every waiting column, not just its own: a column then never misses more
// than this and a band's steps, so a late band does not wait for a few columns'
// long chains of blocks while most warps idle.  Factorization and solve of 64 x 32
// p=2 and 256 x 128 p=3 (ms): 32 34.6 and 817, 64 35.1 and 819, 128 36.3 and 820,
// never 39.8 and 967.
constexpr int QRS_FLUSH = 64;

// A CTA with no more than this many column elements takes every live column into
// the first band: passing over all of them costs less than bands do.
constexpr int QRS_ALL_IN = 32768;

// Band width f^2.  A wide band costs column passes (more active columns than
// can be pivots soon), a narrow one costs a scan and an exchange per few steps;
// so bands of many steps narrow and bands of few steps widen.  The same two
// systems: f = 1.25 throughout 36.7 and 821, 1.5 35.2 and 832, 2 34.9 and 861,
// this rule 35.1 and 819 ms.
template <typename T>
__device__ inline T qrs_band(T f2, int steps) {
  if (steps > 32) return (T)1.5625;           // f = 1.25
  if (steps < 6) return (T)4;                 // f = 2
  return steps >= 12 ? (T)2.25 : f2;          // f = 1.5
}

// The factorization of one interface by the CTA of rank q in a group of G
// (G = 1: a CTA alone, no exchange).  Gx is the group size the exchange waits
// for (G, or G + 1 when a test makes the wait run out).
template <typename T, int NV, int CB, int NB, int BC, int NW>
__device__ bool qrs_task(const QrStreamTask<T>& tk, int q, int G, int Gx, T* prop_v, int* prop_i, GroupSync* gs,
                         unsigned long long* words, int* err, T eps, long poll_limit, unsigned char* smem, int smem_bytes) {
  using VT = Vec16<T>;
  constexpr int VW = VT::W;
  __shared__ T red_v[NW], red_m[NW], red_s[NW];
  __shared__ int red_i[NW];
  __shared__ T s_val, s_alpha;
  __shared__ int s_win, s_ok;
  __shared__ int s_cnt[4];                    // entries of waiting buffers 0 and 1, to bring up, active
  constexpr bool kWords = std::is_same<T, float>::value;
  GroupX<T> xc{q, Gx, prop_v, prop_i, gs, err, nullptr, 0};
  xc.poll_limit = poll_limit;
  const int n = tk.n, c = tk.c, ldw = tk.ldw, ldv = tk.ldv;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  T* v = reinterpret_cast<T*>(smem);
  const int per_cta = (c + G - 1) / G;
  QrsState<T> S;
  S.li = tk.li + (size_t)q * per_cta;
  S.lv = tk.lv + (size_t)q * per_cta;
  S.stride = (size_t)per_cta * G;
  S.cnt = s_cnt;
  S.cur = 0;
  S.tau2 = S.cut2 = 0;
  S.best = S.wmax = -1;
  S.bi = c;
  S.work = 0;
  // the reflector buffer past row n stays zero (padding rows of W are zero)
  for (int i = tid; i < ldw; i += 32 * NW) v[i] = 0;
  const int ncol = q < c ? (c - q + G - 1) / G : 0;   // this CTA's columns j = q + G m
  if (tid < 4) s_cnt[tid] = tid == 0 ? ncol : 0;
  // ---- exact norms of all columns: the first bounds
  for (int m0 = wid * 4; m0 < ncol; m0 += NW * 4) {
    T s4[4] = {0, 0, 0, 0};
    for (int i0 = lane * VW; i0 < n; i0 += 32 * VW)
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (m0 + b < ncol) {
          const typename VT::V a = VT::load(tk.W + (size_t)(q + (long long)G * (m0 + b)) * ldw + i0);
#pragma unroll
          for (int e = 0; e < VW; ++e) s4[b] += VT::get(a, e) * VT::get(a, e);
        }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const T s = warp_sum(s4[b]);
      if (m0 + b < ncol) {
        if (lane == 0) {
          S.w_id(0, m0 + b) = q + G * (m0 + b);
          S.w_last(0, m0 + b) = 0;
          S.w_s(0, m0 + b) = s;
        }
        if (s > S.wmax) S.wmax = s;
      }
    }
  }
  const int kmax = min(n, c);
  T* const gram = tk.gram + (size_t)q * kmax * NB;
  const bool all_in = (long long)n * per_cta <= QRS_ALL_IN;
  const int room = smem_bytes / (int)sizeof(T) - ldw;   // values of T the band pass may use
  int rank = kmax, k = 0, band_k = 0, gram_k = 0, base = 0, nact = 0, cnt = 0;
  unsigned ex = 0;                            // exchanges so far
  T nrm0 = 0, f2 = (T)2.25;
  bool first = true, ok = true;
  while (k < kmax) {
    // ---- this CTA's proposal: its S.best active column, else its largest bound
    if (lane == 0) {
      red_v[wid] = S.best;
      red_i[wid] = S.bi;
      red_m[wid] = S.wmax;
    }
    __syncthreads();
    T gb = lane < NW ? red_v[lane] : (T)-1, gm = lane < NW ? red_m[lane] : (T)-1;
    int gi = lane < NW ? red_i[lane] : c;
    warp_argmax(gb, gi);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    if (Gx > 1) {
      if (kWords) {
        if (tid == 0) {
          __threadfence();                    // this CTA's column updates before its word
          volatile unsigned long long* wq = words + (size_t)(ex & 1) * QR_GMAX + q;
          *wq = gi < c ? qrs_pack((float)gb, gi, (int)ex) : qrs_pack((float)gm, 0xFFFFFF, (int)ex);
        }
        if (tid < 32) {
          gb = gm = -1;
          gi = c;
          bool wok = true;
          for (int r = lane; r < Gx && wok; r += 32) {
            volatile unsigned long long* wr = words + (size_t)(ex & 1) * QR_GMAX + r;
            unsigned long long w = 0;
            long it = 0;
            while (true) {
              w = *wr;
              if ((unsigned)(w & 255ull) == (ex & 255u)) break;
              if (++it > poll_limit) {
                wok = false;
                break;
              }
              if (it > 2048) __nanosleep(64);
            }
            if (wok) {
              const T wv = (T)__uint_as_float((unsigned)(w >> 32));
              const int wi = (int)((w >> 8) & 0xFFFFFFull);
              if (wi != 0xFFFFFF) argmax_pair(gb, gi, wv, wi);
              else if (wv > gm) gm = wv;
            }
          }
          wok = __all_sync(0xffffffffu, wok);
          __threadfence();                    // the others' column updates are visible from here on
          warp_argmax(gb, gi);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
          if (lane == 0) {
            s_val = gi < c ? gb : gm;
            s_win = gi;
            s_ok = wok ? 1 : 0;
            if (!wok) atomicOr(err, 16);
          }
        }
        __syncthreads();
        if (!s_ok) {
          ok = false;
          break;
        }
      } else {
        if (tid == 0) xc.publish(gi < c ? gb : gm, gi);
        if (!(ok = xc.sync())) break;
        if (tid < 32) {
          gb = gm = -1;
          gi = c;
          for (int r = lane; r < G; r += 32) {
            T pv;
            int pi;
            xc.gather(r, pv, pi);
            if (pi < c) argmax_pair(gb, gi, pv, pi);
            else if (pv > gm) gm = pv;
          }
          warp_argmax(gb, gi);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
          if (lane == 0) {
            s_val = gi < c ? gb : gm;
            s_win = gi;
          }
        }
        xc.next_step();
        __syncthreads();
      }
      gb = gm = s_val;
      gi = s_win;
    }
    ++ex;
    const int p = gi;
    if (p >= c) {
      // ---- no active column anywhere: the next band
      const T nrm = sqrt(fmax(gm, (T)0));
      if (first) {
        nrm0 = nrm;
        S.cut2 = (eps * nrm0) * (eps * nrm0);
        first = false;
      } else {
        f2 = qrs_band<T>(f2, k - band_k);
      }
      if (nrm0 == (T)0 || nrm <= eps * nrm0 || gm < (T)0) {
        rank = k;
        break;
      }
      S.tau2 = all_in ? (T)0 : gm / f2;
      band_k = k;
      const int nxt = S.cur ^ 1;
      S.best = -1;
      S.bi = c;
      S.wmax = -1;
      __syncthreads();                        // the red_* arrays and lists of the last phase are no longer read
      if (tid == 0) {
        s_cnt[nxt] = 0;
        s_cnt[2] = 0;
        s_cnt[3] = 0;
      }
      const int nw = s_cnt[S.cur];
      __syncthreads();
      qrs_gram<T, NB, NW>(tk.V, ldv, gram, base, gram_k, k, n);
      gram_k = k;
      const bool flush = k - base >= QRS_FLUSH;
      // the waiting columns: drop, keep, or take into the band
      for (int t0 = wid * 32; t0 < nw; t0 += NW * 32) {
        const int t = t0 + lane;
        const bool in = t < nw;
        const int id = in ? S.w_id(S.cur, t) : 0, la = in ? S.w_last(S.cur, t) : 0;
        const T s = in ? S.w_s(S.cur, t) : (T)-1;
        const bool take = in && S.in_band(s);
        const bool now = take && la == k;     // nothing missed: its bound is its norm
        const bool live = in && !take && s > S.cut2;
        const bool keep = live && !(flush && la < k);
        const bool up = (take && !now) || (live && !keep);
        int at = qrs_append(&s_cnt[nxt], keep, lane);
        if (keep) {
          S.w_id(nxt, at) = id;
          S.w_last(nxt, at) = la;
          S.w_s(nxt, at) = s;
        }
        at = qrs_append(&s_cnt[2], up, lane);
        if (up) {
          S.b_id(at) = id;
          S.b_last(at) = la;
        }
        at = qrs_append(&s_cnt[3], now, lane);
        if (now) {
          S.a_id(at) = id;
          argmax_pair(S.best, S.bi, s, id);
        }
        if (keep && s > S.wmax) S.wmax = s;
      }
      warp_argmax(S.best, S.bi);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) S.wmax = fmax(S.wmax, __shfl_xor_sync(0xffffffffu, S.wmax, o));
      __syncthreads();
      S.cur = nxt;
      {
        QrsState<T> B = S;                    // a copy, so that S itself stays in registers
        qrs_band_pass<T, NB, BC, NW>(tk, B, gram, s_cnt[2], base, k, v + ldw, room);
        S = B;
      }
      if (flush) base = k;
      __syncthreads();
      // the active columns dealt CB at a time: warp w holds groups w, w + NW, ...
      nact = s_cnt[3];
      const int ngr = (nact + CB - 1) / CB, mg = ngr > wid ? (ngr - wid + NW - 1) / NW : 0;
      cnt = mg * CB;
      if (mg > 0 && (wid + (mg - 1) * NW + 1) * CB > nact) cnt -= (wid + (mg - 1) * NW + 1) * CB - nact;
      continue;
    }
    // ---- a pivot step on column p
    const T nrm = sqrt(fmax(gb, (T)0));
    if (nrm <= eps * nrm0) {
      rank = k;
      break;
    }
    const bool owner = (p % G) == q;
    const int kb = k & ~(VW - 1);
    // the reflector from column p (rows k..n-1), identical in every CTA
    const T* colp = tk.W + (size_t)p * ldw;
    T prt = 0;
    for (int i = kb + tid; i < n; i += 32 * NW) {
      const T x = (i < k) ? (T)0 : __ldcg(colp + i);
      v[i] = x;
      if (i > k) prt += x * x;
      if (i == k) s_alpha = x;
    }
    prt = warp_sum(prt);
    if (lane == 0) red_s[wid] = prt;
    __syncthreads();
    const T alpha = s_alpha;
    T sigma = 0;
    for (int w = 0; w < NW; ++w) sigma += red_s[w];
    T tau = 2, scale = 0;                     // column already reduced: H = I - 2 e_k e_k^T
    if (sigma > (T)0) {
      const T beta = -copysign(sqrt(alpha * alpha + sigma), alpha);
      tau = (beta - alpha) / beta;
      scale = (T)1 / (alpha - beta);
    }
    for (int i = kb + tid; i < n; i += 32 * NW) {   // the thread's own entries
      if (i < k) continue;
      const T vi = (i == k) ? (T)1 : v[i] * scale;
      v[i] = vi;
      if (owner) tk.V[(size_t)i + (size_t)k * ldv] = vi;
    }
    if (owner && tid == 0) tk.tau[k] = tau;
    __syncthreads();
    S.best = -1;
    S.bi = c;
    cnt = qrs_step_pass<T, NV, CB, NW>(tk, S, v, tau, p, k, cnt);
    ++k;
  }
  if (S.work && lane == 0 && tk.work) atomicAdd(tk.work, S.work);
  if (q == 0 && tid == 0) *tk.rank = ok ? rank : 0;
  __syncthreads();                          // smem is reused by the next task
  return ok;
}

// Step pass: NV vectors of rows per lane and column in registers; the shorter
// the columns, the more of them (CB) a warp holds.  Band pass: blocks of NB
// reflectors on BC columns.
template <typename T, bool WIDE>
__device__ bool qrs_dispatch(const QrStreamTask<T>& tk, int q, int G, int Gx, T* prop_v, int* prop_i, GroupSync* gs,
                             unsigned long long* words, int* err, T eps, long poll_limit, unsigned char* smem, int smem_bytes) {
  constexpr int VW = Vec16<T>::W, BC = 4 * (int)sizeof(float) / (int)sizeof(T), NW = qrs_warps(WIDE);
  if (tk.n <= 32 * VW * 4)
    return qrs_task<T, 4, 2, QRS_NB, BC, NW>(tk, q, G, Gx, prop_v, prop_i, gs, words, err, eps, poll_limit, smem,
                                             smem_bytes);
  if (tk.n <= 32 * VW * 8)
    return qrs_task<T, 8, 1, QRS_NB, BC, NW>(tk, q, G, Gx, prop_v, prop_i, gs, words, err, eps, poll_limit, smem,
                                             smem_bytes);
  return qrs_task<T, 16, 1, QRS_NB, BC, NW>(tk, q, G, Gx, prop_v, prop_i, gs, words, err, eps, poll_limit, smem,
                                            smem_bytes);
}

// The large interfaces: a cooperative launch of one CTA per SM, the groups of
// desc.  prop_v / prop_i / gs / words hold one slot per task.  fault_task >= 0:
// that task's exchange waits for one CTA more than it has (a test of the
// bounded wait).
template <typename T>
__global__ void __launch_bounds__(32 * qrs_warps(true), 1)
    k_qrcp_stream_group(const QrStreamTask<T>* tasks, const QrGroupDesc* desc, T* prop_v, int* prop_i, GroupSync* gs,
                        unsigned long long* words, int* err, T eps, int poll_log2, int fault_task,
                        int smem_bytes) {
  extern __shared__ __align__(16) unsigned char qrs_smem[];
  const QrGroupDesc d = desc[blockIdx.x];
  const size_t o = (size_t)d.task * 2 * QR_GMAX;
  qrs_dispatch<T, true>(tasks[d.task], d.q, d.G, d.G + (d.task == fault_task ? 1 : 0), prop_v + o, prop_i + o,
                       gs + d.task, words + o, err, eps, 1l << poll_log2, qrs_smem, smem_bytes);
}

// The other interfaces, one CTA each from a shared queue.  A pivot step of one
// is mostly latency (three block barriers, the pivot column's read), so two
// CTAs share an SM and fill each other's waits.
template <typename T>
__global__ void __launch_bounds__(32 * qrs_warps(false), 2)
    k_qrcp_stream_solo(const QrStreamTask<T>* tasks, const int* solo, int n_solo, int* queue, T* prop_v, int* prop_i,
                       GroupSync* gs, unsigned long long* words, int* err, T eps, int poll_log2, int fault_task,
                        int smem_bytes) {
  extern __shared__ __align__(16) unsigned char qrs_smem[];
  __shared__ int s_next;
  bool ok = true;
  while (ok) {
    if (threadIdx.x == 0) s_next = atomicAdd(queue, 1);
    __syncthreads();
    const int t = s_next;
    __syncthreads();
    if (t >= n_solo) break;
    const int task = solo[t];
    const size_t o = (size_t)task * 2 * QR_GMAX;
    ok = qrs_dispatch<T, false>(tasks[task], 0, 1, 1 + (task == fault_task ? 1 : 0), prop_v + o, prop_i + o, gs + task,
                              words + o, err, eps, 1l << poll_log2, qrs_smem, smem_bytes);
  }
}

}  // namespace spand
