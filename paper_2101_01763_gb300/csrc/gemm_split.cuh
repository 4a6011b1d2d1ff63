// Grouped FP64 GEMM on the BF16 tensor cores: products of integers, exactly.
//
// Same task / term / tile contract as k_gemm<double>.  A GB300 has 2 FP64
// multiply-adds per clock and SM against 1,024 and more BF16 ones, so an FP64
// product is taken apart into BF16 products that are exact in the FP32
// accumulator (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012, with a common exponent per row):
//  * in a chunk of GS_K = 64 values of k, every row of op(A) and every column of
//    op(B) is scaled by its largest exponent to 70-bit integers and cut into
//    GS_S = 9 signed base-256 digits, |digit| <= 128, each exact in BF16;
//  * the digit products with s + t = L <= 8 (45 of them) are summed in FP32: at
//    most 9 x 64 terms of at most 2^14, below 2^24, so every sum is exact;
//  * the nine sums are joined in two 64-bit integers and added to the FP64
//    accumulator with two roundings per chunk.
//
// Error.  With E the product of the two scales (the powers of two at the largest
// entries), what is dropped (s + t >= 9: 8 pairs of at most 2^14 2^-138+56 E for
// each of 64 products) and the rounding of an entry to its 70 bits come to at most
// 2^-58.8 E per chunk, about 2^-65 E in the ordinary.  Multiply-adds keep
// 64 x 2^-53 of S, the sum of |a| |b|, per chunk, whatever the scales of rows,
// columns and values of k are; E can be far larger than S.  So
//  * value l of k is scaled by 2^s in op(A) and 2^-s in op(B), s half the
//    difference of the two operands' largest exponents there (exact, and (A D)
//    (D^-1 B) for diagonal D of powers of two is taken apart as A B is); values of
//    k at which either operand is zero throughout the tile are left out;
//  * a tenth plane holds |a| and |b| as BF16 numbers of the same scales, and its
//    product gives the chunk's S of every output;
//  * where E is above 2^GS_SPREAD times the largest S that the output has had in a
//    chunk so far, this chunk's part is summed in FP64 multiply-adds instead: what
//    the digits give is within 2^-47.8 S, less than the multiply-adds' 2^-47 S.
// A chunk with an infinity, a NaN, a denormal or a scale beyond 2^+-400 is summed in
// multiply-adds altogether.  A chunk of no value of k is passed over.
//
// Residual of a direct solve (eps = 0, 16 x 4 p=2) over |A| |z| + |r| for columns
// scaled by up to 2^+-10, 2^+-20 and 2^+-30: 1.2e-16 each time; 2.4e-16 in
// multiply-adds; 1.3e-13, 4.4e-8 and 4.9e-3 with eight digits on one scale per row.
//
// 64 x 32 p=2, useful TFLOP/s (the FP64 rate is 1.25) in multiply-adds and now: Y
// and X products 1.0, 6.1 (most chunks of sparse couplings hold nothing); Schur
// updates 1.0, 3.9; scaling 0.6, 1.5; compression 0.6, 1.2 (a quarter of its
// outputs lie so far below their rows' and columns' scales that a chunk of them is
// summed again); the factorization and solve 312 ms in multiply-adds, 159 ms now.
//
// Bound: the digits (integer arithmetic), 184 mma.sync per warp and 16 values of
// k, and 5 FP64 instructions per output and chunk (of 64 in the plain form).
#pragma once
#include <cstdint>

#include "dense.cuh"

namespace spand {

constexpr int GS_K = 64, GS_S = 9, GS_T = 64;             // chunk, digits, tile
constexpr int GS_SPREAD = 11;                             // log2 E / S up to which the digits are used
constexpr int GS_PITCH = GS_K * 2 + 16;                   // bytes of a row of one digit (conflict-free ldmatrix)
constexpr int GS_PLANE = GS_T * GS_PITCH;
constexpr int GS_OP_BYTES = (GS_S + 1) * GS_PLANE;        // the digits and |.| of one operand
constexpr int GS_SMEM_BYTES = 2 * GS_OP_BYTES + GS_T * GS_T * 2;   // and a list of outputs
constexpr int GS_RPITCH = GS_T + 1;                       // doubles per value of k of a chunk staged as it is
static_assert(2 * GS_K * GS_RPITCH * 8 + GS_T * GS_T * 8 <= 2 * GS_OP_BYTES, "a chunk and its sums fit the digits' room");
constexpr int GS_NONE = -30000;                           // exponent of a row without entries

__device__ inline void gs_ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

__device__ inline void gs_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ inline int gs_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// largest exponent of each of 16 values of k over the warp's 32 rows, to km[0..15];
// returns whether one of this thread's values is a denormal, an infinity or a NaN
__device__ inline bool gs_k_exponents(const double (&x)[16], unsigned short* km, int lane) {
  bool odd = false;
  uint32_t w[8];
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int e = gs_exponent(x[q]);
    odd |= e == 0x7ff || (e == 0 && x[q] != 0.0);
    const uint32_t m = __reduce_max_sync(0xffffffffu, (uint32_t)e);
    if ((q & 1) == 0) w[q >> 1] = m;
    else w[q >> 1] |= m << 16;
  }
  if (lane == 0) {
    *reinterpret_cast<uint4*>(km) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4*>(km + 8) = make_uint4(w[4], w[5], w[6], w[7]);
  }
  return odd;
}

// 16 consecutive k of one row (column): digits and |x| into `dst` (this row in
// digit 0).  Value q counts as x[q] 2^(sg shift[q]); emax: the row's largest exponent.
__device__ inline void gs_digits(const double (&x)[16], const int (&shift)[16], int sg, int emax, unsigned char* dst) {
  uint32_t w[GS_S + 1][2];                                // planes of a pair of pairs, packed
#pragma unroll
  for (int q = 0; q < 16; q += 4) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const long long b = __double_as_longlong(x[q + h]);
      const int e = gs_exponent(x[q + h]);
      const bool zero = e == 0;
      const int d = zero ? 0 : emax - (e + sg * shift[q + h]);   // >= 0
      const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
      // m 2^(17 - d), rounded; for d < 8 without its last 8 bits, which are zero
      long long f;
      if (d < 8) f = m << (9 - d);
      else if (d <= 17) f = m << (17 - d);
      else f = d <= 70 ? (m + (1ll << (d - 18))) >> (d - 17) : 0;
      if (zero) f = 0;
      if (b < 0) f = -f;
      const int last = d < 8 ? 0 : (int)(signed char)(f & 0xff);
      if (d >= 8) f = (f - last) >> 8;
#pragma unroll
      for (int s = GS_S - 1; s >= 0; --s) {
        int lo = last;
        if (s < GS_S - 1) {
          lo = (int)(signed char)(f & 0xff);
          f = (f - lo) >> 8;
        }
        // small integer -> BF16: the top half of its (exact) FP32
        const uint32_t v = __float_as_uint(__int_as_float(0x4B400000 + lo) - 12582912.0f) >> 16;
        if ((h & 1) == 0) w[s][h >> 1] = v;
        else w[s][h >> 1] |= v << 16;
      }
      const uint32_t v = zero || d > 126 ? 0u : ((uint32_t)(127 - d) << 7) | ((uint32_t)(b >> 45) & 0x7f);
      if ((h & 1) == 0) w[GS_S][h >> 1] = v;
      else w[GS_S][h >> 1] |= v << 16;
    }
#pragma unroll
    for (int s = 0; s <= GS_S; ++s) *reinterpret_cast<uint2*>(dst + s * GS_PLANE + q * 2) = make_uint2(w[s][0], w[s][1]);
  }
}

__global__ void __launch_bounds__(256, 1) k_gemm_split(const GemmTask<double>* tasks, const GemmTerm<double>* terms,
                                                       const TileItem* tiles) {
  extern __shared__ __align__(16) unsigned char gs_smem[];
  __shared__ __align__(16) unsigned short s_k[2][2][GS_K];   // largest exponent of a value of k in half the rows of A / columns of B
  __shared__ short s_part[2][4][GS_T];                    // largest exponent of a quarter row of A / column of B
  __shared__ short s_e[2][GS_T];                          // of the whole row / column
  __shared__ int s_n;                                     // outputs in the list
  const TileItem it = tiles[blockIdx.x];
  const GemmTask<double> tk = tasks[it.task];
  const int i0 = it.tm * GS_T, j0 = it.tn * GS_T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp >> 2) * 32, wn = (warp & 3) * 16;
  const int row = tid & 63, kg = tid >> 6;                // this thread's row (column) and 16 values of k
  unsigned char* const sA = gs_smem;
  unsigned char* const sB = gs_smem + GS_OP_BYTES;
  unsigned short* const list = reinterpret_cast<unsigned short*>(gs_smem + 2 * GS_OP_BYTES);
  const uint32_t aA = (uint32_t)__cvta_generic_to_shared(sA) + (wm + (lane & 7) + ((lane >> 3) & 1) * 8) * GS_PITCH +
                      (lane >> 4) * 16;
  const uint32_t aB = (uint32_t)__cvta_generic_to_shared(sB) + (wn + (lane & 7) + ((lane >> 4) & 1) * 8) * GS_PITCH +
                      ((lane >> 3) & 1) * 16;
  // output z = a 8 + b 4 + c of this thread: row out_row(z), column out_col(z) of the tile
  auto out_row = [&](int z) { return wm + (z >> 3) * 16 + (lane >> 2) + ((z & 3) >> 1) * 8; };
  auto out_col = [&](int z) { return wn + ((z >> 2) & 1) * 8 + (lane & 3) * 2 + (z & 1); };
  // 16 values of k of this thread's row of op(A) and column of op(B), from l0 + kg 16 on
  auto load = [&](const GemmTerm<double>& tm, int l0, double (&xa)[16], double (&xb)[16]) {
    const int gi = i0 + row, gj = j0 + row, gl = l0 + kg * 16;
    const double* pa = tm.ta ? tm.A + gl + (size_t)gi * tm.lda : tm.A + gi + (size_t)gl * tm.lda;
    const double* pb = tm.tb ? tm.B + gj + (size_t)gl * tm.ldb : tm.B + gl + (size_t)gj * tm.ldb;
    const size_t da = tm.ta ? 1 : tm.lda, db = tm.tb ? tm.ldb : 1;
    const int ka = gi < tk.m ? tm.k - gl : 0, kb = gj < tk.n ? tm.k - gl : 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) xa[q] = q < ka ? pa[q * da] : 0.0;
#pragma unroll
    for (int q = 0; q < 16; ++q) xb[q] = q < kb ? pb[q * db] : 0.0;
  };
  double cd[16];
  int peak[16];                                           // log2 of the largest S so far, biased by 2046
#pragma unroll
  for (int z = 0; z < 16; ++z) {
    cd[z] = 0;
    peak[z] = -1;
  }
  for (int t = tk.t0; t < tk.t1; ++t) {
    const GemmTerm<double> tm = terms[t];
    const int klim = term_klim(tm, i0, j0, GS_T, GS_T);
    for (int l0 = 0; l0 < klim; l0 += GS_K) {
      // ---- load; largest exponents per value of k
      double xa[16], xb[16];
      load(tm, l0, xa, xb);
      bool odd = gs_k_exponents(xa, &s_k[0][warp & 1][kg * 16], lane);
      odd |= gs_k_exponents(xb, &s_k[1][warp & 1][kg * 16], lane);
      __syncthreads();
      // ---- the scale of each value of k; largest exponents of rows and columns
      int shift[16], ea = GS_NONE, eb = GS_NONE;
      bool some = odd;
#pragma unroll
      for (int q8 = 0; q8 < 16; q8 += 8) {
        const uint4 a0 = *reinterpret_cast<const uint4*>(&s_k[0][0][kg * 16 + q8]);
        const uint4 a1 = *reinterpret_cast<const uint4*>(&s_k[0][1][kg * 16 + q8]);
        const uint4 b0 = *reinterpret_cast<const uint4*>(&s_k[1][0][kg * 16 + q8]);
        const uint4 b1 = *reinterpret_cast<const uint4*>(&s_k[1][1][kg * 16 + q8]);
        const uint32_t ma[4] = {__vmaxu2(a0.x, a1.x), __vmaxu2(a0.y, a1.y), __vmaxu2(a0.z, a1.z), __vmaxu2(a0.w, a1.w)};
        const uint32_t mb[4] = {__vmaxu2(b0.x, b1.x), __vmaxu2(b0.y, b1.y), __vmaxu2(b0.z, b1.z), __vmaxu2(b0.w, b1.w)};
#pragma unroll
        for (int h = 0; h < 8; ++h) {
          const int q = q8 + h;
          const int ma_k = (int)(ma[h >> 1] >> (16 * (h & 1))) & 0xffff, mb_k = (int)(mb[h >> 1] >> (16 * (h & 1))) & 0xffff;
          shift[q] = (mb_k - ma_k) >> 1;
          if (ma_k == 0 || mb_k == 0) {                   // nothing comes of it
            shift[q] = 0;
            xa[q] = xb[q] = 0.0;
          } else {
            some = true;
          }
          const int e = gs_exponent(xa[q]), f = gs_exponent(xb[q]);
          if (e) ea = max(ea, e + shift[q]);
          if (f) eb = max(eb, f - shift[q]);
        }
      }
      s_part[0][kg][row] = (short)ea;
      s_part[1][kg][row] = (short)eb;
      if (!__syncthreads_or(some)) continue;
      ea = max(max(s_part[0][0][row], s_part[0][1][row]), max(s_part[0][2][row], s_part[0][3][row]));
      eb = max(max(s_part[1][0][row], s_part[1][1][row]), max(s_part[1][2][row], s_part[1][3][row]));
      odd |= (ea != GS_NONE && abs(ea - 1023) > 400) || (eb != GS_NONE && abs(eb - 1023) > 400);
      if (kg == 0) {
        s_e[0][row] = (short)ea;
        s_e[1][row] = (short)eb;
      }
      gs_digits(xa, shift, 1, ea, sA + row * GS_PITCH + kg * 32);
      gs_digits(xb, shift, -1, eb, sB + row * GS_PITCH + kg * 32);
      if (tid == 0) s_n = 0;
      uint32_t again = 0;                                 // outputs that take multiply-adds
      if (__syncthreads_or(odd)) {
        again = 0xffff;
      } else {
        // ---- 16 rows of the warp's 32 at a time
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          // acc[L] sums the digit products with s + t = L, acc[GS_S] those of |a| |b|
          float acc[GS_S + 1][2][4];
#pragma unroll
          for (int L = 0; L <= GS_S; ++L)
#pragma unroll
            for (int z = 0; z < 8; ++z) acc[L][z >> 2][z & 3] = 0.f;
#pragma unroll 1
          for (int kk = 0; kk < GS_K; kk += 16) {
            uint32_t fb[GS_S + 1][4];
#pragma unroll
            for (int s = 0; s <= GS_S; ++s) gs_ldmatrix4(fb[s], aB + s * GS_PLANE + kk * 2);
#pragma unroll
            for (int s = 0; s < GS_S; ++s) {
              uint32_t fa[4];
              gs_ldmatrix4(fa, aA + s * GS_PLANE + a * 16 * GS_PITCH + kk * 2);
#pragma unroll
              for (int u = 0; u + s < GS_S; ++u) {
                gs_mma(acc[s + u][0], fa, fb[u][0], fb[u][1]);
                gs_mma(acc[s + u][1], fa, fb[u][2], fb[u][3]);
              }
            }
            uint32_t fa[4];
            gs_ldmatrix4(fa, aA + GS_S * GS_PLANE + a * 16 * GS_PITCH + kk * 2);
            gs_mma(acc[GS_S][0], fa, fb[GS_S][0], fb[GS_S][1]);
            gs_mma(acc[GS_S][1], fa, fb[GS_S][2], fb[GS_S][3]);
          }
          // join: (sum_L acc[L] 256^(8 - L)) 256^8 units of the row times units of the
          // column, which are 2^(e - 1092)
#pragma unroll
          for (int y = 0; y < 8; ++y) {
            const int z = a * 8 + y, b = y >> 2, c = y & 3;
            const int er = s_e[0][out_row(z)], ej = s_e[1][out_col(z)];
            if (er == GS_NONE || ej == GS_NONE) continue;
            long long hi = 0, lo = 0;
#pragma unroll
            for (int L = 0; L < 5; ++L) hi = (hi << 8) + (long long)__float2int_rn(acc[L][b][c]);
#pragma unroll
            for (int L = 5; L < 9; ++L) lo = (lo << 8) + (long long)__float2int_rn(acc[L][b][c]);
            const double v = fma((double)hi, 4294967296.0, (double)lo);
            peak[z] = max(peak[z], er + ej + (int)(__float_as_uint(acc[GS_S][b][c]) >> 23) - 127);
            if (er + ej - peak[z] > GS_SPREAD) again |= 1u << z;
            else cd[z] = fma(v, __hiloint2double((er + ej - 2120 + 1023) << 20, 0), cd[z]);
          }
        }
      }
#pragma unroll
      for (int z = 0; z < 16; ++z) {
        const bool put = again >> z & 1;
        const unsigned m = __ballot_sync(0xffffffffu, put);
        if (m == 0) continue;
        int at = 0;
        if (lane == 0) at = atomicAdd(&s_n, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1));
        if (put) list[at] = (unsigned short)(out_row(z) * GS_T + out_col(z));
      }
      if (__syncthreads_or(again)) {
        // the chunk as it is over the digits, [k][row] and [k][column], and the sums
        double* const ra = reinterpret_cast<double*>(gs_smem);
        double* const rb = ra + GS_K * GS_RPITCH;
        double* const sum = rb + GS_K * GS_RPITCH;
        load(tm, l0, xa, xb);
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          ra[(kg * 16 + q) * GS_RPITCH + row] = xa[q];
          rb[(kg * 16 + q) * GS_RPITCH + row] = xb[q];
        }
        __syncthreads();
        for (int i = tid; i < s_n; i += 256) {
          const int ij = list[i];
          const double *pa = ra + ij / GS_T, *pb = rb + ij % GS_T;
          double s[4] = {0, 0, 0, 0};
#pragma unroll 4
          for (int l = 0; l < GS_K; l += 4)
#pragma unroll
            for (int h = 0; h < 4; ++h) s[h] = fma(pa[(l + h) * GS_RPITCH], pb[(l + h) * GS_RPITCH], s[h]);
          sum[ij] = (s[0] + s[1]) + (s[2] + s[3]);
        }
        __syncthreads();
#pragma unroll
        for (int z = 0; z < 16; ++z)
          if (again >> z & 1) cd[z] += sum[out_row(z) * GS_T + out_col(z)];
      }
    }
  }
  // epilogue: all loads of C before any store, so they overlap
  double cv[16];
#pragma unroll
  for (int z = 0; z < 16; ++z) {
    const int gi = i0 + out_row(z), gj = j0 + out_col(z);
    cv[z] = (tk.beta != 0.0 && gi < tk.m && gj < tk.n) ? tk.C[gi + (size_t)gj * tk.ldc] : 0.0;
  }
#pragma unroll
  for (int z = 0; z < 16; ++z) {
    const int gi = i0 + out_row(z), gj = j0 + out_col(z);
    if (gi < tk.m && gj < tk.n) tk.C[gi + (size_t)gj * tk.ldc] = tk.alpha * cd[z] + tk.beta * cv[z];
  }
}

}  // namespace spand
