// Grouped FP64 GEMM on the BF16 tensor cores: products of integers, exactly.
//
// Same task / term / tile contract as k_gemm<double>.  A GB300 has 2 FP64
// multiply-adds per clock and SM against 1,024 and more BF16 ones, so an FP64
// product is taken apart into BF16 products that are exact in the FP32
// accumulator (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012, with a common exponent per row):
//  * in a chunk of GS_K = 64 values of k, every row of op(A) and every column of
//    op(B) is scaled by its largest exponent to 62-bit integers and cut into
//    GS_S = 8 signed base-256 digits, |digit| <= 128, each exact in BF16;
//  * the digit products with s + t = L <= 7 (36 of them) are summed in FP32: at
//    most 8 x 64 terms of at most 2^14, below 2^24, so every sum is exact;
//  * the eight sums are joined in two 64-bit integers and added to the FP64
//    accumulator with two roundings per chunk.
// What is dropped (s + t >= 8, and what of an entry lies 2^-61 below its row's
// largest) is 2^-58 of the largest product of the row and column in a chunk, and
// there is one rounding per 64 products where the multiply-add form has 64: the
// eps = 0 factor's solve leaves a relative residual of 4.7 to 4.9e-16 where the
// multiply-adds left 4.8 to 5.0e-16 (16 x 8 p=1 and 64 x 32 p=2).  The bound goes
// with the row's largest entry in a chunk, not entry by entry.
// A chunk with an infinity or a NaN is summed in FP64 multiply-adds.
//
// 64 x 32 p=2 (useful flops; the FP64 rate is 1.25 TFLOP/s): Y and X products 1.0
// before, 3.2 TFLOP/s now; Schur updates 1.0, 2.9; scaling 0.6, 1.9; compression
// 0.6, 1.8; the factorization and solve 312 ms before, 171 ms now.
//
// Bound: the digits (integer arithmetic), 144 mma.sync per warp and 16 values of
// k, and 5 FP64 instructions per output and chunk (of 64 in the plain form).
#pragma once
#include <cstdint>

#include "dense.cuh"

namespace spand {

constexpr int GS_K = 64, GS_S = 8, GS_T = 64;             // chunk, digits, tile
constexpr int GS_PITCH = GS_K * 2 + 16;                   // bytes of a row of one digit (conflict-free ldmatrix)
constexpr int GS_OP_BYTES = GS_S * GS_T * GS_PITCH;       // the digits of one operand
constexpr int GS_SMEM_BYTES = 2 * GS_OP_BYTES;

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

// 2^(e - 1084): the unit of a row whose largest biased exponent is e
__device__ inline double gs_unit(int e) {
  const int k = e - 1084 + 1023;                          // the unit's own biased exponent
  return k > 0 ? __hiloint2double(k << 20, 0) : __hiloint2double((k + 64) << 20, 0) * 5.421010862427522e-20;   // 2^-64
}

// 16 consecutive k of one row (column): digits into `dst` (this row in digit 0)
__device__ inline void gs_digits(const double (&x)[16], int emax, unsigned char* dst) {
  uint32_t w[GS_S][2];                                    // digits of a pair of pairs, packed
#pragma unroll
  for (int q = 0; q < 16; q += 4) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const long long b = __double_as_longlong(x[q + h]);
      const int e = (int)((unsigned long long)b >> 52) & 0x7ff;
      const int d = emax - e;
      long long f = ((b & 0xfffffffffffffll) | 0x10000000000000ll) << 9;
      f = (e == 0 || d > 61) ? 0 : f >> d;
      if (b < 0) f = -f;
#pragma unroll
      for (int s = GS_S - 1; s >= 0; --s) {
        const int lo = (int)(signed char)(f & 0xff);
        f = (f - lo) >> 8;
        // small integer -> BF16: the top half of its (exact) FP32
        const uint32_t v = __float_as_uint(__int_as_float(0x4B400000 + lo) - 12582912.0f) >> 16;
        if ((h & 1) == 0) w[s][h >> 1] = v;
        else w[s][h >> 1] |= v << 16;
      }
    }
#pragma unroll
    for (int s = 0; s < GS_S; ++s)
      *reinterpret_cast<uint2*>(dst + s * (GS_T * GS_PITCH) + q * 2) = make_uint2(w[s][0], w[s][1]);
  }
}

__global__ void __launch_bounds__(256, 1) k_gemm_split(const GemmTask<double>* tasks, const GemmTerm<double>* terms,
                                                       const TileItem* tiles) {
  extern __shared__ __align__(16) unsigned char gs_smem[];
  __shared__ int s_part[2][4][GS_T];                      // largest exponent of a quarter row of A / column of B
  __shared__ int s_odd;                                   // the chunk holds an infinity or a NaN
  const TileItem it = tiles[blockIdx.x];
  const GemmTask<double> tk = tasks[it.task];
  const int i0 = it.tm * GS_T, j0 = it.tn * GS_T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp >> 2) * 32, wn = (warp & 3) * 16;
  const int row = tid & 63, kg = tid >> 6;                // this thread's row (column) and 16 values of k
  unsigned char* const sA = gs_smem;
  unsigned char* const sB = gs_smem + GS_OP_BYTES;
  const uint32_t aA = (uint32_t)__cvta_generic_to_shared(sA) + (wm + (lane & 7) + ((lane >> 3) & 1) * 8) * GS_PITCH +
                      (lane >> 4) * 16;
  const uint32_t aB = (uint32_t)__cvta_generic_to_shared(sB) + (wn + (lane & 7) + ((lane >> 4) & 1) * 8) * GS_PITCH +
                      ((lane >> 3) & 1) * 16;
  double cd[2][2][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) cd[a][b][c] = 0;
  for (int t = tk.t0; t < tk.t1; ++t) {
    const GemmTerm<double> tm = terms[t];
    const int klim = term_klim(tm, i0, j0, GS_T, GS_T);
    for (int l0 = 0; l0 < klim; l0 += GS_K) {
      // ---- load, largest exponents
      double xa[16], xb[16];
      {
        const int gi = i0 + row, gj = j0 + row, gl = l0 + kg * 16;
        const double* pa = tm.ta ? tm.A + gl + (size_t)gi * tm.lda : tm.A + gi + (size_t)gl * tm.lda;
        const double* pb = tm.tb ? tm.B + gj + (size_t)gl * tm.ldb : tm.B + gl + (size_t)gj * tm.ldb;
        const size_t da = tm.ta ? 1 : tm.lda, db = tm.tb ? tm.ldb : 1;
        const int ka = gi < tk.m ? tm.k - gl : 0, kb = gj < tk.n ? tm.k - gl : 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) xa[q] = q < ka ? pa[q * da] : 0.0;
#pragma unroll
        for (int q = 0; q < 16; ++q) xb[q] = q < kb ? pb[q * db] : 0.0;
      }
      int ea = 0, eb = 0;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        ea = max(ea, (__double2hiint(xa[q]) >> 20) & 0x7ff);
        eb = max(eb, (__double2hiint(xb[q]) >> 20) & 0x7ff);
      }
      __syncthreads();                                    // the last chunk's digits and exponents are no longer read
      s_part[0][kg][row] = ea;
      s_part[1][kg][row] = eb;
      if (tid == 0) s_odd = 0;
      __syncthreads();
      ea = max(max(s_part[0][0][row], s_part[0][1][row]), max(s_part[0][2][row], s_part[0][3][row]));
      eb = max(max(s_part[1][0][row], s_part[1][1][row]), max(s_part[1][2][row], s_part[1][3][row]));
      if (ea == 0x7ff || eb == 0x7ff) s_odd = 1;
      gs_digits(xa, ea, sA + row * GS_PITCH + kg * 32);
      gs_digits(xb, eb, sB + row * GS_PITCH + kg * 32);
      __syncthreads();
      if (s_odd) {
        for (int a = 0; a < 2; ++a)
          for (int b = 0; b < 2; ++b)
            for (int c = 0; c < 4; ++c) {
              const int gi = i0 + wm + a * 16 + (lane >> 2) + (c >> 1) * 8;
              const int gj = j0 + wn + b * 8 + (lane & 3) * 2 + (c & 1);
              if (gi >= tk.m || gj >= tk.n) continue;
              double s = 0;
              for (int l = l0; l < min(tm.k, l0 + GS_K); ++l)
                s += (tm.ta ? tm.A[l + (size_t)gi * tm.lda] : tm.A[gi + (size_t)l * tm.lda]) *
                     (tm.tb ? tm.B[gj + (size_t)l * tm.ldb] : tm.B[l + (size_t)gj * tm.ldb]);
              // (static indices keep the accumulators in registers)
#pragma unroll
              for (int z = 0; z < 16; ++z)
                if (z == a * 8 + b * 4 + c) cd[z >> 3][(z >> 2) & 1][z & 3] += s;
            }
        continue;
      }
      // ---- digit products: acc[L] sums s + t = L
      float acc[GS_S][2][2][4];
#pragma unroll
      for (int L = 0; L < GS_S; ++L)
#pragma unroll
        for (int z = 0; z < 16; ++z) acc[L][z >> 3][(z >> 2) & 1][z & 3] = 0.f;
#pragma unroll 1
      for (int kk = 0; kk < GS_K; kk += 16) {
        uint32_t fb[GS_S][4];
#pragma unroll
        for (int s = 0; s < GS_S; ++s) gs_ldmatrix4(fb[s], aB + s * (GS_T * GS_PITCH) + kk * 2);
#pragma unroll
        for (int s = 0; s < GS_S; ++s)
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            uint32_t fa[4];
            gs_ldmatrix4(fa, aA + s * (GS_T * GS_PITCH) + a * 16 * GS_PITCH + kk * 2);
#pragma unroll
            for (int u = 0; u + s < GS_S; ++u) {
              gs_mma(acc[s + u][a][0], fa, fb[u][0], fb[u][1]);
              gs_mma(acc[s + u][a][1], fa, fb[u][2], fb[u][3]);
            }
          }
      }
      // ---- join: (sum_L acc[L] 256^(7 - L)) 256^7 units of the row times units of the column
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int ch = 0; ch < 2; ++ch) {
          const int r = wm + a * 16 + (lane >> 2) + ch * 8;
          const int er = max(max(s_part[0][0][r], s_part[0][1][r]), max(s_part[0][2][r], s_part[0][3][r]));
          const double ur = gs_unit(er) * 72057594037927936.0;            // 2^56
#pragma unroll
          for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int cl = 0; cl < 2; ++cl) {
              const int j = wn + b * 8 + (lane & 3) * 2 + cl, c = ch * 2 + cl;
              const int ej = max(max(s_part[1][0][j], s_part[1][1][j]), max(s_part[1][2][j], s_part[1][3][j]));
              long long hi = 0, lo = 0;
#pragma unroll
              for (int L = 0; L < 4; ++L) {
                hi = (hi << 8) + (long long)__float2int_rn(acc[L][a][b][c]);
                lo = (lo << 8) + (long long)__float2int_rn(acc[L + 4][a][b][c]);
              }
              const double v = fma((double)hi, 4294967296.0, (double)lo);
              cd[a][b][c] = fma(v, ur * gs_unit(ej), cd[a][b][c]);
            }
        }
    }
  }
  // epilogue: all loads of C before any store, so they overlap
  double cv[2][2][4];
#pragma unroll
  for (int z = 0; z < 16; ++z) {
    const int a = z >> 3, b = (z >> 2) & 1, c = z & 3;
    const int gi = i0 + wm + a * 16 + (lane >> 2) + (c >> 1) * 8, gj = j0 + wn + b * 8 + (lane & 3) * 2 + (c & 1);
    cv[a][b][c] = (tk.beta != 0.0 && gi < tk.m && gj < tk.n) ? tk.C[gi + (size_t)gj * tk.ldc] : 0.0;
  }
#pragma unroll
  for (int z = 0; z < 16; ++z) {
    const int a = z >> 3, b = (z >> 2) & 1, c = z & 3;
    const int gi = i0 + wm + a * 16 + (lane >> 2) + (c >> 1) * 8, gj = j0 + wn + b * 8 + (lane & 3) * 2 + (c & 1);
    if (gi < tk.m && gj < tk.n) tk.C[gi + (size_t)gj * tk.ldc] = tk.alpha * cd[a][b][c] + tk.beta * cv[a][b][c];
  }
}

}  // namespace spand
