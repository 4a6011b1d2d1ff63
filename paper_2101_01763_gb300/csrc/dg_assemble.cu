// DG residual and Jacobian assembly for 2D Euler (Sec. 2.1.2, Eqs. 3-8).
//
// One CTA per element computes its whole block row: the volume term of Eq. 7
// and its exact derivative, the surface terms of its four faces (Rusanov flux
// evaluated in the face's global L->R orientation, so both neighbours see the
// same flux and the same branch of the max), the mass term M/dtau (Eq. 6) and
// the residual entries.  Each face is evaluated by both adjacent elements;
// no scratch, no atomics, deterministic.  A first pass computes the CFL time
// step of Eq. 8.
//
// Bound: FP64 arithmetic (2 multiply-adds per clock and SM against 5 B^2
// doubles written per element).  The basis is a tensor product, so the Jacobian's
// sums over the quadrature points are taken one direction at a time: over xi
// first (for every eta and every pair of xi degrees), then over eta; a face
// needs one such sum, since the basis is constant across it up to a factor per
// degree.  At p = 3 that is 1.0e5 multiply-adds per element instead of 3.7e5
// (256 x 128 p=3: 47.8 ms with the direct sums, 11.8 ms now, 5.2 ms of it
// multiply-adds and 0.8 ms stores).
//
// Gauss-Legendre nodes (Newton iteration on P_q) and the
// orthonormal Legendre basis (three-term recurrence) are tabulated once on the
// host for the reference element and passed to the kernels by value.
#include <cmath>
#include <cstdint>
#include <cstring>

#include "internal.h"

namespace {

constexpr int PMAX = 3;
constexpr int QMAX = PMAX + 2;            // points per direction
constexpr int NPMAX = (PMAX + 1) * (PMAX + 1);
constexpr int VQMAX = QMAX * QMAX;

struct Flow {
  double gamma, uinf[4], cfl;
  int bc_wall;
};

// Reference-element tables, built once on the host and passed by value:
// Gauss-Legendre rule, 1D basis values / derivatives, basis values at the q x q
// volume points (xi fastest).
struct Tables {
  int q, np, Q;
  double tq[QMAX], wq[QMAX];
  double V[QMAX][PMAX + 1], D[QMAX][PMAX + 1];    // 1D values / derivatives at the points
  double Vend[2][PMAX + 1];                       // 1D values at +1 and -1
  double psi[VQMAX][NPMAX];                       // basis at the q x q volume points (xi fastest)
};

// orthonormal Legendre values / derivatives of degree 0..p at t
__host__ __device__ void legendre(int p, double t, double* V, double* D) {
  double P0 = 1.0, P1 = t, dP0 = 0.0, dP1 = 1.0;
  double P[PMAX + 1], dP[PMAX + 1];
  P[0] = P0;
  dP[0] = dP0;
  if (p >= 1) {
    P[1] = P1;
    dP[1] = dP1;
  }
  for (int a = 1; a < p; ++a) {
    P[a + 1] = ((2 * a + 1) * t * P[a] - a * P[a - 1]) / (a + 1);
    dP[a + 1] = (a + 1) * P[a] + t * dP[a];
  }
  for (int a = 0; a <= p; ++a) {
    double s = sqrt((2 * a + 1) * 0.5);
    V[a] = s * P[a];
    D[a] = s * dP[a];
  }
}

// Gauss-Legendre rule with q points on [-1, 1], ascending nodes
__host__ __device__ void gauss_rule(int q, double* t, double* w) {
  for (int i = 0; i < q; ++i) {
    double x = cos(M_PI * (i + 0.75) / (q + 0.5));
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = x;
      for (int k = 1; k < q; ++k) {
        double p2 = ((2 * k + 1) * x * p1 - k * p0) / (k + 1);
        p0 = p1;
        p1 = p2;
      }
      dp = q * (x * p1 - p0) / (x * x - 1.0);
      double dx = p1 / dp;
      x -= dx;
      if (fabs(dx) < 1e-16) break;
    }
    {
      double p0 = 1.0, p1 = x;
      for (int k = 1; k < q; ++k) {
        double p2 = ((2 * k + 1) * x * p1 - k * p0) / (k + 1);
        p0 = p1;
        p1 = p2;
      }
      dp = q * (x * p1 - p0) / (x * x - 1.0);
    }
    t[q - 1 - i] = x;
    w[q - 1 - i] = 2.0 / ((1.0 - x * x) * dp * dp);
  }
}

__host__ __device__ bool primitive(const double* U, double g, double& rho, double& ux, double& uy, double& p) {
  rho = U[0];
  ux = U[1] / rho;
  uy = U[2] / rho;
  p = (g - 1.0) * (U[3] - 0.5 * rho * (ux * ux + uy * uy));
  return rho > 0.0 && p > 0.0 && isfinite(p);
}

// F.n and d(F.n)/dU (row-major 4x4)
__host__ __device__ void flux_n(const double* U, double nx, double ny, double g, double* F, double* A) {
  double rho, ux, uy, p;
  primitive(U, g, rho, ux, uy, p);
  const double E = U[3], g1 = g - 1.0;
  const double vn = ux * nx + uy * ny;
  F[0] = rho * vn;
  F[1] = U[1] * vn + p * nx;
  F[2] = U[2] * vn + p * ny;
  F[3] = (E + p) * vn;
  if (!A) return;
  const double phi = 0.5 * g1 * (ux * ux + uy * uy), H = (E + p) / rho;
  A[0] = 0.0; A[1] = nx; A[2] = ny; A[3] = 0.0;
  A[4] = phi * nx - ux * vn; A[5] = vn + ux * nx - g1 * ux * nx; A[6] = ux * ny - g1 * uy * nx; A[7] = g1 * nx;
  A[8] = phi * ny - uy * vn; A[9] = uy * nx - g1 * ux * ny; A[10] = vn + uy * ny - g1 * uy * ny; A[11] = g1 * ny;
  A[12] = vn * (phi - H); A[13] = H * nx - g1 * ux * vn; A[14] = H * ny - g1 * uy * vn; A[15] = g * vn;
}

// a = |v.n| + c and da/dU
__host__ __device__ double wave(const double* U, double nx, double ny, double g, double* da) {
  double rho, ux, uy, p;
  primitive(U, g, rho, ux, uy, p);
  const double c = sqrt(g * p / rho), vn = ux * nx + uy * ny, g1 = g - 1.0;
  const double sg = vn >= 0.0 ? 1.0 : -1.0;
  const double k = g / (2.0 * c * rho);
  da[0] = sg * (-vn / rho) + k * 0.5 * g1 * (ux * ux + uy * uy) - c / (2.0 * rho);
  da[1] = sg * (nx / rho) - k * g1 * ux;
  da[2] = sg * (ny / rho) - k * g1 * uy;
  da[3] = k * g1;
  return fabs(vn) + c;
}

// Rusanov F*.n with dF/dUL, dF/dUR (row-major 4x4); L branch of the max on ties
__host__ __device__ void rusanov(const double* UL, const double* UR, double nx, double ny, double g,
                        double* F, double* dL, double* dR) {
  double FL[4], FR[4], AL[16], AR[16], daL[4], daR[4];
  flux_n(UL, nx, ny, g, FL, AL);
  flux_n(UR, nx, ny, g, FR, AR);
  double aL = wave(UL, nx, ny, g, daL), aR = wave(UR, nx, ny, g, daR);
  const bool takeL = aL >= aR;
  const double lam = takeL ? aL : aR;
  double dU[4];
  for (int v = 0; v < 4; ++v) {
    dU[v] = UR[v] - UL[v];
    F[v] = 0.5 * (FL[v] + FR[v]) - 0.5 * lam * dU[v];
  }
  for (int v = 0; v < 4; ++v)
    for (int w = 0; w < 4; ++w) {
      double id = (v == w) ? 1.0 : 0.0;
      dL[v * 4 + w] = 0.5 * AL[v * 4 + w] + 0.5 * lam * id - 0.5 * dU[v] * (takeL ? daL[w] : 0.0);
      dR[v * 4 + w] = 0.5 * AR[v * 4 + w] - 0.5 * lam * id - 0.5 * dU[v] * (takeL ? 0.0 : daR[w]);
    }
}

__host__ __device__ void corners(const double* X, int n_theta, int i, int j, double C[4][2]) {
  const int jp = (j + 1) % n_theta;
  const int idx[4] = {i * n_theta + j, i * n_theta + jp, (i + 1) * n_theta + jp, (i + 1) * n_theta + j};
  for (int c = 0; c < 4; ++c) {
    C[c][0] = X[2 * idx[c]];
    C[c][1] = X[2 * idx[c] + 1];
  }
}

__host__ __device__ void jac_map(const double C[4][2], double xi, double eta, double* dxi, double* deta) {
  for (int d = 0; d < 2; ++d) {
    dxi[d] = 0.25 * (-(1 - eta) * C[0][d] + (1 - eta) * C[1][d] + (1 + eta) * C[2][d] - (1 + eta) * C[3][d]);
    deta[d] = 0.25 * (-(1 - xi) * C[0][d] - (1 + xi) * C[1][d] + (1 + xi) * C[2][d] + (1 - xi) * C[3][d]);
  }
}

__device__ inline void atomic_min_pos(double* addr, double v) {
  // non-negative doubles order like their bit patterns
  atomicMin(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

// ------------------------------------------------------------------ time step
__global__ void k_time_step(const double* X, int n_theta, int n_r, int p, const double* uh, Flow fl,
                            double* dtau, int* bad, const __grid_constant__ Tables T) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_theta * n_r) return;
  const int q = T.q, np = T.np;
  const int i = e / n_theta, j = e % n_theta;
  double C[4][2];
  corners(X, n_theta, i, j, C);
  double area = 0.0, smax = 0.0;
  for (int b = 0; b < q; ++b)
    for (int a = 0; a < q; ++a) {
      double dxi[2], deta[2];
      jac_map(C, T.tq[a], T.tq[b], dxi, deta);
      area += T.wq[a] * T.wq[b] * (dxi[0] * deta[1] - deta[0] * dxi[1]);
      const int pt = b * q + a;
      double U[4] = {0, 0, 0, 0};
      for (int m = 0; m < np; ++m)
        for (int v = 0; v < 4; ++v) U[v] += T.psi[pt][m] * uh[(size_t)e * np * 4 + m * 4 + v];
      double rho, ux, uy, pr;
      if (!primitive(U, fl.gamma, rho, ux, uy, pr)) atomicExch(bad, 1);
      smax = fmax(smax, sqrt(ux * ux + uy * uy) + sqrt(fl.gamma * pr / rho));
    }
  double perim = 0.0;
  for (int c = 0; c < 4; ++c) {
    double dx = C[(c + 1) % 4][0] - C[c][0], dy = C[(c + 1) % 4][1] - C[c][1];
    perim += sqrt(dx * dx + dy * dy);
  }
  const double lam = smax * (2 * p + 1) * perim / area;
  double v = fl.cfl / lam;
  if (!(v > 0.0) || !isfinite(v)) {
    atomicExch(bad, 1);
    return;
  }
  atomic_min_pos(dtau, v);
}

// ------------------------------------------------------------------ pattern
// first block of row e: each element with its face neighbours (periodic in
// theta, open in r), columns ascending
__host__ __device__ inline int row_start(int e, int n_theta, int n_r) {
  if (n_r == 1) return 3 * e;
  const int i = e / n_theta;
  if (i == 0) return 4 * e;
  if (i < n_r - 1) return 4 * n_theta + 5 * (e - n_theta);
  return 4 * n_theta + 5 * n_theta * (n_r - 2) + 4 * (e - (n_r - 1) * n_theta);
}

// the row's columns in local order (self, east, west, north, south; -1: none)
// and the place of each among the ascending ones
__device__ inline int row_columns(int e, int n_theta, int n_r, int cols[5], int rank[5]) {
  const int i = e / n_theta, j = e % n_theta;
  cols[0] = e;
  cols[1] = i * n_theta + (j + 1) % n_theta;
  cols[2] = i * n_theta + (j + n_theta - 1) % n_theta;
  cols[3] = (i < n_r - 1) ? e + n_theta : -1;
  cols[4] = (i > 0) ? e - n_theta : -1;
  int n = 0;
  for (int a = 0; a < 5; ++a) {
    rank[a] = -1;
    if (cols[a] < 0) continue;
    ++n;
    int r = 0;
    for (int b = 0; b < 5; ++b)
      if (cols[b] >= 0 && cols[b] < cols[a]) ++r;
    rank[a] = r;
  }
  return n;
}

__global__ void k_pattern(int n_theta, int n_r, int* row_ptr, int* col) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x, K = n_theta * n_r;
  if (e >= K) return;
  int cols[5], rank[5];
  const int n = row_columns(e, n_theta, n_r, cols, rank), rp = row_start(e, n_theta, n_r);
  row_ptr[e] = rp;
  if (e == K - 1) row_ptr[K] = rp + n;
  for (int a = 0; a < 5; ++a)
    if (cols[a] >= 0) col[rp + rank[a]] = cols[a];
}

// ------------------------------------------------------------------ assembly
template <int P>
struct Smem {
  static constexpr int NA = P + 1, NP = NA * NA, Q1 = P + 2, Q = Q1 * Q1;
  double uh[5][NP][4];                      // self + 4 neighbours
  double gx[Q][NP], gy[Q][NP];
  double wdet[Q];
  double Fx[Q][4], Fy[Q][4];
  double A1[Q][16], A2[Q][16];              // flux Jacobians along xi and eta, with weight and metric
  double hws[4][Q1];                        // signed half-length x weight
  double Fs[4][Q1][4], dFs[4][Q1][16], dFn[4][Q1][16];
  double V[Q1][NA], D[Q1][NA], Vend[2][NA];
  // sums over xi, for every eta point and pair of xi degrees (test, trial)
  double T1[Q1][NA * NA][16], T2[Q1][NA * NA][16], Tm[Q1][NA * NA];
  // sums along a face, for every pair of running degrees: own and neighbour's trial
  double Ks[4][NA * NA][16], Kn[4][NA * NA][16];
  int nb[4];                                // neighbour element per local face or -1
  int rank[5];                              // BSR position of self / faces
};

template <int P>
__host__ __device__ constexpr int assemble_threads() { return P == 3 ? 256 : P == 2 ? 96 : 64; }

// vw = 0 and 3 (mass flux against density and energy) are zero in every Euler flux Jacobian
__device__ constexpr bool flux_zero(int vw) { return vw == 0 || vw == 3; }

template <int P>
__global__ void __launch_bounds__(assemble_threads<P>(), P == 3 ? 3 : 6) k_assemble(const double* X, int n_theta, int n_r,
                                                                    const double* uh, Flow fl, const double* dtau_p,
                                                                    double* rhs, double* val, int* bad, int vec,
                                                                    const __grid_constant__ Tables T) {
  extern __shared__ double smem_raw[];
  typedef Smem<P> SM;
  SM& S = *reinterpret_cast<SM*>(smem_raw);
  constexpr int NA = SM::NA, NP = SM::NP, q = SM::Q1, Q = SM::Q, B = 4 * NP, NT = assemble_threads<P>();
  const int e = blockIdx.x;
  const int i = e / n_theta, j = e % n_theta;
  const int tid = threadIdx.x;
  const double g = fl.gamma;
  // mode m at point k of local face f
  auto face_psi = [&](int f, int k, int m) {
    const int a = m % NA, b = m / NA;
    return f < 2 ? S.Vend[f & 1][a] * S.V[k][b] : S.V[k][a] * S.Vend[f & 1][b];
  };
  if (tid < q * NA) {
    S.V[tid / NA][tid % NA] = T.V[tid / NA][tid % NA];
    S.D[tid / NA][tid % NA] = T.D[tid / NA][tid % NA];
  }
  if (tid < 2 * NA) S.Vend[tid / NA][tid % NA] = T.Vend[tid / NA][tid % NA];
  if (tid == 0) {
    int cols[5];
    row_columns(e, n_theta, n_r, cols, S.rank);
    // east, north: self is L (outer boundary if -1); west, south: self is R (airfoil if -1)
    for (int f = 0; f < 4; ++f) S.nb[f] = cols[f + 1];
  }
  __syncthreads();
  for (int t = tid; t < 5 * NP * 4; t += NT) {
    int s = t / (NP * 4), r = t % (NP * 4);
    int el = (s == 0) ? e : S.nb[s - 1];
    S.uh[s][r / 4][r % 4] = (el >= 0) ? uh[(size_t)el * NP * 4 + r] : 0.0;
  }
  __syncthreads();
  if (tid < Q) {
    // ---- volume point
    double C[4][2];
    corners(X, n_theta, i, j, C);
    const int a = tid % q, b = tid / q;
    const double xi = T.tq[a], eta = T.tq[b], w = T.wq[a] * T.wq[b];
    double dxi[2], deta[2];
    jac_map(C, xi, eta, dxi, deta);
    const double det = dxi[0] * deta[1] - deta[0] * dxi[1];
    double U[4] = {0, 0, 0, 0};
    for (int m = 0; m < NP; ++m) {
      const double ps = S.V[a][m % NA] * S.V[b][m / NA];
      const double px = S.D[a][m % NA] * S.V[b][m / NA], pe = S.V[a][m % NA] * S.D[b][m / NA];
      S.gx[tid][m] = w * (deta[1] * px - dxi[1] * pe);
      S.gy[tid][m] = w * (-deta[0] * px + dxi[0] * pe);
      for (int v = 0; v < 4; ++v) U[v] += ps * S.uh[0][m][v];
    }
    S.wdet[tid] = w * det;
    double rho, ux, uy, pr;
    if (!primitive(U, g, rho, ux, uy, pr)) atomicExch(bad, 1);
    double Ax[16], Ay[16];
    flux_n(U, 1.0, 0.0, g, S.Fx[tid], Ax);
    flux_n(U, 0.0, 1.0, g, S.Fy[tid], Ay);
    for (int vw = 0; vw < 16; ++vw) {
      S.A1[tid][vw] = w * (deta[1] * Ax[vw] - deta[0] * Ay[vw]);
      S.A2[tid][vw] = w * (dxi[0] * Ay[vw] - dxi[1] * Ax[vw]);
    }
  } else if (tid >= 32 && tid < 32 + 4 * q) {
    // ---- face point: local face f, point k
    const int f = (tid - 32) / q, k = (tid - 32) % q;
    int node_a, node_b;                                   // edge end points (node ids)
    const int jp = (j + 1) % n_theta;
    bool self_is_L;
    int nf;                                               // neighbour's local face
    double nx, ny;
    if (f == 0) { node_a = i * n_theta + jp; node_b = (i + 1) * n_theta + jp; self_is_L = true; nf = 1; }
    else if (f == 1) { node_a = i * n_theta + j; node_b = (i + 1) * n_theta + j; self_is_L = false; nf = 0; }
    else if (f == 2) { node_a = (i + 1) * n_theta + j; node_b = (i + 1) * n_theta + jp; self_is_L = true; nf = 3; }
    else { node_a = i * n_theta + j; node_b = i * n_theta + jp; self_is_L = false; nf = 2; }
    const double tx = X[2 * node_b] - X[2 * node_a], ty = X[2 * node_b + 1] - X[2 * node_a + 1];
    const double len = sqrt(tx * tx + ty * ty);
    // global L->R normal: east/west faces use the L element's east edge, north/south its north edge
    if (f <= 1) { nx = ty / len; ny = -tx / len; }
    else { nx = -ty / len; ny = tx / len; }
    const int nbe = S.nb[f];
    const bool boundary = nbe < 0;
    if (boundary && f == 3) {            // airfoil: the element is L with outward normal
      nx = -nx; ny = -ny; self_is_L = true;
    }
    double Us[4] = {0, 0, 0, 0}, Un[4] = {0, 0, 0, 0};
    for (int m = 0; m < NP; ++m) {
      const double ps = face_psi(f, k, m), pn = face_psi(nf, k, m);
      for (int v = 0; v < 4; ++v) {
        Us[v] += ps * S.uh[0][m][v];
        if (!boundary) Un[v] += pn * S.uh[f + 1][m][v];
      }
    }
    double W[16];
    bool wall = false;
    if (boundary) {
      wall = (f == 3) && fl.bc_wall;
      if (wall) {
        for (int a = 0; a < 16; ++a) W[a] = 0.0;
        W[0] = 1.0; W[15] = 1.0;
        W[5] = 1.0 - 2.0 * nx * nx; W[6] = -2.0 * nx * ny;
        W[9] = -2.0 * nx * ny; W[10] = 1.0 - 2.0 * ny * ny;
        for (int v = 0; v < 4; ++v) {
          Un[v] = 0.0;
          for (int w2 = 0; w2 < 4; ++w2) Un[v] += W[v * 4 + w2] * Us[w2];
        }
      } else {
        for (int v = 0; v < 4; ++v) Un[v] = fl.uinf[v];
      }
    }
    double F[4], dL[16], dR[16];
    const double* UL = self_is_L ? Us : Un;
    const double* UR = self_is_L ? Un : Us;
    {
      double r0, a0, b0, c0;
      if (!primitive(Us, g, r0, a0, b0, c0) || !primitive(Un, g, r0, a0, b0, c0)) atomicExch(bad, 1);
    }
    rusanov(UL, UR, nx, ny, g, F, dL, dR);
    const double sgn = self_is_L ? 1.0 : -1.0;
    const double hw = sgn * 0.5 * len * T.wq[k];
    S.hws[f][k] = hw;
    for (int v = 0; v < 4; ++v) S.Fs[f][k][v] = F[v];
    const double* dSelf = self_is_L ? dL : dR;
    const double* dNb = self_is_L ? dR : dL;
    for (int a = 0; a < 16; ++a) {
      double ds = dSelf[a];
      if (wall) {                                          // chain rule through the ghost state
        const int v = a / 4, w2 = a % 4;
        for (int u = 0; u < 4; ++u) ds += dR[v * 4 + u] * W[u * 4 + w2];
      }
      S.dFs[f][k][a] = hw * ds;
      S.dFn[f][k][a] = boundary ? 0.0 : hw * dNb[a];
    }
  }
  __syncthreads();
  // ---- residual
  for (int t = tid; t < NP * 4; t += NT) {
    const int m = t / 4, v = t % 4;
    double r = 0.0;
    for (int a = 0; a < Q; ++a) r -= S.gx[a][m] * S.Fx[a][v] + S.gy[a][m] * S.Fy[a][v];
    for (int f = 0; f < 4; ++f)
      for (int k = 0; k < q; ++k) r += S.hws[f][k] * face_psi(f, k, m) * S.Fs[f][k][v];
    rhs[(size_t)e * B + t] = -r;
  }
  // ---- sums over xi and along the faces
  for (int t = tid; t < q * NA * NA * 16; t += NT) {
    const int vw = t % 16, aa = t / 16 % (NA * NA), y = t / 16 / (NA * NA), ai = aa / NA, aj = aa % NA;
    double s1 = 0.0, s2 = 0.0;
    if (!flux_zero(vw)) {
#pragma unroll
      for (int x = 0; x < q; ++x) {
        const double vj = S.V[x][aj];
        s1 += S.D[x][ai] * vj * S.A1[y * q + x][vw];
        s2 += S.V[x][ai] * vj * S.A2[y * q + x][vw];
      }
    }
    S.T1[y][aa][vw] = s1;
    S.T2[y][aa][vw] = s2;
    if (vw == 0) {
      double sm = 0.0;
#pragma unroll
      for (int x = 0; x < q; ++x) sm += S.V[x][ai] * S.V[x][aj] * S.wdet[y * q + x];
      S.Tm[y][aa] = sm;
    }
  }
  for (int t = tid; t < 4 * NA * NA * 16; t += NT) {
    const int vw = t % 16, rr = t / 16 % (NA * NA), f = t / 16 / (NA * NA), ri = rr / NA, rj = rr % NA;
    double s1 = 0.0, s2 = 0.0;
#pragma unroll
    for (int k = 0; k < q; ++k) {
      const double vv = S.V[k][ri] * S.V[k][rj];
      s1 += vv * S.dFs[f][k][vw];
      s2 += vv * S.dFn[f][k][vw];
    }
    S.Ks[f][rr][vw] = s1;
    S.Kn[f][rr][vw] = s2;
  }
  __syncthreads();
  // ---- Jacobian blocks: a thread per (row mode mi, column mode mj); the row mode
  // runs over the lanes, so that a warp writes contiguous rows of a block column
  const double inv_dt = 1.0 / *dtau_p;
  const size_t bb = (size_t)B * B;
  double* const row = val + (size_t)row_start(e, n_theta, n_r) * bb;
  for (int t = tid; t < NP * NP; t += NT) {
    const int mi = t % NP, mj = t / NP, ai = mi % NA, bi = mi / NA, aj = mj % NA, bj = mj / NA;
    const int aa = ai * NA + aj, bbx = bi * NA + bj;
    double J[16];
#pragma unroll
    for (int vw = 0; vw < 16; ++vw) J[vw] = 0.0;
    double mass = 0.0;
#pragma unroll
    for (int y = 0; y < q; ++y) {
      const double vj = S.V[y][bj], c1 = S.V[y][bi] * vj, c2 = S.D[y][bi] * vj;
#pragma unroll
      for (int vw = 0; vw < 16; ++vw)
        if (!flux_zero(vw)) J[vw] -= c1 * S.T1[y][aa][vw] + c2 * S.T2[y][aa][vw];
      mass += c1 * S.Tm[y][aa];
    }
    // face f: the fixed degrees give factors, the running ones index the face sums
    auto put = [&](int rank, const double (&M)[16]) {
      double* blk = row + rank * bb + (size_t)mj * 4 * B + mi * 4;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        if (vec) {
          *reinterpret_cast<double2*>(blk + w * B) = make_double2(M[w], M[4 + w]);
          *reinterpret_cast<double2*>(blk + w * B + 2) = make_double2(M[8 + w], M[12 + w]);
        } else {
          for (int v = 0; v < 4; ++v) blk[w * B + v] = M[4 * v + w];
        }
      }
    };
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int s = f & 1, fi = f < 2 ? ai : bi, fj = f < 2 ? aj : bj, rr = f < 2 ? bbx : aa;
      const double ci = S.Vend[s][fi], cs = ci * S.Vend[s][fj], cn = ci * S.Vend[s ^ 1][fj];
#pragma unroll
      for (int vw = 0; vw < 16; ++vw) J[vw] += cs * S.Ks[f][rr][vw];
      if (S.nb[f] >= 0) {
        double M[16];
#pragma unroll
        for (int vw = 0; vw < 16; ++vw) M[vw] = cn * S.Kn[f][rr][vw];
        put(S.rank[f + 1], M);
      }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) J[v * 4 + v] += mass * inv_dt;
    put(S.rank[0], J);
  }
}

template <int P>
int launch_assemble(int K, const double* X, int nt, int nr, const double* uh, const Flow& fl, const double* dtau,
                    double* rhs, double* val, int* bad, const Tables& T, cudaStream_t st) {
  const size_t smem = sizeof(Smem<P>);
  if (spand::set_dyn_smem((const void*)k_assemble<P>, smem) < (long long)smem) return SPAND_ERR_UNSUPPORTED;
  const int vec = (reinterpret_cast<uintptr_t>(val) & 15) == 0;   // 16-byte stores
  spand::note_launch();
  k_assemble<P><<<K, assemble_threads<P>(), smem, st>>>(X, nt, nr, uh, fl, dtau, rhs, val, bad, vec, T);
  return SPAND_OK;
}

}  // namespace

extern "C" int dg_assemble_jacobian(const dg_mesh* mesh, int p, const double* u_hat,
                                    const dg_flow_params* flow, double* rhs, bsr_matrix* A,
                                    double* dtau_out, cudaStream_t stream) {
  if (!mesh || !flow || !A || !u_hat || !rhs || !mesh->nodes || !A->row_ptr || !A->col || !A->val)
    return SPAND_ERR_ARG;
  if (p < 1 || p > PMAX || mesh->n_theta < 4 || mesh->n_r < 1) return SPAND_ERR_UNSUPPORTED;
  const int nt = mesh->n_theta, nr = mesh->n_r, K = nt * nr, B = 4 * (p + 1) * (p + 1);
  A->K = K;
  A->B = B;
  A->nnzb = row_start(K - 1, nt, nr) + (nr == 1 ? 3 : 4);
  spand::note_launch();
  k_pattern<<<(K + 127) / 128, 128, 0, stream>>>(nt, nr, A->row_ptr, A->col);
  Flow fl;
  fl.gamma = flow->gamma;
  fl.cfl = flow->cfl;
  fl.bc_wall = flow->bc_mode == SPAND_BC_WALL;
  {
    const double a = flow->alpha_deg * M_PI / 180.0, g = flow->gamma;
    const double u = flow->mach * cos(a), v = flow->mach * sin(a), pr = 1.0 / g;
    fl.uinf[0] = 1.0;
    fl.uinf[1] = u;
    fl.uinf[2] = v;
    fl.uinf[3] = pr / (g - 1.0) + 0.5 * (u * u + v * v);
  }
  Tables T;
  memset(&T, 0, sizeof(T));
  T.q = p + 2;
  T.np = (p + 1) * (p + 1);
  T.Q = T.q * T.q;
  gauss_rule(T.q, T.tq, T.wq);
  for (int k = 0; k < T.q; ++k) legendre(p, T.tq[k], T.V[k], T.D[k]);
  for (int e = 0; e < 2; ++e) {
    double d[PMAX + 1];
    legendre(p, e ? -1.0 : 1.0, T.Vend[e], d);
  }
  for (int b = 0; b < T.q; ++b)
    for (int a = 0; a < T.q; ++a)
      for (int m = 0; m < T.np; ++m) T.psi[b * T.q + a][m] = T.V[a][m % (p + 1)] * T.V[b][m / (p + 1)];
  double* d_scr = nullptr;  // [0] = dtau, [1] = bad flag (as int)
  SPAND_CUDA_TRY(cudaMallocAsync(&d_scr, 2 * sizeof(double), stream));
  const double big = 1e300;
  SPAND_CUDA_TRY(cudaMemcpyAsync(d_scr, &big, sizeof(double), cudaMemcpyHostToDevice, stream));
  SPAND_CUDA_TRY(cudaMemsetAsync(d_scr + 1, 0, sizeof(double), stream));
  int* d_bad = reinterpret_cast<int*>(d_scr + 1);
  spand::note_launch();
  k_time_step<<<(K + 127) / 128, 128, 0, stream>>>(mesh->nodes, nt, nr, p, u_hat, fl, d_scr, d_bad, T);
  auto launch = p == 1 ? launch_assemble<1> : p == 2 ? launch_assemble<2> : launch_assemble<3>;
  SPAND_TRY(launch(K, mesh->nodes, nt, nr, u_hat, fl, d_scr, rhs, A->val, d_bad, T, stream));
  SPAND_CUDA_TRY(cudaGetLastError());
  double h[2];
  SPAND_CUDA_TRY(cudaMemcpyAsync(h, d_scr, 2 * sizeof(double), cudaMemcpyDeviceToHost, stream));
  SPAND_CUDA_TRY(cudaFreeAsync(d_scr, stream));
  SPAND_CUDA_TRY(cudaStreamSynchronize(stream));
  int badv;
  memcpy(&badv, &h[1], sizeof(int));
  if (dtau_out) *dtau_out = h[0];
  if (badv) return SPAND_ERR_NONFINITE;
  return SPAND_OK;
}
