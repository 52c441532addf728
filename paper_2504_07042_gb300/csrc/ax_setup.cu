// Setup-stage kernels (FP64 arithmetic; run once per context):
//   - validation: det J > 0 at every GLL node (analytic trilinear Jacobian),
//   - STORED: the seven factors per node from the standard discrete Jacobian
//     of Sec. 3.2 (nodal coordinates, then the discrete gradient D of
//     Table 1), then Eq. 7,
//   - PARALLELEPIPED: h0..h6 of Algorithm 3 from the constant Jacobian, plus
//     a check that every element is affine,
//   - TRILINEAR kinds: vertex coordinates relative to vertex 0 (24 words),
//   - PARTIAL: the per-node scalar w_i w_j w_k / det J (Sec. 4.2.2),
//   - node coordinates (Eq. 8 at the GLL points).
// Results are written in the storage format of the context's precision:
// float64, float32, or a double-word pair (float hi, float lo).
#include <cstdint>

#include "ax_internal.h"
#include "tables.cuh"

namespace ax {
namespace setup {

static __constant__ double c_D[kTabD];
static __constant__ double c_w[kTabV];
static __constant__ double c_x[kTabV];

enum Store { kF64 = 0, kF32 = 1, kDW = 2 };

// Write v in the storage format.  FP32-based formats: values above 1e30 are
// counted as out of range (products of them could overflow); values below
// 1e-30 are stored as zero (an absolute error far below the tolerances).
__device__ __forceinline__ void store(void *base, int64_t idx, double v, int fmt, int *flags) {
  if (fmt == kF64) {
    ((double *)base)[idx] = v;
    return;
  }
  const double a = fabs(v);
  if (!(a <= 1e30)) atomicAdd(&flags[2], 1);
  if (a < 1e-30) v = 0.0;
  if (fmt == kF32) {
    ((float *)base)[idx] = (float)v;
  } else {
    const float hi = (float)v;
    const float lo = (float)(v - (double)hi);
    ((float2 *)base)[idx] = make_float2(hi, lo);
  }
}

// Trilinear map (Eq. 8) at reference point (r,s,t).
__device__ void map_point(const double *V, double r, double s, double t, double X[3]) {
  for (int c = 0; c < 3; ++c) X[c] = 0.0;
  for (int v = 0; v < 8; ++v) {
    const double wv = (1.0 + ((v & 1) ? r : -r)) * (1.0 + ((v & 2) ? s : -s)) * (1.0 + ((v & 4) ? t : -t)) * 0.125;
    for (int c = 0; c < 3; ++c) X[c] += wv * V[3 * v + c];
  }
}

// Analytic Jacobian of the trilinear map, J[c][d] = d x_c / d ref_d.
__device__ void map_jacobian(const double *V, double r, double s, double t, double J[9]) {
  for (int q = 0; q < 9; ++q) J[q] = 0.0;
  for (int v = 0; v < 8; ++v) {
    const double sr = (v & 1) ? 1.0 : -1.0, ss = (v & 2) ? 1.0 : -1.0, st = (v & 4) ? 1.0 : -1.0;
    const double fr = 1.0 + sr * r, fs = 1.0 + ss * s, ft = 1.0 + st * t;
    const double d[3] = {sr * fs * ft * 0.125, fr * ss * ft * 0.125, fr * fs * st * 0.125};
    for (int c = 0; c < 3; ++c)
      for (int q = 0; q < 3; ++q) J[3 * c + q] += d[q] * V[3 * v + c];
  }
}

__device__ double det3(const double J[9]) {
  return J[0] * (J[4] * J[8] - J[5] * J[7]) - J[1] * (J[3] * J[8] - J[5] * J[6]) + J[2] * (J[3] * J[7] - J[4] * J[6]);
}

// G = W |J| J^-1 J^-T = W adj(J) adj(J)^T / det J  (6 entries), gwj = W det J.
__device__ void factors_from_J(const double J[9], double W, double g[7]) {
  const double det = det3(J);
  double A[9];  // adjugate (transpose of the cofactor matrix): J^-1 = A / det
  A[0] = J[4] * J[8] - J[5] * J[7];
  A[1] = J[2] * J[7] - J[1] * J[8];
  A[2] = J[1] * J[5] - J[2] * J[4];
  A[3] = J[5] * J[6] - J[3] * J[8];
  A[4] = J[0] * J[8] - J[2] * J[6];
  A[5] = J[2] * J[3] - J[0] * J[5];
  A[6] = J[3] * J[7] - J[4] * J[6];
  A[7] = J[1] * J[6] - J[0] * J[7];
  A[8] = J[0] * J[4] - J[1] * J[3];
  const int pr[6][2] = {{0, 0}, {0, 1}, {0, 2}, {1, 1}, {1, 2}, {2, 2}};
  for (int q = 0; q < 6; ++q) {
    const int p = pr[q][0], m = pr[q][1];
    const double dot = A[3 * p] * A[3 * m] + A[3 * p + 1] * A[3 * m + 1] + A[3 * p + 2] * A[3 * m + 2];
    g[q] = W * dot / det;
  }
  g[6] = W * det;
}

// Element extents the FP32-based formats (float32, double-word pairs) handle
// at full accuracy: the trilinear geometry forms products of up to four
// Jacobian entries (adj(J^T J)); with entries of size L/2 these stay inside
// float32's normal range, low words and error terms included, for element
// extents L in [2^-20, 2^24] (adj ~ L^4 between about 2^-84 and 2^92).
constexpr double kMinExtent = 0x1p-20, kMaxExtent = 0x1p24;

// One thread per node.  flags[0] += nodes with det J <= 0; for the
// FP32-based formats flags[3] += elements whose extent (largest vertex
// coordinate difference from vertex 0) lies outside [kMinExtent, kMaxExtent].
__global__ void validate_kernel(int64_t E, int N1, const double *__restrict__ V, int fmt, int *flags) {
  const int64_t n3 = (int64_t)N1 * N1 * N1;
  const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gidx >= E * n3) return;
  const int64_t e = gidx / n3;
  const int l = (int)(gidx % n3), i = l % N1, j = (l / N1) % N1, k = l / (N1 * N1);
  const double *cx = c_x + tab_off_v(N1);
  double J[9];
  map_jacobian(V + 24 * e, cx[i], cx[j], cx[k], J);
  if (!(det3(J) > 0.0)) atomicAdd(&flags[0], 1);
  if (fmt != kF64 && l == 0) {
    const double *Ve = V + 24 * e;
    double ext = 0.0;
    for (int v = 1; v < 8; ++v)
      for (int c = 0; c < 3; ++c) ext = fmax(ext, fabs(Ve[3 * v + c] - Ve[c]));
    if (!(ext >= kMinExtent && ext <= kMaxExtent)) atomicAdd(&flags[3], 1);
  }
}

// STORED: discrete Jacobian of Sec. 3.2 -- the derivative along each reference
// direction is D applied to the nodal coordinates on the line through the node.
__global__ void stored_factors_kernel(int64_t E, int N1, const double *__restrict__ V, void *G, int fmt, int *flags) {
  const int64_t n3 = (int64_t)N1 * N1 * N1;
  const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gidx >= E * n3) return;
  const int64_t e = gidx / n3;
  const int l = (int)(gidx % n3), i = l % N1, j = (l / N1) % N1, k = l / (N1 * N1);
  const double *cD = c_D + tab_off_D(N1), *cx = c_x + tab_off_v(N1), *cw = c_w + tab_off_v(N1);
  const double *Ve = V + 24 * e;
  double J[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (int n = 0; n < N1; ++n) {
    double Xr[3], Xs[3], Xt[3];
    map_point(Ve, cx[n], cx[j], cx[k], Xr);
    map_point(Ve, cx[i], cx[n], cx[k], Xs);
    map_point(Ve, cx[i], cx[j], cx[n], Xt);
    for (int c = 0; c < 3; ++c) {
      J[3 * c + 0] += cD[i * N1 + n] * Xr[c];
      J[3 * c + 1] += cD[j * N1 + n] * Xs[c];
      J[3 * c + 2] += cD[k * N1 + n] * Xt[c];
    }
  }
  double g[7];
  factors_from_J(J, cw[i] * cw[j] * cw[k], g);
  for (int q = 0; q < 7; ++q) store(G, (e * 7 + q) * n3 + l, g[q], fmt, flags);
}

// Vertices relative to vertex 0 (24 words per element; row 0 is zero).
// TRILINEAR record: the trilinear map of Eq. 8 written in the monomial basis,
//   x(r,s,t) = x0 + A r + B s + C t + D rs + E rt + F st + G rst,
// each coefficient (1/8) sum_v sigma(v) (V_v - V_0) with the sign pattern of
// its monomial (sigma = +-1 from the vertex's corner, v = a + 2b + 4c); the
// vertex-0 offset cancels in every sign sum, and subtracting it first keeps
// the sums free of cancellation far from the origin.  Words: A B C D E F G
// (3 coordinates each) and 3 zero pads.  Then the Jacobian's columns are
//   J0 = (A + D s) + t (E + G s),  J1 = (B + D r) + t (F + G r),
//   J2 = C + E r + F s + G r s.
__global__ void trilinear_coeffs_kernel(int64_t E, const double *__restrict__ V, void *out, int fmt, int *flags) {
  const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gidx >= E * 24) return;
  const int64_t e = gidx / 24;
  const int q = (int)(gidx % 24), m = q / 3, c = q % 3;
  double acc = 0.0;
  if (m < 7) {
    // monomials r, s, t, rs, rt, st, rst: which of (a, b, c) enter the sign
    const int use[7] = {1, 2, 4, 3, 5, 6, 7};
    for (int v = 0; v < 8; ++v) {
      int sgn = 1;
      for (int d = 0; d < 3; ++d)
        if ((use[m] >> d) & 1) sgn *= ((v >> d) & 1) ? 1 : -1;
      acc += sgn * (V[24 * e + 3 * v + c] - V[24 * e + c]);
    }
    acc *= 0.125;
  }
  store(out, gidx, acc, fmt, flags);
}

// PARALLELEPIPED: J = [v1-v0, v2-v0, v4-v0] / 2 (columns) is constant;
// h0..h5 = |J| J^-1 J^-T, h6 = |J| (Algorithm 3 input, without GLL weights).
// flags[1] += elements whose vertices deviate from v0 + a e1 + b e2 + c e3.
__global__ void parallelepiped_kernel(int64_t E, const double *__restrict__ V, void *out, int fmt, int *flags) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  const double *Ve = V + 24 * e;
  double J[9], scale = 0.0;
  for (int c = 0; c < 3; ++c) {
    J[3 * c + 0] = 0.5 * (Ve[3 + c] - Ve[c]);
    J[3 * c + 1] = 0.5 * (Ve[6 + c] - Ve[c]);
    J[3 * c + 2] = 0.5 * (Ve[12 + c] - Ve[c]);
    for (int d = 0; d < 3; ++d) scale = fmax(scale, fabs(J[3 * c + d]));
  }
  double dev = 0.0;
  for (int v = 0; v < 8; ++v) {
    const int a = v & 1, b = (v >> 1) & 1, cc = (v >> 2) & 1;
    for (int c = 0; c < 3; ++c) {
      const double pred = Ve[c] + 2.0 * (a * J[3 * c] + b * J[3 * c + 1] + cc * J[3 * c + 2]);
      dev = fmax(dev, fabs(pred - Ve[3 * v + c]));
    }
  }
  if (dev > 1e-12 * scale) atomicAdd(&flags[1], 1);
  double g[7];
  factors_from_J(J, 1.0, g);
  for (int q = 0; q < 7; ++q) store(out, e * kParWords + q, g[q], fmt, flags);
  store(out, e * kParWords + 7, 0.0, fmt, flags);
}

// PARTIAL: lam = w_i w_j w_k / det J at every node.
__global__ void partial_lam_kernel(int64_t E, int N1, const double *__restrict__ V, void *out, int fmt, int *flags) {
  const int64_t n3 = (int64_t)N1 * N1 * N1;
  const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gidx >= E * n3) return;
  const int64_t e = gidx / n3;
  const int l = (int)(gidx % n3), i = l % N1, j = (l / N1) % N1, k = l / (N1 * N1);
  const double *cx = c_x + tab_off_v(N1), *cw = c_w + tab_off_v(N1);
  double J[9];
  map_jacobian(V + 24 * e, cx[i], cx[j], cx[k], J);
  store(out, gidx, cw[i] * cw[j] * cw[k] / det3(J), fmt, flags);
}

__global__ void node_coords_kernel(int64_t E, int N1, const double *__restrict__ V, double *xyz) {
  const int64_t n3 = (int64_t)N1 * N1 * N1;
  const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gidx >= E * n3) return;
  const int64_t e = gidx / n3;
  const int l = (int)(gidx % n3), i = l % N1, j = (l / N1) % N1, k = l / (N1 * N1);
  const double *cx = c_x + tab_off_v(N1);
  double X[3];
  map_point(V + 24 * e, cx[i], cx[j], cx[k], X);
  for (int c = 0; c < 3; ++c) xyz[(e * 3 + c) * n3 + l] = X[c];
}

// Y = w_i w_j w_k det J * F at every node (the seventh factor times F).
template <typename T>
__global__ void mass_kernel(int64_t E, int N1, const double *__restrict__ V, const T *__restrict__ F, T *__restrict__ Y) {
  const int64_t n3 = (int64_t)N1 * N1 * N1;
  const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gidx >= E * n3) return;
  const int64_t e = gidx / n3;
  const int l = (int)(gidx % n3), i = l % N1, j = (l / N1) % N1, k = l / (N1 * N1);
  const double *cx = c_x + tab_off_v(N1), *cw = c_w + tab_off_v(N1);
  double J[9];
  map_jacobian(V + 24 * e, cx[i], cx[j], cx[k], J);
  Y[gidx] = (T)(cw[i] * cw[j] * cw[k] * det3(J) * (double)F[gidx]);
}

// Diagonal of the element matrix D^T G D at node l = (i,j,k):
//   sum_n (D[n][i]^2 g00(n,j,k) + D[n][j]^2 g11(i,n,k) + D[n][k]^2 g22(i,j,n))
//   + 2 (D[i][i] D[j][j] g01 + D[i][i] D[k][k] g02 + D[j][j] D[k][k] g12)(l)
//
// One thread per (i,j), all its k: bound by the FP64 pipe (2 operations per
// clock and SM), so the split keeps the FP64 operations few.  The Jacobian of
// the trilinear map is formed from its monomial coefficients
//   x = x0 + A r + B s + C t + D rs + E rt + F st + G rst  (Eq. 8)
// (8 additions per coefficient, shared by the element), in the columns
//   J0 = (A + D s) + t (E + G s),  J1 = (B + D r) + t (F + G r),
//   J2 = C + E r + F s + G r s,
// of which only six multiply-adds change along k; with the cofactor rows
// c0 = J1 x J2, c1 = J2 x J0, c2 = J0 x J1, det J = J2 . c2 and
// g_ab = (w / det J) c_a . c_b.  g00 and g11 are summed along their own
// directions through shared memory, g22 in the thread's own registers.
// About 60 + 3 N1 FP64 operations per node.  The form it replaces (all seven
// factors of every node by the discrete Jacobian of Sec. 3.2, N1 map
// evaluations per direction and node, written to and read back from HBM)
// took 200 N1 and more, 18.8 ms for 16 meshes of orders 3 to 9 (7.9M nodes)
// on GB300; a batched solve of 20 iterations on them, which starts with it,
// went from 26.4 to 8.1 ms.
template <int N1>
struct DiagShape {
  static constexpr int F = N1 * N1, n3 = F * N1, EPB = F >= 128 ? 1 : 128 / F, threads = F * EPB;
  static constexpr int P = N1 + 1;                // padded row of the shared factors
  static constexpr int ES = F * P;                // padded element
  static constexpr size_t words = 2 * (size_t)EPB * ES + EPB * 21 + F;  // g00, g11, coefficients, D^2
};
template <typename T, int N1>
__global__ void __launch_bounds__(DiagShape<N1>::threads)
    diag_kernel(int64_t E, const double *__restrict__ V, T *__restrict__ out) {
  using Sh = DiagShape<N1>;
  constexpr int F = Sh::F, EPB = Sh::EPB, P = Sh::P;
  extern __shared__ double sm_diag[];
  double *g00 = sm_diag, *g11 = g00 + EPB * Sh::ES, *coef = g11 + EPB * Sh::ES, *D2 = coef + EPB * 21;
  const double *cD = c_D + tab_off_D(N1), *cx = c_x + tab_off_v(N1), *cw = c_w + tab_off_v(N1);
  const int tid = threadIdx.x, z = tid / F, q = tid % F, i = q % N1, j = q / N1;
  for (int m = tid; m < F; m += Sh::threads) D2[m] = cD[m] * cD[m];
  const double r = cx[i], s = cx[j], wij = cw[i] * cw[j];
  const double di = cD[i * N1 + i], dj = cD[j * N1 + j];
  const int64_t nblk = (E + EPB - 1) / EPB;
  for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    const int64_t e0 = blk * EPB;
    const int nel = (int)((E - e0) < EPB ? (E - e0) : EPB);
    // monomial coefficients: (1/8) sum_v sigma(v) (V_v - V_0), as trilinear_coeffs_kernel
    for (int m = tid; m < nel * 21; m += Sh::threads) {
      const int el = m / 21, mono = (m % 21) / 3, c = m % 3;
      const int use = mono < 2 ? mono + 1 : mono == 2 ? 4 : mono == 3 ? 3 : mono + 1;  // 1 2 4 3 5 6 7
      const double *Ve = V + 24 * (e0 + el);
      double acc = 0.0;
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const double d = Ve[3 * v + c] - Ve[c];
        acc += (__popc(use & ~v) & 1) ? -d : d;
      }
      coef[m] = acc * 0.125;
    }
    __syncthreads();
    const bool live = z < nel;
    double y[N1];
    if (live) {
      const double *M = coef + z * 21;  // A B C D E F G
      double E0[3], E1[3], F0[3], F1[3], J2[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        E0[c] = fma(M[9 + c], s, M[c]);
        E1[c] = fma(M[18 + c], s, M[12 + c]);
        F0[c] = fma(M[9 + c], r, M[3 + c]);
        F1[c] = fma(M[18 + c], r, M[15 + c]);
        J2[c] = fma(E1[c], r, fma(M[15 + c], s, M[6 + c]));
      }
#pragma unroll
      for (int k = 0; k < N1; ++k) y[k] = 0.0;
      double *g0 = g00 + z * Sh::ES + i + P * j, *g1 = g11 + z * Sh::ES + i + P * j;
#pragma unroll
      for (int k = 0; k < N1; ++k) {
        const double t = cx[k], dk = cD[k * N1 + k];
        double J0[3], J1[3], c0[3], c1[3], c2[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          J0[c] = fma(t, E1[c], E0[c]);
          J1[c] = fma(t, F1[c], F0[c]);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int a = (c + 1) % 3, b = (c + 2) % 3;
          c0[c] = J1[a] * J2[b] - J1[b] * J2[a];
          c1[c] = J2[a] * J0[b] - J2[b] * J0[a];
          c2[c] = J0[a] * J1[b] - J0[b] * J1[a];
        }
        const double det = J2[0] * c2[0] + J2[1] * c2[1] + J2[2] * c2[2];
        const double lam = wij * cw[k] / det;
        auto dot = [](const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
        g0[P * N1 * k] = lam * dot(c0, c0);
        g1[P * N1 * k] = lam * dot(c1, c1);
        const double g22 = lam * dot(c2, c2);
        // D[i][i] (D[j][j] g01 + D[k][k] g02) + D[j][j] D[k][k] g12
        const double cross = di * (dj * dot(c0, c1) + dk * dot(c0, c2)) + dj * dk * dot(c1, c2);
        y[k] = fma(2.0 * lam, cross, y[k]);
#pragma unroll
        for (int n = 0; n < N1; ++n) y[n] = fma(D2[k * N1 + n], g22, y[n]);
      }
    }
    __syncthreads();  // every g00, g11 is in place
    if (live) {
      T *o = out + (e0 + z) * (int64_t)Sh::n3 + i + N1 * j;
#pragma unroll 1
      for (int n = 0; n < N1; ++n) {
        const double a = D2[n * N1 + i], b = D2[n * N1 + j];
        const double *g0 = g00 + z * Sh::ES + n + P * j, *g1 = g11 + z * Sh::ES + i + P * n;
#pragma unroll
        for (int k = 0; k < N1; ++k) y[k] = fma(a, g0[P * N1 * k], fma(b, g1[P * N1 * k], y[k]));
      }
#pragma unroll
      for (int k = 0; k < N1; ++k) o[F * k] = (T)y[k];
    }
    __syncthreads();  // the next block reuses the shared buffers
  }
}

template <typename T, int N1>
cudaError_t launch_diag(int64_t E, const double *V, T *out, cudaStream_t s) {
  using Sh = DiagShape<N1>;
  constexpr size_t bytes = Sh::words * sizeof(double);
  const int64_t nblk = (E + Sh::EPB - 1) / Sh::EPB;
  const unsigned grid = (unsigned)(nblk < 0x7fffffffLL ? nblk : 0x7fffffffLL);
  if (bytes > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(diag_kernel<T, N1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
  }
  diag_kernel<T, N1><<<grid, Sh::threads, bytes, s>>>(E, V, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_diag_n(int N1, int64_t E, const double *V, T *out, cudaStream_t s) {
  switch (N1) {
#define AX_DIAG(n) \
  case n: return launch_diag<T, n>(E, V, out, s);
    AX_DIAG(2) AX_DIAG(3) AX_DIAG(4) AX_DIAG(5) AX_DIAG(6) AX_DIAG(7) AX_DIAG(8) AX_DIAG(9)
    AX_DIAG(10) AX_DIAG(11) AX_DIAG(12) AX_DIAG(13) AX_DIAG(14) AX_DIAG(15) AX_DIAG(16)
#undef AX_DIAG
    default: return cudaErrorInvalidValue;
  }
}

static unsigned grid_for(int64_t n, int block) { return (unsigned)((n + block - 1) / block); }

}  // namespace setup

static UploadOnce g_once_setup;

cudaError_t upload_tables_setup(int device) {
  std::lock_guard<std::mutex> lock(g_once_setup.mu);
  if (device < 64 && (g_once_setup.done >> device) & 1ull) return cudaSuccess;
  static double D[kTabD], w[kTabV], x[kTabV];
  if (!build_packed_tables(D, w, x)) return cudaErrorInvalidValue;
  cudaError_t err = cudaMemcpyToSymbol(setup::c_D, D, sizeof(D));
  if (err == cudaSuccess) err = cudaMemcpyToSymbol(setup::c_w, w, sizeof(w));
  if (err == cudaSuccess) err = cudaMemcpyToSymbol(setup::c_x, x, sizeof(x));
  if (err == cudaSuccess && device < 64) g_once_setup.done |= 1ull << device;
  return err;
}

cudaError_t setup_geometry(const Ctx &c, const double *V, void *geo, void *lam, int *flags, cudaStream_t s) {
  using namespace setup;
  const int fmt = (c.prec == AX_FP64) ? kF64 : (c.prec == AX_F64DW ? kDW : kF32);
  const int64_t nodes = c.E * (int64_t)c.n3;
  const int B = 256;
  if (c.E == 0) return cudaSuccess;
  if ((nodes + B - 1) / B > 0x7fffffffLL) return cudaErrorInvalidValue;
  validate_kernel<<<grid_for(nodes, B), B, 0, s>>>(c.E, c.N1, V, fmt, flags);
  switch (c.kind) {
    case AX_GEOM_STORED:
      stored_factors_kernel<<<grid_for(nodes, B), B, 0, s>>>(c.E, c.N1, V, geo, fmt, flags);
      break;
    case AX_GEOM_PARALLELEPIPED:
      parallelepiped_kernel<<<grid_for(c.E, B), B, 0, s>>>(c.E, V, geo, fmt, flags);
      break;
    case AX_GEOM_TRILINEAR_PARTIAL:
      partial_lam_kernel<<<grid_for(nodes, B), B, 0, s>>>(c.E, c.N1, V, lam, fmt, flags);
      trilinear_coeffs_kernel<<<grid_for(c.E * 24, B), B, 0, s>>>(c.E, V, geo, fmt, flags);
      break;
    case AX_GEOM_TRILINEAR:
      trilinear_coeffs_kernel<<<grid_for(c.E * 24, B), B, 0, s>>>(c.E, V, geo, fmt, flags);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t setup_node_coords(const Ctx &c, const double *V, double *xyz, cudaStream_t s) {
  const int64_t nodes = c.E * (int64_t)c.n3;
  if (nodes == 0) return cudaSuccess;
  setup::node_coords_kernel<<<setup::grid_for(nodes, 256), 256, 0, s>>>(c.E, c.N1, V, xyz);
  return cudaGetLastError();
}

}  // namespace ax

namespace ax {

cudaError_t setup_mass(const Ctx &c, const double *V, const void *F, void *Y, bool f64, cudaStream_t s) {
  const int64_t nodes = c.E * (int64_t)c.n3;
  if (nodes == 0) return cudaSuccess;
  if (f64)
    setup::mass_kernel<double><<<setup::grid_for(nodes, 256), 256, 0, s>>>(c.E, c.N1, V, (const double *)F, (double *)Y);
  else
    setup::mass_kernel<float><<<setup::grid_for(nodes, 256), 256, 0, s>>>(c.E, c.N1, V, (const float *)F, (float *)Y);
  return cudaGetLastError();
}

cudaError_t setup_diag(const Ctx &c, const double *V, void *diag, bool f64, cudaStream_t s) {
  if (c.E == 0) return cudaSuccess;
  return f64 ? setup::launch_diag_n<double>(c.N1, c.E, V, (double *)diag, s)
             : setup::launch_diag_n<float>(c.N1, c.E, V, (float *)diag, s);
}

}  // namespace ax
