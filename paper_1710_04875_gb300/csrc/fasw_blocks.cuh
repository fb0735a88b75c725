// The diagonal block of a cell and its LU factors, shared by the kernels that set up the preconditioner.
#pragma once
#include "fasw_fp64.cuh"
#include "fasw_internal.cuh"

namespace fasw {

// c_i and sigma of D_i = sigma I + c_i (A+_e - A-_w + B+_n - B-_s).
template <typename T>
__device__ __forceinline__ void diag_scales(const LevelDev& L, int aw, double eta, int c, double& coef, double& sigma) {
  if (aw) {
    const double ed = eta * L.dts[c];
    coef = sizeof(T) == 8 ? div64(ed, L.vol[c], L.rvol[c]) : ed / L.vol[c];
    sigma = is_zero(L.a_t) ? 1.0 : 1.0 + ed * L.a_t;
  } else {
    coef = L.rvol[c];
    sigma = L.a_t;
  }
}

// LU without pivoting of A: unit L below the diagonal, U on and above with the reciprocal of its
// diagonal stored on the diagonal.
template <typename T>
__device__ __forceinline__ void lu4(T A[16]) {
  if constexpr (sizeof(T) == 8) {  // each pivot's reciprocal once, for its column's multipliers too
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double d = A[5 * k];
      A[5 * k] = rcp64(d);
#pragma unroll
      for (int r = k + 1; r < 4; ++r) {
        const double m = div64(A[4 * r + k], d, A[5 * k]);
        A[4 * r + k] = m;
#pragma unroll
        for (int cc = k + 1; cc < 4; ++cc) A[4 * r + cc] -= m * A[4 * k + cc];
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int r = k + 1; r < 4; ++r) {
        const T m = A[4 * r + k] / A[4 * k + k];
        A[4 * r + k] = m;
#pragma unroll
        for (int cc = k + 1; cc < 4; ++cc) A[4 * r + cc] -= m * A[4 * k + cc];
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) A[5 * k] = T(1) / A[5 * k];
  }
}

// D's LU factors of cell c; stores c_i (returned in cf too) and u^(0), the state the blocks are frozen at.
template <typename T>
__device__ __forceinline__ void cell_lu(const LevelDev& L, const T* blk, int aw, double eta, int c, T A[16], T& cf) {
  const int ni = L.ni, i = c % ni, j = c / ni;
  double coef, sigma;
  diag_scales<T>(L, aw, eta, c, coef, sigma);
  L.coef[c] = coef;
  {
    const int g = (j + 2) * L.P + (i + 2);
#pragma unroll
    for (int k = 0; k < 4; ++k) L.u0[k * L.n + c] = L.u[k * L.Gn + g];
  }
  const int fw = j * (ni + 1) + i, fe = fw + 1, fs = j * ni + i, fn = fs + ni;
  const T* Axp = blk;
  const T* Axm = blk + 16 * L.nfx;
  const T* Aep = blk + 32 * L.nfx;
  const T* Aem = blk + 32 * L.nfx + 16 * L.nfe;
  cf = from64<T>(coef);
  const T sg = from64<T>(sigma);
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const T v = (Axp[e * L.nfx + fe] - Axm[e * L.nfx + fw]) + (Aep[e * L.nfe + fn] - Aem[e * L.nfe + fs]);
    A[e] = ((e % 5 == 0) ? sg : T(0)) + cf * v;
  }
  lu4<T>(A);
}

}  // namespace fasw
