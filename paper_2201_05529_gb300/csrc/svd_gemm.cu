// FP64 GEMM of the SVD's finish (App. A.2): U_D = D V_D on the columns the truncation keeps,
// batched over the bonds of a layer with each bond's live dims read from its info words.
#include "kernels.h"

namespace ptk {

namespace {

__device__ __forceinline__ void shape(const BondWork& W, int* Ma, int* Na) {
  const int mD = W.info[0], nD = W.info[1];
  const bool tr = W.info[2] != 0;
  *Ma = (mD > 0 && nD > 0) ? (tr ? nD : mD) : 0;
  *Na = (mD > 0 && nD > 0) ? (tr ? mD : nD) : 0;
}

constexpr int TB = 16;   // GEMM tile: one output per thread, so that a layer of two bonds fills more SMs (a 2 x 2
                         // block per thread in 32 x 32 tiles: 90 us for two 144 x 144 x 40, FP64 issue on 20 SMs; 45 us so)
constexpr int TK = 16;   // GEMM K tile

// C[m x n] = op(A)[m x k] * B[k x n], column-major; op = conjugate transpose if conjA.
// 256 threads, one entry of a 16 x 16 tile each.
// bcol: column c of B is column bcol[c] of the stored matrix (NULL: c). K runs from k_from (a multiple of TK).
// div: column c of the result is divided by div[bcol[c]] (a zero gives a zero column).
__device__ void gemm_tile(const double2* A, int lda, bool conjA, const double2* B, int ldb, double2* C, int ldc,
                          int m, int n, int k, int tm, int tn, const int* bcol = nullptr, int k_from = 0,
                          const double* div = nullptr) {
  __shared__ double2 As[TK][TB + 1];
  __shared__ double2 Bs[TK][TB + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;      // row tx, column ty of the tile
  double2 acc = make_double2(0.0, 0.0), acc2 = acc;
  for (int k0 = k_from; k0 < k; k0 += TK) {
    {
      // thread (mm, kk) loads one element of each operand's tile
      const int mm = tx, kk = ty;
      const int row = tm * TB + mm, col = k0 + kk;
      double2 a = make_double2(0.0, 0.0);
      if (row < m && col < k) {
        if (conjA) {
          const double2 x = A[col + (size_t)row * lda];     // (A^H)[row, col] = conj(A[col, row])
          a = make_double2(x.x, -x.y);
        } else {
          a = A[row + (size_t)col * lda];
        }
      }
      As[kk][mm] = a;
      const int br = k0 + tx, bc = tn * TB + ty;            // B's tile along its columns
      Bs[tx][ty] = (bc < n && br < k) ? B[br + (size_t)(bcol ? bcol[bc] : bc) * ldb] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; kk += 2) {
      const double2 a = As[kk][tx], b = Bs[kk][ty], c = As[kk + 1][tx], d = Bs[kk + 1][ty];
      acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
      acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
      acc2.x = fma(c.x, d.x, fma(-c.y, d.y, acc2.x));
      acc2.y = fma(c.x, d.y, fma(c.y, d.x, acc2.y));
    }
    __syncthreads();
  }
  const int row = tm * TB + tx, col = tn * TB + ty;
  if (row < m && col < n) {
    double2 v = make_double2(acc.x + acc2.x, acc.y + acc2.y);
    if (div) {
      const double s = div[bcol[col]];
      v = s > 0.0 ? make_double2(v.x / s, v.y / s) : make_double2(0.0, 0.0);
    }
    C[row + (size_t)col * ldc] = v;
  }
}

}  // namespace

// Y64[:, c] = A V[:, perm[c]] for the kept columns c < lam_chi[bond] (grid: tiles x tiles x items)
__global__ void __launch_bounds__(256) k_mix_gemm(const BondWork* work, int n_work, const int* lam_chi) {
  const int w = blockIdx.z;
  if (w >= n_work) return;
  const BondWork& W = work[w];
  int Ma, Na;
  shape(W, &Ma, &Na);
  const int tm = blockIdx.x, tn = blockIdx.y;
  const int n = min(lam_chi[W.lam_l + 1], Na);
  if (tm * TB >= Ma || tn * TB >= n) return;
  gemm_tile(W.A, Ma, false, W.V, Na, W.Y64, Ma, Ma, n, Na, tm, tn, W.perm);
}

void launch_mix_gemm_av(const BondWork* work, int n_work, int k_cap, int m_cap, const int* lam_chi, cudaStream_t st) {
  const int tk = (k_cap + TB - 1) / TB, tmm = (m_cap + TB - 1) / TB;
  k_mix_gemm<<<dim3(tmm, tk, n_work), 256, 0, st>>>(work, n_work, lam_chi);
}

// Ur = R Wr / S on the kept columns (grid: tiles x tiles x items): R upper triangular in G64, so K starts at the
// tile's diagonal. What the Jacobi would spend on accumulating this factor (8 of its 20 FP64 operations per row and
// rotated pair, ~9 sweeps) is one product of 4 l^2 chi operations here.
__global__ void __launch_bounds__(256) k_rsvd_left(const BondWork* work, int n_work, const int* lam_chi) {
  const int w = blockIdx.z;
  if (w >= n_work) return;
  const BondWork& W = work[w];
  int Ma, Na;
  shape(W, &Ma, &Na);
  const int l = Ma > 0 ? W.info[9] : 0;
  const int n = min(lam_chi[W.lam_l + 1], l);
  const int tm = blockIdx.x, tn = blockIdx.y;
  if (tm * TB >= l || tn * TB >= n) return;
  gemm_tile(W.G64, l, false, W.V, l, W.RH, l, l, n, l, tm, tn, W.perm, tm * TB, W.sig);
}

void launch_rsvd_left(const BondWork* work, int n_work, int l_cap, const int* lam_chi, cudaStream_t st) {
  const int t = (l_cap + TB - 1) / TB;
  k_rsvd_left<<<dim3(t, t, n_work), 256, 0, st>>>(work, n_work, lam_chi);
}

}  // namespace ptk
