// The standalone FP64 SVD after two QR factorisations (Drmac and Veselic's preconditioning, with the columns and
// rows sorted by norm once instead of pivoting):
//   P' A P = Q1 R1,  R1^H = Q2 R2,  R2^H = W S Z^H by the Jacobi   ->   A = (P'^T Q1 W) S (P Q2 Z)^H
// (A^H instead of A where it is wide). What bounds the Jacobi is the number of sweeps and the length of the columns: on
// a matrix with singular values over four decades it takes 16 sweeps at 64 x 64 and 20 at 256 x 256, on R1^H 10 and 12,
// on R2^H 8 and 9 (a third QR would save none at 256), and the rows beyond n leave it with the first QR. The two QRs
// (qr_block.cu) and the two products run on the tensor cores at the accuracy of FP64 products and cost about two
// sweeps of the 256 x 256 Jacobi. The sorting keeps R1 graded along its diagonal, so that columns or rows of very different
// scale keep their own accuracy (each singular value of B D or D B, B well conditioned, D over twelve decades: 3e-14 relative).
#include <algorithm>
#include <vector>

#include "kernels.h"

namespace ptk {

namespace {

constexpr int TT = 32;                     // tile edge of the transposing kernels, 32 x 8 threads

__device__ __forceinline__ double2 conj2(double2 v) { return make_double2(v.x, -v.y); }

// squared norms of the columns of A (of A^H: the rows) of row-major A_b, up to an order: 32 columns x 8 row classes
__global__ void k_svd_norms(const double2* A, int m, int n, bool tr, double* nrm) {
  __shared__ double s[8][TT + 1];
  const int b = blockIdx.y, Na = tr ? m : n, len = tr ? n : m;
  const double2* Ab = A + (size_t)b * m * n;
  if (tr) {                                // a warp per row
    const int c = blockIdx.x * 8 + threadIdx.y;
    if (c >= Na) return;                   // uniform across the warp
    double v = 0;
    for (int r = threadIdx.x; r < len; r += 32) {
      const double2 x = Ab[(size_t)c * n + r];
      v = fma(x.x, x.x, fma(x.y, x.y, v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) nrm[(size_t)b * Na + c] = v;
    return;
  }
  const int c = blockIdx.x * TT + threadIdx.x;
  double v = 0;
  if (c < Na)
    for (int r = threadIdx.y; r < len; r += 8) {
      const double2 x = Ab[(size_t)r * n + c];
      v = fma(x.x, x.x, fma(x.y, x.y, v));
    }
  s[threadIdx.y][threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.y == 0 && c < Na) {
    for (int k = 1; k < 8; ++k) v += s[k][threadIdx.x];
    nrm[(size_t)b * Na + c] = v;
  }
}

// pos[c]: the rank of column c, largest norm first, by index on ties; compared as bits, so that the ranks are a
// permutation whatever the values
__global__ void k_svd_rank(const double* nrm, int Na, int batch, int* pos) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= Na * batch) return;
  const double* s = nrm + (size_t)(idx / Na) * Na;
  const int c = idx % Na;
  const unsigned long long me = (unsigned long long)__double_as_longlong(s[c]);
  int rk = 0;
  for (int k = 0; k < Na; ++k) {
    const unsigned long long o = (unsigned long long)__double_as_longlong(__ldg(s + k));
    rk += o > me || (o == me && k < c);
  }
  pos[idx] = rk;
}

// entry (prow[r], pcol[c]) of out_b (column-major, Ma rows) = entry (r, c) of A_b, or of A_b^H
__global__ void k_svd_load_sorted(const double2* A, int m, int n, bool tr, const int* prow, const int* pcol,
                                  double2* out) {
  __shared__ double2 t[TT][TT + 1];
  const int b = blockIdx.z, Ma = tr ? n : m, Na = tr ? m : n;
  const double2* Ab = A + (size_t)b * m * n;
  double2* o = out + (size_t)b * Ma * Na;
  const int *pc = pcol + (size_t)b * Na, *pr = prow + (size_t)b * Ma;
  const int j0 = blockIdx.x * TT, i0 = blockIdx.y * TT;        // row-major tile: rows i0.., columns j0..
  for (int k = threadIdx.y; k < TT; k += 8) {
    const int i = i0 + k, j = j0 + threadIdx.x;
    if (i >= m || j >= n) continue;
    const double2 v = Ab[(size_t)i * n + j];
    if (tr) o[pr[j] + (size_t)pc[i] * Ma] = conj2(v);
    else t[k][threadIdx.x] = v;
  }
  if (tr) return;
  __syncthreads();
  for (int k = threadIdx.y; k < TT; k += 8) {
    const int i = i0 + threadIdx.x, j = j0 + k;
    if (i < m && j < n) o[pr[i] + (size_t)pc[j] * Ma] = t[threadIdx.x][k];
  }
}

// out_b = (upper triangle of R_b)^H, n x n column-major
__global__ void k_svd_adjoint(const double2* R, int n, double2* out) {
  __shared__ double2 t[TT][TT + 1];
  const size_t base = (size_t)blockIdx.z * n * n;
  const int r0 = blockIdx.x * TT, c0 = blockIdx.y * TT;
  for (int k = threadIdx.y; k < TT; k += 8) {
    const int r = r0 + threadIdx.x, c = c0 + k;
    t[k][threadIdx.x] = r < n && c < n && r <= c ? R[base + r + (size_t)c * n] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int k = threadIdx.y; k < TT; k += 8) {
    const int r = r0 + k, c = c0 + threadIdx.x;
    if (r < n && c < n) out[base + c + (size_t)r * n] = conj2(t[threadIdx.x][k]);
  }
}

// row-major out_b (rows x k) from column-major in_b: out[i, c] = in[pos[i], c]
__global__ void k_svd_rows(const double2* in, int rows, int k, const int* pos, double2* out) {
  __shared__ double2 t[TT][TT + 1];
  const int b = blockIdx.z;
  const int i0 = blockIdx.x * TT, c0 = blockIdx.y * TT;
  for (int q = threadIdx.y; q < TT; q += 8) {
    const int i = i0 + threadIdx.x, c = c0 + q;
    if (i < rows && c < k)
      t[q][threadIdx.x] = in[((size_t)b * k + c) * rows + pos[(size_t)b * rows + i]];
  }
  __syncthreads();
  for (int q = threadIdx.y; q < TT; q += 8) {
    const int i = i0 + q, c = c0 + threadIdx.x;
    if (i < rows && c < k) out[((size_t)b * rows + i) * k + c] = t[threadIdx.x][q];
  }
}

__global__ void k_svd_sigma(const double* sig, const int* perm, int Na, int batch, double* out) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < Na * batch) out[idx] = sig[(size_t)(idx / Na) * Na + perm[idx]];
}

int cdiv(int a, int b) { return (a + b - 1) / b; }

}  // namespace

size_t svd_qr_layout(int Ma, int Na, int batch, SvdQr* out, char* base) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    char* r = base ? base + o : nullptr;
    o += (bytes + 255) & ~size_t(255);
    return r;
  };
  const size_t nn = sizeof(double2) * (size_t)Na * Na * batch, nb = batch;
  SvdQr s{};
  s.Y = (double2*)take(sizeof(double2) * (size_t)Ma * Na * nb);
  s.T = (double2*)take(nn);
  s.M = (double2*)take(nn);
  s.Vp = (double2*)take(nn);
  s.tau = (double*)take(sizeof(double) * Na * nb);
  s.nrm = (double*)take(sizeof(double) * Ma * nb);
  s.pcol = (int*)take(sizeof(int) * Na * nb);
  s.prow = (int*)take(sizeof(int) * Ma * nb);
  s.qr = (QRItem*)take(sizeof(QRItem) * 2 * nb);
  s.blk = (QRBlk*)take(sizeof(QRBlk) * nb);
  s.mul = (ZGemmItem*)take(sizeof(ZGemmItem) * 2 * nb);
  s.ops = (ZGemmItem*)take(sizeof(ZGemmItem) * qr_block_ops(batch, Na));
  s.per_blk = qr_block_bytes(Ma, Na, nullptr, nullptr);
  s.blk_ws = take(s.per_blk * nb);
  s.per_a = zgemm9_pack_bytes(Ma, Na, 0);
  s.per_b = zgemm9_pack_bytes(Na, Na, 1);
  s.pack = (unsigned char*)take(2 * nb * (s.per_a + s.per_b));
  if (out) *out = s;
  return o;
}

// From 96 columns on, or from 32 where the matrix is at least four times as long; the blocked QR's panel has to fit and
// the two products of every matrix have to go into one launch. Measured with the direct call beside it, singular values
// over four decades: 96 x 96 4.0 against 5.5 ms, four 128 x 128 6.2 / 8.7, 256 x 256 14.8 / 24.7, two 256 x 64 2.7 / 4.6,
// two 1000 x 40 2.0 / 4.5 (64 x 64 gained a fifth with QRs of 2.9 ms). With random entries and columns graded over four
// decades the Jacobi alone is quick as well: 96 x 96 4.0 / 3.0, ten 160 x 160 10.2 / 10.3, two 256 x 256 14.3 / 13.9; a
// line further down would lose more there than a bond's matrix gains.
bool svd_qr_shape(int Ma, int Na, int batch) {
  return (Na >= 96 || (Na >= 32 && Ma / 4 >= Na)) && 2LL * batch <= zgemm_max_items() && Ma <= QR_BLOCK_MAX_ROWS;
}

bool svd_qr_fits(int Ma, int Na, int batch) {
  return svd_qr_shape(Ma, Na, batch) && qr_block_cluster(batch, Ma) > 0 && qr_block_cluster(batch, Na) > 0;
}

void launch_svd_qr(const double2* A, int m, int n, int batch, const BondWork* items, double2* wA, double2* wV,
                   double* sig, int* perm, const SvdQr& s, SvdQrHost* h, int max_sweeps, int* status,
                   unsigned* sync3, double* sigma, double2* U, double2* V, cudaStream_t st) {
  const bool tr = m < n;
  const int Ma = std::max(m, n), Na = std::min(m, n);
  const size_t sA = (size_t)Ma * Na, sV = (size_t)Na * Na;
  h->qr.resize(2 * (size_t)batch);
  h->blk.resize(batch);
  h->mul.assign(2 * (size_t)batch, ZGemmItem{});
  for (int b = 0; b < batch; ++b) {
    h->qr[b] = QRItem{wA + b * sA, s.Y + b * sA, s.T + b * sV, s.tau + (size_t)b * Na, Ma, Na};
    h->qr[batch + b] = QRItem{s.M + b * sV, s.Y + b * sV, wV + b * sV, s.tau + (size_t)b * Na, Na, Na};
    qr_block_bytes(Ma, Na, &h->blk[b], s.blk_ws + (size_t)b * s.per_blk);
    for (int k = 0; k < 2; ++k) {          // U' = Q1 W and V' = Q2 Z, columns by falling singular value
      ZGemmItem it{};
      const int rows = k == 0 ? Ma : Na;
      it.A = k == 0 ? wA + b * sA : s.M + b * sV;
      it.B = k == 0 ? s.T + b * sV : wV + b * sV;
      it.C = k == 0 ? s.Y + b * sA : s.Vp + b * sV;
      it.lda = it.ldc = rows;
      it.ldb = Na;
      it.M = rows;
      it.N = it.K = Na;
      it.bcol = perm + (size_t)b * Na;
      it.TA = s.pack + (2 * (size_t)b + k) * (s.per_a + s.per_b);
      it.TB = it.TA + s.per_a;
      it.cap_m = rows;
      it.cap_n = it.cap_k = Na;
      h->mul[2 * b + k] = it;
    }
  }
  cudaMemcpyAsync(s.qr, h->qr.data(), sizeof(QRItem) * h->qr.size(), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(s.blk, h->blk.data(), sizeof(QRBlk) * h->blk.size(), cudaMemcpyHostToDevice, st);
  cudaMemcpyAsync(s.mul, h->mul.data(), sizeof(ZGemmItem) * h->mul.size(), cudaMemcpyHostToDevice, st);
  const dim3 th(TT, 8);
  auto rank = [&](bool rows_of_a, int len, int* pos) {
    k_svd_norms<<<dim3(rows_of_a ? cdiv(len, 8) : cdiv(len, TT), batch), th, 0, st>>>(A, m, n, rows_of_a, s.nrm);
    k_svd_rank<<<cdiv(len * batch, 128), 128, 0, st>>>(s.nrm, len, batch, pos);
  };
  rank(tr, Na, s.pcol);
  rank(!tr, Ma, s.prow);
  k_svd_load_sorted<<<dim3(cdiv(n, TT), cdiv(m, TT), batch), th, 0, st>>>(A, m, n, tr, s.prow, s.pcol, wA);
  auto qr = [&](const QRItem* list, int rows) {
    if (qr_small_fits(rows, Na)) {
      launch_qr_small(list, batch, rows, Na, status, st);
      return;
    }
    QRBlkList L;
    L.blk = s.blk;
    L.ops = s.ops;
    L.n_items = batch;
    L.m_cap = rows;
    L.n_cap = Na;
    L.cluster = qr_block_cluster(batch, rows);
    launch_qr_block(Tables{}, nullptr, list, L, status, st);
  };
  const dim3 nn(cdiv(Na, TT), cdiv(Na, TT), batch);
  qr(s.qr, Ma);
  k_svd_adjoint<<<nn, th, 0, st>>>(s.T, Na, s.M);
  qr(s.qr + batch, Na);
  k_svd_adjoint<<<nn, th, 0, st>>>(wV, Na, s.T);
  launch_svd_jacobi(items, batch, Na, Na, max_sweeps, status, sync3, st);
  const long long tiles = ((long long)cdiv(Ma, 128) + cdiv(Na, 128)) * cdiv(Na, 32) * batch;
  launch_zgemm9(s.mul, 2 * batch, tiles, Ma, Na, Na, status, st);
  k_svd_sigma<<<cdiv(Na * batch, 128), 128, 0, st>>>(sig, perm, Na, batch, sigma);
  k_svd_rows<<<dim3(cdiv(Ma, TT), cdiv(Na, TT), batch), th, 0, st>>>(s.Y, Ma, Na, s.prow, tr ? V : U);
  k_svd_rows<<<nn, th, 0, st>>>(s.Vp, Na, Na, s.pcol, tr ? U : V);
}

}  // namespace ptk
