// QR-preconditioned one-sided Jacobi for the bond SVD (App. A.2).
//
// A one-sided Jacobi on a rank-deficient, strongly graded D needs many sweeps (17-23 on the
// five-site chain's 256x256 blocks); after a column-pivoted QR, D P = Q R, the same Jacobi on R^H
// converges in ~8 (Drmac and Veselic's preconditioning). Here:
//   1. the pivoted Householder QR of D, with B = R^H written directly: one thread-block cluster per matrix, the
//      columns in shared memory, or in global memory where a matrix's share does not fit (k_qrcp_cl);
//   2. the grid Jacobi on B gives B = U' S V'^H, i.e. R = V' S U'^H and D = (Q V') S (P U')^H;
//   3. after the truncation, k_qrcp_vd: V_D = P U' (rows permuted back) on the kept columns;
//   4. U_D = D V_D S^{-1} on the kept columns by an FP64 GEMM (k_mix_gemm) and a column scaling
//      (k_qrcp_ud). Its error in column c is ~eps ||D|| / s_c, and that column enters the truncated
//      state scaled by s_c, so the state error stays at rounding level; Q is never formed.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "kernels.h"

namespace cg = cooperative_groups;

namespace ptk {

namespace {

__device__ __forceinline__ void shape(const BondWork& W, int* Ma, int* Na) {
  const int mD = W.info[0], nD = W.info[1];
  const bool tr = W.info[2] != 0;
  *Ma = (mD > 0 && nD > 0) ? (tr ? nD : mD) : 0;
  *Na = (mD > 0 && nD > 0) ? (tr ? mD : nD) : 0;
}

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

constexpr int QR_CW = 16;                 // column warps; one more warp computes the reflector's scalars
constexpr int QR_THREADS = 32 * (QR_CW + 1);
constexpr int QR_MAX_C = 16;

// a CTA's best remaining column, pushed to every CTA of the cluster: its norm's bits + 1 (0: none left; a NaN counts as
// zero), exact squared norm, entry in row j, storage index
struct QrCand {
  unsigned long long key;
  double nrm2;
  double2 alpha;
  int idx, pad[3];
};

__device__ __forceinline__ unsigned long long qr_key(double v) {
  return v >= 0.0 ? (unsigned long long)__double_as_longlong(v) + 1 : 1;
}

// the lane with the largest key (smallest idx on ties) among the warp
__device__ __forceinline__ int qr_best(unsigned long long key, int idx) {
  const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  const bool in = hi == mh && lo == ml;
  const unsigned mi = __reduce_min_sync(0xffffffffu, in ? (unsigned)idx : 0xffffffffu);
  return __ffs(__ballot_sync(0xffffffffu, in && (unsigned)idx == mi)) - 1;
}

__host__ __device__ __forceinline__ size_t qr_head_bytes(int lq, int m_cap, int n_cap) {
  const size_t b = sizeof(double2) * (size_t)m_cap + sizeof(double) * (size_t)lq + sizeof(int) * 2 * ((size_t)n_cap + lq);
  return (b + 15) & ~size_t(15);
}

// The factorisation with one thread-block cluster per matrix. Storage column s belongs to CTA s % C at local index
// s / C; GL = false keeps the columns in the CTAs' shared memory (pivot columns read through distributed shared
// memory), GL = true in the workspace Y64 (through L2). Pivoting is logical: the pivot column is not moved, its position
// is recorded (qp[j] = p), so R[i, j] is row i of storage column qp[j] (i < j), and R[j, j] = beta is put in its row j.
//
// What bounds it: the latency of one step, and the FP64 pipe, which takes 64 cycles of a sub-partition per instruction
// of a warp whatever its lanes. So per step:
//   * one cluster barrier: every CTA pushes its candidate (QrCand) to all others before it;
//   * every warp picks the pivot from the C candidates by itself, in integer instructions;
//   * the reflector's scalars (square root and reciprocals, ~1400 cycles) follow from the candidate alone, so one extra
//     warp forms them while the others fetch the pivot column x and form s_k = sum_{r > j} conj(x_r) a_rk;
//   * a column is shared by L = 4 .. 32 lanes, few columns' lanes to a warp where there are many columns (fewer
//     reduction steps) and whole warps where there are few (step_lanes below). The same lanes then update it:
//     a <- a - v kappa (s_k + conj(v_j) a_jk), and form its exact norm over the rows that remain, which the next
//     pivot and its reflector use: no downdating, and no second sum over the pivot column;
//   * finished columns leave the list of active ones, so lanes stay busy.
// Before (one warp per column with a butterfly each, the pivot's norm and scalars after the barrier on one thread, ~9000
// cycles a step; a second kernel spread a layer's columns over the whole GPU with a grid barrier per step) -> now: all
// pivoted QRs of the five-site chain's first eight steps 44 -> 26 ms (136 x 136 now 6.9 us a step, 64 x 64 5.0, 256 x
// 256 10.1 against 13.4), the three-site chain's 8 -> 6 ms, the 16 chains' first four steps 62 -> 17 ms, of that the most
// by clusters sized by the number of matrices (qr_pick_cluster).
// Rank-revealing stop: the factorisation ends at the first step j whose pivot column (the largest remaining one) has
// an exact norm^2 <= tau^2 ||D||_F^2, with tau the noise level of D: u = 2^-53 when D was formed in FP64 (the level
// below which the Jacobi does not rotate a column either), 2^-40 for the fixed-point-slice tensor-core product (whose
// error in D's null space is ~3e-14 of ||D||_F). Every remaining column is then noise, and the trailing block R22 they
// form, ||R22||_F <= sqrt(n) tau ||D||_F, is dropped -- for tau = u a perturbation within the backward error of any
// FP64 SVD, for 2^-40 one far below every truncation threshold (>= 1e-10 sigma_1). R is then k x n (k = j, recorded in
// info[8]) and B = R^H is n x k, so the Jacobi runs on k columns. (The workloads' D are often exactly rank deficient: a
// conserved magnetisation leaves ~n/4 nonzero singular values.)
template <bool GL>
__device__ __forceinline__ void qrcp_run(const BondWork& W, int Ma, int Na, int C, int rank, double2* X, int x_ld,
                                         double2* hv, double* nrm, int* act, int* apos, int* qp, int* pos, double tau2,
                                         int kmax) {
  cg::cluster_group cl = cg::this_cluster();
  __shared__ QrCand s_cand[2][QR_MAX_C];
  __shared__ double2 s_vj, s_beta;
  __shared__ double s_kap, s_fro, s_red[QR_CW + 1];
  __shared__ int s_na;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int Ln = rank < Na ? (Na - rank + C - 1) / C : 0;
  auto colp = [&](int l) -> double2* {
    return GL ? W.Y64 + (size_t)(rank + l * C) * Ma : X + (size_t)l * x_ld;
  };
  auto ld = [](const double2* q) -> double2 { return GL ? __ldcg(q) : *q; };
  auto st = [](double2* q, double2 v) {
    if (GL) __stcg(q, v);
    else *q = v;
  };
  // the own columns and their norms
  {
    double fro = 0;
    for (int l = wid; l < Ln; l += QR_CW + 1) {
      double sq = 0;
      double2* a = colp(l);
      const double2* from = W.A + (size_t)(rank + l * C) * Ma;
      for (int r = lane; r < Ma; r += 32) {
        const double2 v = from[r];
        st(a + r, v);
        sq = fma(v.x, v.x, fma(v.y, v.y, sq));
      }
      sq = wsum(sq);
      fro += sq;
      if (lane == 0) {
        nrm[l] = sq;
        act[l] = l;
        apos[l] = l;
      }
    }
    if (lane == 0) s_red[wid] = fro;
    if (tid == 0) s_na = Ln;
  }
  __syncthreads();
  if (tid == 0) {
    double f = 0;
    for (int k = 0; k <= QR_CW; ++k) f += s_red[k];
    s_fro = f;
  }
  // warp 0: the best active column, its entry in row j, to every CTA's slot par
  auto publish = [&](int par, int na, int j) {
    unsigned long long key = 0;
    int bl = -1;
    for (int i = lane; i < na; i += 32) {
      const int l = act[i];
      const unsigned long long k = qr_key(nrm[l]);
      if (k > key || (k == key && (unsigned)l < (unsigned)bl)) {
        key = k;
        bl = l;
      }
    }
    const int src = qr_best(key, bl);
    QrCand c{};
    c.key = __shfl_sync(0xffffffffu, key, src);
    const int l = __shfl_sync(0xffffffffu, bl, src);
    c.idx = l >= 0 ? rank + l * C : 0x7fffffff;
    if (l >= 0) {
      c.nrm2 = nrm[l];
      if (j < Ma) c.alpha = ld(colp(l) + j);
    }
    if (lane < C) *cl.map_shared_rank(&s_cand[par][rank], lane) = c;
  };
  cl.sync();                                // every CTA runs: its shared memory may be written
  if (wid == 0) publish(0, Ln, 0);
  cl.sync();
  double thr2;                              // tau^2 ||D||_F^2, the C shares summed in the same order in every CTA
  {
    const double f = lane < C ? *cl.map_shared_rank(&s_fro, lane) : 0.0;
    thr2 = tau2 * wsum(f);
  }
  int kq = Na;
  for (int j = 0; j < Na; ++j) {
    const int par = j & 1;
    // 1. the pivot, picked by every warp
    const QrCand& cand = s_cand[par][lane < C ? lane : 0];
    const int win = qr_best(lane < C ? cand.key : 0, lane < C ? cand.idx : 0x7fffffff);
    const int p = s_cand[par][win].idx, owner = p % C, lp = p / C;
    const double nrm2 = s_cand[par][win].nrm2;
    if (nrm2 <= thr2 || j >= kmax) {        // the same decision in every warp of every CTA
      kq = j;
      break;
    }
    const int na = s_na, rows = Ma - j - 1;
    const int own = rank == owner ? lp : -1;
    // 2. the pivot column's rows below j; the scalars of its reflector
    if (wid < QR_CW) {
      const double2* src = GL ? W.Y64 + (size_t)p * Ma : cl.map_shared_rank(X, owner) + (size_t)lp * x_ld;
      for (int r = j + 1 + tid; r < Ma; r += 32 * QR_CW) hv[r] = ld(src + r);
      asm volatile("bar.sync 1, %0;" ::"r"(32 * QR_CW) : "memory");
    } else {
      // H = I - kappa v v^H with v = x - beta e_j, beta = -phase(alpha) ||x||: v^H v = 2 ||x|| (||x|| + |alpha|), so
      // kappa = 1 / (||x|| (||x|| + |alpha|)), v_j = phase (|alpha| + ||x||). Lane 0: ||x||, lane 1: |alpha|
      const double2 al = s_cand[par][win].alpha;
      const double a2 = fma(al.x, al.x, al.y * al.y), sq = lane == 0 ? nrm2 : a2;
      const double ir = sq == 0.0 ? 0.0 : rsqrt(sq);
      double root = sq * ir;
      root = fma(0.5 * ir, fma(-root, root, sq), root);
      const double xn = __shfl_sync(0xffffffffu, root, 0), aabs = __shfl_sync(0xffffffffu, root, 1);
      const double ix = __shfl_sync(0xffffffffu, ir, 0), ia = __shfl_sync(0xffffffffu, ir, 1);
      const double2 ph = a2 == 0.0 ? make_double2(1.0, 0.0) : make_double2(al.x * ia, al.y * ia);
      const double sum = aabs + xn;
      if (lane == 0) {
        s_kap = nrm2 == 0.0 ? 0.0 : ix / sum;
        s_vj = make_double2(ph.x * sum, ph.y * sum);
        s_beta = nrm2 == 0.0 ? al : make_double2(-ph.x * xn, -ph.y * xn);
        qp[j] = p;
      }
    }
    // 3. the remaining columns: L lanes each
    int L = 32;
    {
      // the instructions of a sub-partition: ten per row and about twelve besides, three per reduction step
      int best = 0x7fffffff;
#pragma unroll
      for (int lg = GL ? 4 : 2; lg <= 5; ++lg) {          // from L2 in runs of 256 bytes or more
        const int warps = ((((na << lg) + 31) >> 5) + 3) >> 2;
        const int cost = warps * (10 * ((rows + (1 << lg) - 1) >> lg) + 3 * lg + 12);
        if (cost < best) {
          best = cost;
          L = 1 << lg;
        }
      }
    }
    const int ln = lane & (L - 1), per = 32 / L, groups = QR_CW * per;
    bool first = true;
    double kap = 0;
    double2 vj = make_double2(0.0, 0.0);
    // group g takes active columns g, g + groups, ...; the loop is uniform in the warp
    for (int i0 = wid < QR_CW ? wid * per : na; i0 < na || first; i0 += groups) {
      const int i = i0 + lane / L;
      const int l = wid < QR_CW && i < na ? act[i] : -1;
      const bool on = l >= 0 && l != own;
      double2* a = on ? colp(l) : nullptr;
      double sr = 0, si = 0;
      if (on) {
        int r = j + 1 + ln;
        for (; r + 3 * L < Ma; r += 4 * L) {      // four rows' loads in flight
          double2 v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) v[q] = ld(a + r + q * L);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const double2 u = hv[r + q * L];
            sr = fma(u.x, v[q].x, fma(u.y, v[q].y, sr));
            si = fma(u.x, v[q].y, fma(-u.y, v[q].x, si));
          }
        }
        for (; r < Ma; r += L) {
          const double2 u = hv[r], v = ld(a + r);
          sr = fma(u.x, v.x, fma(u.y, v.y, sr));
          si = fma(u.x, v.y, fma(-u.y, v.x, si));
        }
      }
      // real parts to the lower half of the group, imaginary parts to the upper, then both to all
      const bool up = ln >= (L >> 1);
      double s = (up ? si : sr) + __shfl_xor_sync(0xffffffffu, up ? sr : si, L >> 1);
      for (int o = L >> 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const double other = __shfl_xor_sync(0xffffffffu, s, L >> 1);
      sr = up ? other : s;
      si = up ? s : other;
      if (first) {
        __syncthreads();
        first = false;
        kap = s_kap;
        vj = s_vj;
      }
      double nn = 0;
      double2 aj = make_double2(0.0, 0.0);
      if (on) {
        aj = ld(a + j);
        const double wr = fma(vj.x, aj.x, fma(vj.y, aj.y, sr)), wi = fma(vj.x, aj.y, fma(-vj.y, aj.x, si));
        const double tr = kap * wr, ti = kap * wi;
        int r = j + 1 + ln;
        for (; r + 3 * L < Ma; r += 4 * L) {
          double2 v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) v[q] = ld(a + r + q * L);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const double2 u = hv[r + q * L];
            v[q].x = fma(-u.x, tr, fma(u.y, ti, v[q].x));
            v[q].y = fma(-u.x, ti, fma(-u.y, tr, v[q].y));
            st(a + r + q * L, v[q]);
            nn = fma(v[q].x, v[q].x, fma(v[q].y, v[q].y, nn));
          }
        }
        for (; r < Ma; r += L) {
          const double2 u = hv[r];
          double2 v = ld(a + r);
          v.x = fma(-u.x, tr, fma(u.y, ti, v.x));
          v.y = fma(-u.x, ti, fma(-u.y, tr, v.y));
          st(a + r, v);
          nn = fma(v.x, v.x, fma(v.y, v.y, nn));
        }
        aj.x = fma(-vj.x, tr, fma(vj.y, ti, aj.x));
        aj.y = fma(-vj.x, ti, fma(-vj.y, tr, aj.y));
      }
      for (int o = L >> 1; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
      if (on && ln == 0) {                  // all lanes of the group have read row j
        st(a + j, aj);
        nrm[l] = nn;
      }
    }
    __syncthreads();
    if (wid == 0) {
      int left = na;
      if (own >= 0) {                       // the pivot column: R's diagonal entry, out of the list
        --left;
        if (lane == 0) {
          st(colp(own) + j, s_beta);
          const int i = apos[own], last = act[left];
          act[i] = last;
          apos[last] = i;
          s_na = left;
        }
        __syncwarp();
      }
      publish(par ^ 1, left, j + 1);
    }
    cl.sync();                              // candidates published; pivot column reads done
  }
  // permutation (every CTA holds the same qp): the k pivots in order, then the remaining columns by index; B = R^H
  // (Na x k) rows of the own columns
  __syncthreads();
  for (int j = tid; j < Na; j += blockDim.x) pos[j] = -1;
  __syncthreads();
  for (int j = tid; j < kq; j += blockDim.x) pos[qp[j]] = j;
  __syncthreads();
  if (wid == 0) {
    int i = kq;
    for (int s0 = 0; s0 < Na; s0 += 32) {
      const int s = s0 + lane;
      const bool rem = s < Na && pos[s] < 0;
      const unsigned bal = __ballot_sync(0xffffffffu, rem);
      if (rem) {
        const int at = i + __popc(bal & ((1u << lane) - 1u));
        pos[s] = at;
        qp[at] = s;
      }
      i += __popc(bal);
    }
  }
  __syncthreads();
  if (rank == 0) {
    for (int j = tid; j < Na; j += blockDim.x) W.qperm[j] = qp[j];
    if (tid == 0) W.info[8] = kq;
  }
  for (int l = wid; l < Ln; l += QR_CW + 1) {
    const int s = rank + l * C, i = pos[s];
    const double2* a = colp(l);
    for (int c = lane; c < kq; c += 32) {
      double2 v = make_double2(0.0, 0.0);           // B[i, c] = conj(R[c, i])
      if (c <= i) {
        const double2 x = ld(a + c);
        v = make_double2(x.x, -x.y);
      }
      W.G64[i + (size_t)c * Na] = v;
    }
  }
  cl.sync();                                      // no CTA leaves while its memory may be read
}

}  // namespace

// Dynamic shared memory: hv[m_cap] (double2), nrm[lq_cap] (double), qp[n_cap] | pos[n_cap] | act[lq_cap] |
// apos[lq_cap] (int, to a multiple of 16 bytes), then x_elems entries of columns: a matrix whose share does not fit
// them stays in global memory.
__global__ void __launch_bounds__(QR_THREADS, 1)
    k_qrcp_cl(const BondWork* work, int n_work, int lq_cap, int m_cap, int n_cap, int x_elems, double tau2, int kmax,
              int* status) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int w = blockIdx.x / C;
  if (w >= n_work) return;                        // uniform across the cluster
  const BondWork& W = work[w];
  int Ma, Na;
  shape(W, &Ma, &Na);
  if (Na <= 0) return;
  const int lq = (Na + C - 1) / C;
  if (Ma > m_cap || Na > n_cap || lq > lq_cap || Ma < Na) {
    if (rank == 0 && threadIdx.x == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  extern __shared__ double2 sm[];
  double2* hv = sm;
  double* nrm = (double*)(hv + m_cap);
  int* qp = (int*)(nrm + lq_cap);
  int *pos = qp + n_cap, *act = pos + n_cap, *apos = act + lq_cap;
  double2* X = sm + qr_head_bytes(lq_cap, m_cap, n_cap) / sizeof(double2);
  if ((long long)lq * Ma <= x_elems)
    qrcp_run<false>(W, Ma, Na, C, rank, X, Ma, hv, nrm, act, apos, qp, pos, tau2, kmax);
  else
    qrcp_run<true>(W, Ma, Na, C, rank, X, Ma, hv, nrm, act, apos, qp, pos, tau2, kmax);
}

// The finish forms only the columns the truncation keeps (it runs after k_truncate): kept column c
// is Jacobi column perm[c], c < chi = the bond's new dimension.
// V_D = P U' on the kept columns: V[qperm[r], perm[c]] = U'[r, perm[c]] (U' = the normalised columns
// of B after the Jacobi)
__global__ void k_qrcp_vd(const BondWork* work, int n_work, const int* lam_chi) {
  const int w = blockIdx.y;
  if (w >= n_work) return;
  const BondWork& W = work[w];
  int Ma, Na;
  shape(W, &Ma, &Na);
  const int kept = min(lam_chi[W.lam_l + 1], Na);
  const size_t tot = (size_t)Na * kept;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < tot; idx += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(idx % Na), col = W.perm[idx / Na];
    W.V[W.qperm[r] + (size_t)col * Na] = W.G64[r + (size_t)col * Na];
  }
}

// U_D = (D V_D) / sigma on the kept columns (Y64 holds D V_D in kept order)
__global__ void k_qrcp_ud(const BondWork* work, int n_work, const int* lam_chi) {
  const int w = blockIdx.y;
  if (w >= n_work) return;
  const BondWork& W = work[w];
  int Ma, Na;
  shape(W, &Ma, &Na);
  const int kept = min(lam_chi[W.lam_l + 1], Na);
  const size_t tot = (size_t)Ma * kept;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < tot; idx += (size_t)gridDim.x * blockDim.x) {
    const int col = W.perm[idx / Ma];
    const double s = W.sig[col];
    const double2 y = W.Y64[idx];
    W.A[idx % Ma + (size_t)col * Ma] = s > 0.0 ? make_double2(y.x / s, y.y / s) : make_double2(0.0, 0.0);
  }
}

namespace {

constexpr int QR_SMEM = 208 * 1024;          // 227 KB less the static arrays
constexpr int QR_MAX_DEV = 64;
struct QrClusters {
  std::once_flag once;                       // filled by one thread while the others wait
  int active[QR_MAX_C + 1] = {};             // clusters of c CTAs the device holds at once
};
QrClusters g_qr_tab[QR_MAX_DEV];

cudaLaunchConfig_t qr_cfg(int n_work, int cluster, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_work * cluster, 1, 1);
  cfg.blockDim = dim3(QR_THREADS, 1, 1);
  cfg.dynamicSmemBytes = QR_SMEM;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

const QrClusters& qr_clusters() {
  int dev = 0;
  cudaGetDevice(&dev);
  QrClusters& t = g_qr_tab[std::max(0, std::min(dev, QR_MAX_DEV - 1))];
  std::call_once(t.once, [&t] {
    cudaFuncSetAttribute(k_qrcp_cl, cudaFuncAttributeMaxDynamicSharedMemorySize, QR_SMEM);
    cudaFuncSetAttribute(k_qrcp_cl, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int c = 1; c <= QR_MAX_C; ++c) {
      cudaLaunchAttribute at[1];
      cudaLaunchConfig_t cfg = qr_cfg(1, c, 0, at);
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_qrcp_cl, &cfg) == cudaSuccess) t.active[c] = n;
      cudaGetLastError();
    }
  });
  return t;
}

// entries of columns that a CTA's shared memory holds beside its other arrays; < 0: not even those fit
long long qr_x_elems(int c, int m_cap, int n_cap) {
  const long long head = (long long)qr_head_bytes((n_cap + c - 1) / c, m_cap, n_cap);
  return head > QR_SMEM ? -1 : (QR_SMEM - head) / (long long)sizeof(double2);
}

// CTAs per matrix for n_work matrices: the shortest estimate of a step, the waves of clusters times (4000 cycles of
// latency + the arithmetic of a third of a matrix of half the capacities, ten instructions of 19 cycles per 32 entries,
// over the cluster), for matrices of equal size and for a quarter of them large (a correlation front): the waves of both
// are added. Equal sizes alone took 10 CTAs for a layer of ten with two of 592 x 592 (280000 cycles a step). Whether a
// matrix stays in shared memory is seen on the device from its live size.
int qr_pick_cluster(int n_work, int m_cap, int n_cap) {
  const QrClusters& t = qr_clusters();
  int best = 0;
  double cost = 1e300;
  for (int c = 1; c <= QR_MAX_C; ++c) {
    if (t.active[c] <= 0 || qr_x_elems(c, m_cap, n_cap) < 0) continue;
    const int quarter = (n_work + 3) / 4;
    const double v = (double)((n_work + t.active[c] - 1) / t.active[c] + (quarter + t.active[c] - 1) / t.active[c]) *
                     (4000.0 + 19.0 * 10.0 / 32.0 / 3.0 * (0.5 * n_cap) * (0.5 * m_cap) / c);
    if (v < cost) {
      cost = v;
      best = c;
    }
  }
  return best;
}

}  // namespace

// Cluster size for the shared-memory factorisation of matrices up to m_cap x n_cap; 0 if they do
// not fit (the columns then stay in global memory).
int qrcp_smem_cluster(int m_cap, int n_cap) {
  for (int c = QR_MAX_C; c >= 2; c >>= 1)
    if (qr_clusters().active[c] > 0 && (long long)((n_cap + c - 1) / c) * m_cap <= qr_x_elems(c, m_cap, n_cap)) return c;
  return 0;
}

void launch_qrcp_precondition(const BondWork* work, int n_work, int cluster, int k_cap, int m_cap, double tau2,
                              int kmax, int* status, cudaStream_t st) {
  const int c = cluster > 0 ? cluster : std::max(1, qr_pick_cluster(n_work, m_cap, k_cap));
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t cfg = qr_cfg(n_work, c, st, at);
  // arrays beyond a CTA's shared memory: the launch fails
  cfg.dynamicSmemBytes = std::max((size_t)QR_SMEM, qr_head_bytes((k_cap + c - 1) / c, m_cap, k_cap));
  cudaLaunchKernelEx(&cfg, k_qrcp_cl, work, n_work, (k_cap + c - 1) / c, m_cap, k_cap,
                     (int)std::max(0LL, qr_x_elems(c, m_cap, k_cap)), tau2, kmax, status);
}

void launch_qrcp_finish(const BondWork* work, int n_work, int k_cap, int m_cap, const int* lam_chi,
                        cudaStream_t st) {
  k_qrcp_vd<<<dim3(128, n_work), 256, 0, st>>>(work, n_work, lam_chi);
  launch_mix_gemm_av(work, n_work, k_cap, m_cap, lam_chi, st);
  k_qrcp_ud<<<dim3(128, n_work), 256, 0, st>>>(work, n_work, lam_chi);
}

}  // namespace ptk
