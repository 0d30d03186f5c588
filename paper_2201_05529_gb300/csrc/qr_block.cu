// Blocked Householder QR with the explicit Q for a list of matrices: the outer blocks of a bond layer (App. A.2's exact
// reductions) and the sketches of the fast path's range finder (rsvd.cu).
//
// What bounds a QR here: GB300's FP64 pipe (1.0 TFLOP/s) and, column by column, the latency of one reflector. The
// unblocked factorisation (hqr_grid.cu) pays a grid barrier and two passes of a warp over a whole column per
// reflector and does every operation on the FP64 pipe (ten 1120 x 160: 10.6 ms, twenty 2048 x 512: 224 ms). Here
//   * panels of 32 columns are factored by one thread-block cluster per matrix, the panel's rows split over the CTAs
//     and held in shared memory: per reflector one exchange of the partial inner products x^H a_k through
//     distributed shared memory and one cluster barrier (k_qr_panel);
//   * everything outside the panels runs on the tensor cores, as products of nine exact BF16 slices with 64-bit integer
//     sums (tc_zgemm.cu, Z9), whose error is at the level of an FP64 product's own rounding:
//       forward,  panel p:  W = A2^H V_p, S = V_p^H V_p;  X = W T;    A2 <- A2 - V_p X^H
//       backward, panel p:  W = Q2^H V_p;                 X = W T^H;  Q2 <- Q2 - V_p X^H
//     (P_1 ... P_32 = I - V T V^H with T^-1 = striu(S) + diag(1 / tau): X comes from a triangular solve with S, k_qr_wt;
//     A2 the columns right of the panel, Q2 the columns from the panel on, [I; 0] at the start).
// K = m is long and the product W small, so its K chunks are separate units of work whose parts k_qr_wt adds in order.
//
// Reflectors P_j = I - tau_j u_j u_j^H with u_j[j] = 1, the diagonal of R = -phase(alpha_j) ||x_j||, as in hqr_grid.cu;
// H receives the columns u_j with their zeros and ones.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "kernels.h"

namespace cg = cooperative_groups;

namespace ptk {

namespace {

constexpr int NB = 32;                     // panel width
constexpr int PT = 512;                    // threads of a panel CTA
constexpr int PW = PT / 32;
constexpr int PANEL_T = PT + 32;           // and a warp for the scalars
constexpr int SMALL_N = 32;                // columns of a matrix that one CTA factors whole
constexpr int MAX_C = 16;                  // CTAs per cluster
constexpr int PANEL_SMEM = 200 * 1024;     // panel rows of one CTA (227 KB less the exchange buffers)
static_assert(QR_BLOCK_MAX_ROWS == MAX_C * (PANEL_SMEM / (NB * (int)sizeof(double2))), "rows of the largest cluster");
constexpr int MAX_PARTS = 16;               // K chunks of a product W, unless chunks of the longest kind are more
constexpr int WT_ROWS = 8;                 // rows of W per block of k_qr_wt, one warp each

// lane 0 ends with the total of a, lane 16 with the total of b
__device__ __forceinline__ double wsum2(double a, double b, int lane) {
  const bool hi = (lane & 16) != 0;
  double keep = hi ? b : a;
  keep += __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, o);
  return keep;
}

// sums of a and b over the L lanes of a group (half: the upper half of it), in every lane
__device__ __forceinline__ double2 group_sum(double a, double b, int L, bool half) {
  double s = (half ? b : a) + __shfl_xor_sync(0xffffffffu, half ? a : b, L >> 1);
  for (int o = L >> 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const double other = __shfl_xor_sync(0xffffffffu, s, L >> 1);
  return half ? make_double2(other, s) : make_double2(s, other);
}

// 1 where 1 / (nrm sum), sum = |alpha| + nrm, has no FP64 value (||x||^2 below 2^-1024; its factors have one), as the trip count
// of a loop around the rare arithmetic (behind a short if the compiler issues it always, 64 cycles an instruction).
__device__ __forceinline__ int no_value(double ti) {
  int n = __double2hiint(ti) >= 0x7ff00000;
  asm("" : "+r"(n));
  return n;
}

// Length of the K chunks of W = A^H V (steps of 16) for n_items products of `cols` rows: the shortest estimate, waves of
// units over the SMs times (steps + 2.5 for a unit's start and epilogue). 256-long chunks alone leave few units for few
// matrices and a second, nearly empty wave for others (160 units of ten 2048 x 160 on 152 SMs): two 256 x 256 QRs 2.54 ->
// 2.36 ms, ten 1120 x 160 3.22 -> 3.05, the 21-site chain's first four steps 410 -> 388.
__device__ __forceinline__ int split_steps(int n_items, int cols, int k, int sms) {
  const int ks = (k + 15) / 16, tiles = n_items * ((cols + 127) / 128);
  int best = Z9_KSTEPS;
  float cost = 3e38f;
  for (int c = Z9_KSTEPS; c >= 1; --c) {
    const int parts = (ks + c - 1) / c;
    if (parts > MAX_PARTS && c < Z9_KSTEPS) break;
    const float t = (float)((tiles * parts + sms - 1) / sms) * ((float)min(c, ks) + 2.5f);
    if (t < cost) {
      cost = t;
      best = c;
    }
  }
  return best;
}

__device__ __forceinline__ bool live(const QRItem& q) { return q.m > 0 && q.n > 0 && q.n <= q.m; }

}  // namespace

// live shapes of this call (from a list, or the outer blocks of a layer's bonds) and the products of every panel:
// one thread per (matrix, panel). ops: per panel n each of forward W and S (one product: the rows of [A2, V_p]^H V_p),
// forward update, backward W, backward update.
__global__ void k_qrb_plan(Tables T, const BondWork* work, const QRItem* list, QRBlk* blk, int n_items, int panels,
                           ZGemmItem* ops, int sms, int* status) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_items * panels) return;
  const int i = idx % n_items, p = idx / n_items;
  QRBlk& B = blk[i];
  QRItem q{};
  if (list) {
    q = list[i];
  } else {
    const BondWork& W = work[i >> 1];
    const BondDims d = bond_dims(T, W);
    if (bond_fits(d, W)) {
      if ((i & 1) == 0 && d.qrL) q = QRItem{W.QL, W.HH, W.RL, W.aux, d.mL, d.nL};
      if ((i & 1) == 1 && d.lqR) q = QRItem{W.QR, W.HH + (size_t)W.mL_cap * W.nL_cap, W.LR, W.sig, d.nR, d.mR};
    }
  }
  if (!live(q) || q.m > B.m_cap || q.n > B.n_cap) {
    if (live(q) && p == 0) atomicOr(status, ST_CAPACITY);
    q.m = q.n = 0;
  }
  if (p == 0) B.q = q;
  ZGemmItem* o = ops + (size_t)p * 4 * n_items;
  ZGemmItem w{}, u{}, bw{}, bu{};
  const int row0 = p * NB, nc = min(NB, q.n - row0), trail = q.n - row0 - NB, rows = q.m - row0;
  if (nc > 0) {
    const double2* V = q.H + row0 + (size_t)row0 * q.m;
    double2* A0 = q.A + row0 + (size_t)row0 * q.m;
    auto inner = [&](const double2* A, int M) {
      ZGemmItem it{};
      it.A = A;
      it.lda = q.m;
      it.opA = ZOP_C;
      it.B = V;
      it.ldb = q.m;
      it.opB = ZOP_N;
      it.C = B.Wp;
      it.ldc = B.n_cap + NB;
      it.M = M;
      it.N = nc;
      it.K = rows;
      it.TA = B.TA;
      it.TB = B.TB;
      it.cap_m = B.n_cap + NB;
      it.cap_n = NB;
      it.cap_k = B.m_cap;
      it.split = (long long)it.ldc * NB;
      it.split_ks = split_steps(n_items, M, rows, sms);
      return it;
    };
    auto outer = [&](double2* C, int N) {
      ZGemmItem it{};
      it.A = V;
      it.lda = q.m;
      it.opA = ZOP_N;
      it.B = B.X;
      it.ldb = B.n_cap;
      it.opB = ZOP_C;
      it.C = C;
      it.ldc = q.m;
      it.M = rows;
      it.N = N;
      it.K = nc;
      it.TA = B.TA2;
      it.TB = B.TB2;
      it.cap_m = B.m_cap;
      it.cap_n = B.n_cap;
      it.cap_k = NB;
      it.acc = -1;
      return it;
    };
    w = inner(A0 + (size_t)NB * q.m, max(0, trail) + nc);
    w.A2 = V;
    w.a_split = max(0, trail);
    if (trail > 0) u = outer(A0 + (size_t)NB * q.m, trail);
    bw = inner(A0, q.n - row0);
    bu = outer(A0, q.n - row0);
  }
  o[i] = w;
  o[n_items + i] = u;
  o[2 * n_items + i] = bw;
  o[3 * n_items + i] = bu;
}

// Panel p of every matrix: one cluster per matrix. Dynamic shared memory: the CTA's rows of the panel, column-major.
// Per column j: L lanes per column k >= j form s_k = sum_{r > j} conj(x_r) a_k,r (x = column j) and send it, with row j
// from its owner, to every CTA; after the cluster barrier the same lanes add the parts while an extra warp forms the
// reflector's scalars from those of s_j; then they apply w_k = tau u^H a_k to their column. An FP64 instruction takes 64
// cycles of a sub-partition whatever its lanes: so columns share warps where there are many (L = 4 or 8: fewer
// reduction steps than a warp per column has), the scalars' square roots go to two lanes of one instruction and start from
// FP32. Two matrices of 256 rows on 16 CTAs each: 10400 cycles per reflector with one warp for the sums over CTAs and the
// scalars of all columns (which had come down from ~15000 besides the rows' arithmetic, all of it done by every warp for
// its own columns), 7100 so; ten of 1120 rows, mostly the rows' arithmetic, 292 us a panel.
__global__ void __launch_bounds__(PANEL_T, 1) k_qr_panel(const QRBlk* blk, int n_items, int p, int rc_cap, int* status) {
  extern __shared__ __align__(16) double2 s_p[];
  __shared__ double2 s_part[2][MAX_C][NB];
  __shared__ double2 s_row[2][NB];
  __shared__ double2 s_u, s_cr, s_scale[NB];
  __shared__ double s_ti, s_rn, s_inv, s_taus[NB];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), C = (int)cl.num_blocks();
  const int i = blockIdx.x / C;
  const QRItem q = blk[i].q;
  const int row0 = p * NB, nc = min(NB, q.n - row0), rows = q.m - row0;
  if (q.m <= 0 || nc <= 0) return;         // the whole cluster
  const int rc = (rows + C - 1) / C;
  if (rc > rc_cap) {
    if (rank == 0 && threadIdx.x == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int lo = min(rows, rank * rc), mine = min(rows, lo + rc) - lo;
  double2* A = q.A + row0 + (size_t)row0 * q.m;
  for (int k = warp; k < nc; k += PANEL_T / 32)
    for (int r = lane; r < mine; r += 32) s_p[(size_t)k * rc + r] = A[lo + r + (size_t)k * q.m];
  // R above the panel: rows 0 .. row0 - 1 of its columns are final
  for (int idx = rank * PANEL_T + tid; idx < row0 * nc; idx += C * PANEL_T) {
    const int r = idx % row0, k = idx / row0;
    q.R[r + (size_t)(row0 + k) * q.n] = q.A[r + (size_t)(row0 + k) * q.m];
  }
  cl.sync();
  const int grp_rows = min(rc, rows);
  for (int j = 0; j < nc; ++j) {
    const int par = j & 1, own = j / rc, jl = j - lo;          // row j's CTA; row j's local index
    const double2* x = s_p + (size_t)j * rc;
    const int from = max(0, jl + 1);                           // first local row below j
    // lanes per column: the instructions of a sub-partition, eight per row and four per reduction step; the same in
    // every CTA, and so that one pass of the 16 warps takes all columns
    int lg = 5;
    {
      const int nk = nc - j;
      int best = 0x7fffffff;
#pragma unroll
      for (int t = 2; t <= 5; ++t) {
        const int warps = ((((nk << t) + 31) >> 5) + 3) >> 2;
        const int c = warps * (8 * ((grp_rows + (1 << t) - 1) >> t) + 4 * t + 8);
        if (c < best && (nk << t) <= 32 * PW) {
          best = c;
          lg = t;
        }
      }
    }
    const int L = 1 << lg, ln = lane & (L - 1);
    const int k = warp < PW ? j + ((warp * 32 + lane) >> lg) : nc;         // this group's column
    const bool on = k < nc, half = ln >= (L >> 1);
    double2* y = s_p + (size_t)(on ? k : j) * rc;
    if (__any_sync(0xffffffffu, on)) {
      double a0 = 0, b0 = 0;
      if (on) {
        int r = from + ln;
        for (; r + 3 * L < mine; r += 4 * L) {       // one warp may have a sub-partition: four rows' loads at once
          double2 u[4], v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            u[q] = x[r + q * L];
            v[q] = y[r + q * L];
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            a0 = fma(u[q].x, v[q].x, fma(u[q].y, v[q].y, a0));
            b0 = fma(u[q].x, v[q].y, fma(-u[q].y, v[q].x, b0));
          }
        }
        for (; r < mine; r += L) {
          const double2 u = x[r], v = y[r];
          a0 = fma(u.x, v.x, fma(u.y, v.y, a0));
          b0 = fma(u.x, v.y, fma(-u.y, v.x, b0));
        }
      }
      const double2 t = group_sum(a0, b0, L, half);
      if (on) {
        for (int to = ln; to < C; to += L) {
          *cl.map_shared_rank(&s_part[par][rank][k], to) = t;
          if (rank == own) *cl.map_shared_rank(&s_row[par][k], to) = y[jl];
        }
      }
    }
    cl.sync();
    double2 tot = make_double2(0.0, 0.0);
    if (warp == PW) {
      // alpha = row j of column j, nrm = ||x||: u_j = alpha - beta = phase (|alpha| + nrm), 2 / |u|^2 = 1 / (nrm (nrm +
      // |alpha|)): w_k = (conj(phase) a_k,j + s_k / (nrm + |alpha|)) / nrm. Lane 0: alpha, lane 1: x
      double v = lane < C ? s_part[par][lane][j].x : 0.0;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const double2 al = s_row[par][j];
      const double a2 = fma(al.x, al.x, al.y * al.y), n2 = v + a2;
      const double q = lane == 0 ? a2 : n2;
      const double ri = __double_as_longlong(q) == 0 ? 0.0 : inv_sqrt(q);
      double rt = q * ri;
      rt = fma(0.5 * ri, fma(-rt, rt, q), rt);
      const double ra = __shfl_sync(0xffffffffu, ri, 0), rn = __shfl_sync(0xffffffffu, ri, 1);
      const double aabs = __shfl_sync(0xffffffffu, rt, 0), nrm = __shfl_sync(0xffffffffu, rt, 1);
      const bool some = __double_as_longlong(n2) != 0;
      // an instruction of this warp takes 64 cycles whatever its lanes: the phase's two products and the ten at the end
      // go to a lane each
      const double pv = (lane == 0 ? al.x : al.y) * ra;
      double px = __shfl_sync(0xffffffffu, pv, 0), py = __shfl_sync(0xffffffffu, pv, 1);
      if (__double_as_longlong(a2) == 0) {
        px = 1.0;
        py = 0.0;
      }
      const double sum = aabs + nrm, inv = some ? inverse(sum) : 0.0;
      const double f = lane < 2 ? rn : (lane < 4 ? sum : (lane < 6 ? inv : (lane < 8 ? rn : nrm)));
      const double g = lane == 6 ? inv : (lane == 7 ? sum : ((lane & 1) ? py : px));
      double v10 = f * g;
      if (lane == 5 || lane >= 8) v10 = __hiloint2double(__double2hiint(v10) ^ 0x80000000, __double2loint(v10));
      double* dst = lane < 2 ? &s_cr.x + lane                                    // conj(phase) / nrm
                  : lane < 4 ? &s_u.x + (lane - 2)                               // alpha - beta
                  : lane < 6 ? &s_scale[j].x + (lane - 4)                        // 1 / (alpha - beta)
                  : lane == 6 ? &s_ti : lane == 7 ? &s_taus[j]
                  : &s_p[(size_t)j * rc + max(0, jl)].x + (lane - 8);            // beta
      if (lane < 8 || (lane < 10 && rank == own && some)) *dst = v10;
      if (lane == 10) s_rn = rn;
      if (lane == 11) s_inv = inv;
    } else if (__any_sync(0xffffffffu, on && k > j)) {
      // the parts, in the same order in every CTA
      double a0 = 0, b0 = 0;
      if (on)
        for (int c = ln; c < C; c += L) {
          const double2 t = s_part[par][c][k];
          a0 += t.x;
          b0 += t.y;
        }
      tot = group_sum(a0, b0, L, half);
    }
    __syncthreads();
    if (on && k > j) {
      const double2 cr = s_cr, yj = s_row[par][k];
      double ti = s_ti;
#pragma unroll 1
      for (int q = no_value(ti); q > 0; --q) {
        tot.x = s_rn * (s_inv * tot.x);
        tot.y = s_rn * (s_inv * tot.y);
        ti = 1.0;
      }
      const double wx = fma(cr.x, yj.x, fma(cr.y, yj.y, ti * tot.x)), wy = fma(cr.x, yj.y, fma(-cr.y, yj.x, ti * tot.y));
      int r = from + ln;
      for (; r + 3 * L < mine; r += 4 * L) {
        double2 u[4], v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          u[q] = x[r + q * L];
          v[q] = y[r + q * L];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          v[q].x = fma(-u[q].x, wx, fma(u[q].y, wy, v[q].x));
          v[q].y = fma(-u[q].x, wy, fma(-u[q].y, wx, v[q].y));
          y[r + q * L] = v[q];
        }
      }
      for (; r < mine; r += L) {
        const double2 u = x[r];
        double2 v = y[r];
        v.x = fma(-u.x, wx, fma(u.y, wy, v.x));
        v.y = fma(-u.x, wy, fma(-u.y, wx, v.y));
        y[r] = v;
      }
      if (rank == own && ln == 0) {
        const double2 uj = s_u;
        y[jl].x = yj.x - (uj.x * wx - uj.y * wy);
        y[jl].y = yj.y - (uj.x * wy + uj.y * wx);
      }
    }
    __syncthreads();
  }
  // the panel's rows of R, the reflectors with their zeros and ones, tau
  for (int k = warp; k < nc; k += PANEL_T / 32) {
    const double2 s = s_scale[k];
    double2* H = q.H + row0 + (size_t)(row0 + k) * q.m;
    for (int r = lane; r < mine; r += 32) {
      const int g = lo + r;
      const double2 x = s_p[(size_t)k * rc + r];
      if (g < nc) q.R[row0 + g + (size_t)(row0 + k) * q.n] = g <= k ? x : make_double2(0.0, 0.0);
      double2 u = make_double2(g == k ? 1.0 : 0.0, 0.0);
      if (g > k) u = make_double2(x.x * s.x - x.y * s.y, x.x * s.y + x.y * s.x);
      H[g] = u;
    }
    if (rank == 0 && lane == 0) q.tau[row0 + k] = s_taus[k];
  }
  // zeros of R below the panel
  const int below = q.n - row0 - nc;
  for (int idx = rank * PANEL_T + tid; idx < below * nc; idx += C * PANEL_T)
    q.R[row0 + nc + idx % below + (size_t)(row0 + idx / below) * q.n] = make_double2(0.0, 0.0);
  cl.sync();                               // no CTA leaves while another may still write to its shared memory
}

// X = W T (forward) or W T^H (backward) from the parts of W, eight rows per block, one warp per row: x_k = tau_k (w_k -
// sum_{i < k} x_i S_ik), or from the last column up with conj(S_ki). Forward also adds S's parts, the rows below
// W's (kept for backward). S is scaled by tau_i first, so a step of the solve is four FP64 operations of a warp.
__global__ void __launch_bounds__(32 * WT_ROWS) k_qr_wt(const QRBlk* blk, const ZGemmItem* ops, int p, int backward) {
  __shared__ double2 s_s[NB][NB + 1];
  __shared__ double2 s_w[WT_ROWS][NB + 1];
  const int i = blockIdx.y;
  const QRBlk& B = blk[i];
  const QRItem q = B.q;
  const int row0 = p * NB, nc = min(NB, q.n - row0);
  if (q.m <= 0 || nc <= 0) return;
  const int n_rows = backward ? q.n - row0 : q.n - row0 - NB;
  const int r0 = blockIdx.x * WT_ROWS;
  if (r0 >= n_rows && (backward || blockIdx.x > 0)) return;
  const int ks = ops[i].split_ks, nch = ((q.m - row0 + 15) / 16 + ks - 1) / ks;      // W's K chunks
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t ldw = B.n_cap + NB, chunk = ldw * NB;
  double2* S = B.S + (size_t)p * NB * NB;
  auto sum = [&](size_t at) {
    double2 v = make_double2(0.0, 0.0);
    for (int c = 0; c < nch; ++c) {
      const double2 t = B.Wp[c * chunk + at];
      v.x += t.x;
      v.y += t.y;
    }
    return v;
  };
  // s_s[c][k]: tau_c S_ck (forward, k > c) or tau_c conj(S_kc) (backward, k < c)
  // S_ab, a < b: a warp takes column 16 + i and column 15 - i (an FP64 instruction takes as long
  // for half a warp's lanes)
  for (int e = tid; e < NB * NB / 2; e += blockDim.x) {
    const int l = e % NB, d = NB / 2 + e / NB, a = l < d ? l : NB - 1 - l, b = l < d ? d : NB - 1 - d;
    if (l == d || b >= nc) continue;
    double2 v;
    if (backward) {
      v = S[a + b * NB];
    } else {
      v = sum(max(0, n_rows) + a + (size_t)b * ldw);
      if (blockIdx.x == 0) S[a + b * NB] = v;
    }
    const double t = q.tau[row0 + (backward ? b : a)];
    if (backward) s_s[b][a] = make_double2(v.x * t, -v.y * t);
    else s_s[a][b] = make_double2(v.x * t, v.y * t);
  }
  for (int e = tid; e < WT_ROWS * NB; e += blockDim.x) {
    const int r = r0 + e % WT_ROWS, k = e / WT_ROWS;
    s_w[e % WT_ROWS][k] = (r < n_rows && k < nc) ? sum(r + (size_t)k * ldw) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  double2 w = s_w[warp][lane];
  for (int step = 0; step < nc; ++step) {
    const int c = backward ? nc - 1 - step : step;
    const double xr = __shfl_sync(0xffffffffu, w.x, c), xi = __shfl_sync(0xffffffffu, w.y, c);
    if (lane < nc && (backward ? lane < c : lane > c)) {
      const double2 s = s_s[c][lane];
      w.x = fma(-xr, s.x, fma(xi, s.y, w.x));
      w.y = fma(-xr, s.y, fma(-xi, s.x, w.y));
    }
  }
  const double tk = lane < nc ? q.tau[row0 + lane] : 0.0;
  s_w[warp][lane] = make_double2(w.x * tk, w.y * tk);
  __syncthreads();
  for (int e = tid; e < WT_ROWS * NB; e += blockDim.x) {
    const int r = r0 + e % WT_ROWS, k = e / WT_ROWS;
    if (r < n_rows && k < nc) B.X[r + (size_t)k * B.n_cap] = s_w[e % WT_ROWS][k];
  }
}

// Small matrices whole: one CTA per matrix, which stays in shared memory from the load to the explicit Q (formed in place,
// last reflector first). For what one SM's FP64 pipe does in the time that the panels' launches and exchanges take
// (through the C ABI, against one panel and the whole-GPU kernel: ten 61 x 24 0.24, 0.33, 0.35 ms; six 300 x 16 0.29,
// 0.38, 0.36; ten 61 x 32 0.36, 0.37, 0.45; but six 300 x 32 0.86, 0.44, 0.66): see qr_small_fits.
__global__ void __launch_bounds__(PT, 1) k_qr_small(const QRItem* items, int n_items, int elems_cap, int* status) {
  extern __shared__ __align__(16) double2 s_p[];
  __shared__ double2 s_tot[SMALL_N], s_w[SMALL_N], s_s;
  __shared__ double s_tau[SMALL_N];
  const QRItem q = items[blockIdx.x];
  if (!live(q)) return;
  const int m = q.m, n = q.n;
  if (n > SMALL_N || m * n > elems_cap) {
    if (threadIdx.x == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int e = tid; e < m * n; e += PT) s_p[e] = q.A[e];
  __syncthreads();
  // s_tot[k] = sum_{r > j} conj(x_r) a_k,r of this warp's columns k >= from (k mod 16), x = column j
  auto dots = [&](int j, int from) {
    const double2* x = s_p + (size_t)j * m;
    for (int k = from + ((warp - from) & (PW - 1)); k < n; k += PW) {
      const double2* y = s_p + (size_t)k * m;
      double a = 0, b = 0;
      for (int r = j + 1 + lane; r < m; r += 32) {
        const double2 u = x[r], v = y[r];
        a = fma(u.x, v.x, fma(u.y, v.y, a));
        b = fma(u.x, v.y, fma(-u.y, v.x, b));
      }
      __syncwarp();
      const double t = wsum2(a, b, lane);
      if (lane == 0) s_tot[k].x = t;
      if (lane == 16) s_tot[k].y = t;
    }
  };
  // a_k -= x s w_k below row j for the same columns
  auto update = [&](int j, int from) {
    const double2* x = s_p + (size_t)j * m;
    for (int k = from + ((warp - from) & (PW - 1)); k < n; k += PW) {
      double2* y = s_p + (size_t)k * m;
      const double2 w = s_w[k];
      for (int r = j + 1 + lane; r < m; r += 32) {
        const double2 u = x[r];
        double2 v = y[r];
        v.x = fma(-u.x, w.x, fma(u.y, w.y, v.x));
        v.y = fma(-u.x, w.y, fma(-u.y, w.x, v.y));
        y[r] = v;
      }
    }
  };
  for (int j = 0; j < n; ++j) {
    dots(j, j);
    __syncthreads();
    if (warp == 0) {
      // as in k_qr_panel; lanes 0 and 1 take the two inverse square roots at the same time
      const double2 al = s_p[j + (size_t)j * m];
      const double a2 = fma(al.x, al.x, al.y * al.y), n2 = s_tot[j].x + a2;
      const double v = lane == 0 ? a2 : n2;
      const double ri = v > 0.0 || v != v ? rsqrt(v) : 0.0;
      double rt = v * ri;
      rt = fma(0.5 * ri, fma(-rt, rt, v), rt);
      const double ra = __shfl_sync(0xffffffffu, ri, 0), rn = __shfl_sync(0xffffffffu, ri, 1);
      const double aabs = __shfl_sync(0xffffffffu, rt, 0), nrm = __shfl_sync(0xffffffffu, rt, 1);
      const double2 ph = a2 > 0.0 ? make_double2(al.x * ra, al.y * ra) : make_double2(1.0, 0.0);
      const bool some = n2 > 0.0 || n2 != n2;
      const double sum = aabs + nrm, inv = some ? 1.0 / sum : 0.0;
      const double cr = rn * ph.x, ci = rn * ph.y, ti = rn * inv;
      auto row_j = [&](int k, double2 yj, double2 w) {
        s_w[k] = w;
        const double ux = ph.x * sum, uy = ph.y * sum;
        s_p[j + (size_t)k * m] = make_double2(yj.x - (ux * w.x - uy * w.y), yj.y - (ux * w.y + uy * w.x));
      };
      if (!no_value(ti)) {
        for (int k = j + 1 + lane; k < n; k += 32) {
          const double2 yj = s_p[j + (size_t)k * m], t = s_tot[k];
          row_j(k, yj, make_double2(fma(cr, yj.x, fma(ci, yj.y, ti * t.x)), fma(cr, yj.y, fma(-ci, yj.x, ti * t.y))));
        }
      } else {
        for (int k = j + 1 + lane; k < n; k += 32) {
          const double2 yj = s_p[j + (size_t)k * m], t = make_double2(rn * (inv * s_tot[k].x), rn * (inv * s_tot[k].y));
          row_j(k, yj, make_double2(fma(cr, yj.x, fma(ci, yj.y, t.x)), fma(cr, yj.y, fma(-ci, yj.x, t.y))));
        }
      }
      if (lane == 0) {
        s_s = make_double2(ph.x * inv, -ph.y * inv);
        s_tau[j] = some ? sum * rn : 0.0;
        if (some) s_p[j + (size_t)j * m] = make_double2(-ph.x * nrm, -ph.y * nrm);
      }
    }
    __syncthreads();
    update(j, j + 1);
    __syncthreads();
    // u below the diagonal, with u_j = 1
    const double2 s = s_s;
    for (int r = j + 1 + tid; r < m; r += PT) {
      const double2 x = s_p[r + (size_t)j * m];
      s_p[r + (size_t)j * m] = make_double2(x.x * s.x - x.y * s.y, x.x * s.y + x.y * s.x);
    }
  }
  __syncthreads();
  for (int e = tid; e < n * n; e += PT) {
    const int r = e % n, k = e / n;
    q.R[e] = r <= k ? s_p[r + (size_t)k * m] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  for (int j = n - 1; j >= 0; --j) {
    dots(j, j + 1);
    __syncthreads();
    const double tau = s_tau[j];
    if (warp == 0)
      for (int k = j + 1 + lane; k < n; k += 32) {
        // row j of a later column of Q is zero before P_j
        const double2 w = make_double2(tau * s_tot[k].x, tau * s_tot[k].y);
        s_w[k] = w;
        s_p[j + (size_t)k * m] = make_double2(-w.x, -w.y);
      }
    __syncthreads();
    update(j, j + 1);
    __syncthreads();
    for (int r = tid; r < m; r += PT) {
      double2& x = s_p[r + (size_t)j * m];
      x = r < j ? make_double2(0.0, 0.0) : (r == j ? make_double2(1.0 - tau, 0.0) : make_double2(-tau * x.x, -tau * x.y));
    }
    __syncthreads();
  }
  for (int e = tid; e < m * n; e += PT) q.A[e] = s_p[e];
}

// A <- [I; 0] (R has been copied out); grid (x: elements, y: matrices)
__global__ void k_qr_identity(const QRBlk* blk, int n_items) {
  const QRItem q = blk[blockIdx.y].q;
  const size_t tot = (size_t)max(0, q.m) * max(0, q.n);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (size_t)gridDim.x * blockDim.x)
    q.A[e] = make_double2(e % q.m == e / q.m ? 1.0 : 0.0, 0.0);
}

namespace {

// clusters of c CTAs (one CTA per SM) that fit the device at the same time, c = 1 .. MAX_C; 0: not launchable. Filled once
// per device, by one thread while the others wait
struct ClusterTable {
  std::once_flag once;
  int active[MAX_C + 1] = {};
};
constexpr int MAX_DEV = 64;
ClusterTable g_tab[MAX_DEV];

cudaLaunchConfig_t panel_cfg(int clusters, int c, size_t smem, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * c, 1, 1);
  cfg.blockDim = dim3(PANEL_T, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = c;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

const ClusterTable& cluster_table() {
  int dev = 0;
  cudaGetDevice(&dev);
  ClusterTable& t = g_tab[std::max(0, std::min(dev, MAX_DEV - 1))];
  std::call_once(t.once, [&t] {
    cudaFuncSetAttribute(k_qr_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, PANEL_SMEM);
    cudaFuncSetAttribute(k_qr_panel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int c = 1; c <= MAX_C; ++c) {
      cudaLaunchAttribute at[1];
      cudaLaunchConfig_t cfg = panel_cfg(1, c, PANEL_SMEM, 0, at);
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_qr_panel, &cfg) == cudaSuccess) t.active[c] = n;
      cudaGetLastError();
    }
  });
  return t;
}

size_t up(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

// CTAs per cluster for n matrices of at most m rows: the shortest estimate of a panel column's time, waves of clusters
// times (76 cycles of FP64 work per row of a CTA, for the 16 columns a panel has right of a column on average, + 4000
// cycles of exchange, scalars and barriers); 0: the panel does not fit
int qr_block_cluster(int n, int m) {
  const ClusterTable& t = cluster_table();
  int best = 0;
  double cost = 1e300;
  for (int c = 1; c <= MAX_C; ++c) {
    const int rc = (m + c - 1) / c;
    if (t.active[c] <= 0 || (size_t)rc * NB * sizeof(double2) > (size_t)PANEL_SMEM) continue;
    const double v = (double)((n + t.active[c] - 1) / t.active[c]) * (76.0 * rc + 4000.0);
    if (v < cost) {
      cost = v;
      best = c;
    }
  }
  return best;
}

size_t qr_block_bytes(int m, int n, QRBlk* B, char* base) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    char* r = base ? base + o : nullptr;
    o += up(bytes);
    return r;
  };
  const size_t ch = std::max(zgemm9_chunks(m), std::min(MAX_PARTS, (m + 15) / 16)), pn = (n + NB - 1) / NB;
  QRBlk b{};
  b.m_cap = m;
  b.n_cap = n;
  b.Wp = (double2*)take(sizeof(double2) * ch * (n + NB) * NB);
  b.X = (double2*)take(sizeof(double2) * n * NB);
  b.S = (double2*)take(sizeof(double2) * pn * NB * NB);
  b.TA = (unsigned char*)take(zgemm9_pack_bytes(n + NB, m, 0));
  b.TB = (unsigned char*)take(zgemm9_pack_bytes(NB, m, 1));
  b.TA2 = (unsigned char*)take(zgemm9_pack_bytes(m, NB, 0));
  b.TB2 = (unsigned char*)take(zgemm9_pack_bytes(n, NB, 1));
  if (B) *B = b;
  return o;
}

// Up to 16 columns and 5120 entries, or 32 and 2560: between the sizes measured at k_qr_small.
int qr_small_fits(int m, int n) { return n <= SMALL_N && m * (long long)n <= (n <= 16 ? 5120 : 2560); }

void launch_qr_small(const QRItem* items, int n_items, int m_cap, int n_cap, int* status, cudaStream_t st) {
  // at most 80 KB
  cudaFuncSetAttribute(k_qr_small, cudaFuncAttributeMaxDynamicSharedMemorySize, 5120 * (int)sizeof(double2));
  k_qr_small<<<n_items, PT, (size_t)m_cap * n_cap * sizeof(double2), st>>>(items, n_items, m_cap * n_cap, status);
}

size_t qr_block_ops(int n_items, int n_cap) { return (size_t)4 * n_items * ((n_cap + NB - 1) / NB); }

void launch_qr_block(const Tables& T, const BondWork* work, const QRItem* list, const QRBlkList& L, int* status,
                     cudaStream_t st) {
  const int n = L.n_items, panels = (L.n_cap + NB - 1) / NB;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  k_qrb_plan<<<(n * panels + 127) / 128, 128, 0, st>>>(T, work, list, L.blk, n, panels, L.ops, std::max(1, sms), status);
  const int rc = (L.m_cap + L.cluster - 1) / L.cluster;
  const long long ch = std::max(zgemm9_chunks(L.m_cap), MAX_PARTS);

  auto tiles = [](int m, int k) { return (long long)((m + 127) / 128) * ((k + 31) / 32); };
  for (int p = 0; p < panels; ++p) {
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = panel_cfg(n, L.cluster, (size_t)rc * NB * sizeof(double2), st, at);
    cudaLaunchKernelEx(&cfg, k_qr_panel, (const QRBlk*)L.blk, n, p, rc, status);
    const ZGemmItem* o = L.ops + (size_t)p * 4 * n;
    const int trail = std::max(0, L.n_cap - (p + 1) * NB), rows = std::max(1, L.m_cap - p * NB);
    launch_zgemm9(o, n, tiles(trail + NB, 1) * ch * n, trail + NB, NB, L.m_cap, status, st);
    k_qr_wt<<<dim3(std::max(1, (trail + WT_ROWS - 1) / WT_ROWS), n), 32 * WT_ROWS, 0, st>>>(L.blk, o, p, 0);
    if (trail > 0) launch_zgemm9(o + n, n, tiles(rows, trail) * n, rows, trail, NB, status, st);
  }
  k_qr_identity<<<dim3(std::min(64, (L.m_cap * std::min(L.n_cap, 64) + 255) / 256), n), 256, 0, st>>>(L.blk, n);
  for (int p = panels - 1; p >= 0; --p) {
    const ZGemmItem* o = L.ops + (size_t)p * 4 * n;
    const int cols = L.n_cap - p * NB, rows = std::max(1, L.m_cap - p * NB);
    launch_zgemm9(o + 2 * n, n, tiles(cols, 1) * ch * n, cols, NB, L.m_cap, status, st);
    k_qr_wt<<<dim3((cols + WT_ROWS - 1) / WT_ROWS, n), 32 * WT_ROWS, 0, st>>>(L.blk, o + 2 * n, p, 1);
    launch_zgemm9(o + 3 * n, n, tiles(rows, cols) * n, rows, cols, NB, status, st);
  }
}

}  // namespace ptk
