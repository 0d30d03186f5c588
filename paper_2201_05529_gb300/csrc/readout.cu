// Readout of the augmented MPS (App. A.3): every augmented leg closed by its cap C^(k), the Liouville legs by
// vec(I) except vec(O^T) on the measured site, the bond weights in between.
//
//   M_n[p][l][r] = sum_a Gamma_n[l,p,a,r] C_n[a], V_n = M_n[0] + M_n[3]         (k_observe_m, all sites at once)
//   L_{n+1} = (L_n V_n) lambda_{n+1},  R_n = V_n (lambda_{n+1} R_{n+1})            (k_observe_pass)
//   E_n[p] = L_n M_n[p] (lambda_{n+1} R_{n+1}),  <O>_n = sum_p vec(O^T)_p E_n[p]   (k_observe_sites)
//
// What bounds it: the passes are a chain of N dependent matrix-vector products, and FP64 issues one warp
// instruction per 19 cycles and SM, so a 64 x 64 complex product takes 7 us on one SM. Each pass (left and
// right of every chain, at the same time) therefore runs on a cluster of eight CTAs that split the output
// entries and exchange the vector through distributed shared memory, one cluster barrier per site; the site
// expectations form the four products E_n[p] once instead of one contraction per operator, one CTA per (site, p).
// With one CTA per chain for all of it, reading out three operators of a 21-site state (chi 64, kappa 16) took 2.19 ms through the C ABI; now 0.16 ms.
#include <cooperative_groups.h>

#include <utility>

#include "kernels.h"

namespace cg = cooperative_groups;

namespace ptk {

namespace {
constexpr int RD_THREADS = 256;
constexpr int RD_WARPS = RD_THREADS / 32;
constexpr int RD_CLUSTER = 8;              // CTAs per pass (1 below RD_SMALL: a barrier costs more than it saves)
constexpr int RD_SMALL = 24;

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
}  // namespace

// planes [5][chi_l][chi_r] of one site: M[0..3] and V. grid: x over elements, y over chains, z over sites
__global__ void k_observe_m(Tables T, int n_chains, double2* Mbuf, const size_t* moff) {
  const int c = blockIdx.y, n = blockIdx.z;
  if (c >= n_chains || n >= T.chain_N[c]) return;
  const int k = *T.step;
  const int s = T.chain_site0[c] + n, B = T.chain_lam0[c] + n;
  const int chl = T.lam_chi[B], chr = T.lam_chi[B + 1], kap = T.site_kappa[s];
  const double2* G = T.site_gam[s];
  const int m = T.site_mpo[s];
  const double2* capv = m >= 0 ? T.mpo_cap[T.mpo_cap_off[m] + k] : nullptr;
  double2* M = Mbuf + moff[s];
  const int plane = chl * chr;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < 2 * plane; idx += gridDim.x * blockDim.x) {
    // a thread closes p = 0 and 3 of one (l, r), or p = 1 and 2
    const int e = idx % plane, outer = idx / plane == 0;
    const int r = e % chr, l = e / chr;
    const int p0 = outer ? 0 : 1, p1 = outer ? 3 : 2;
    const double2* g0 = G + (((size_t)l * 4 + p0) * kap) * chr + r;
    const double2* g1 = G + (((size_t)l * 4 + p1) * kap) * chr + r;
    double2 v0 = cmk(0, 0), v1 = cmk(0, 0);
    for (int a = 0; a < kap; ++a) {
      const double2 cv = capv ? capv[a] : cmk(1, 0);
      v0 = cfma(g0[(size_t)a * chr], cv, v0);
      v1 = cfma(g1[(size_t)a * chr], cv, v1);
    }
    M[(size_t)p0 * plane + e] = v0;
    M[(size_t)p1 * plane + e] = v1;
    if (outer) M[(size_t)4 * plane + e] = cadd(v0, v1);
  }
}

// One cluster per (chain, direction): cluster 2 chain + direction. Shared memory: two vectors of ld entries.
__global__ void __launch_bounds__(RD_THREADS) k_observe_pass(Tables T, int n_chains, int n_max, double2* Lbuf,
                                                             double2* Rbuf, int ld, const double2* Mbuf,
                                                             const size_t* moff) {
  extern __shared__ double2 s_vec[];       // [2][ld]
  __shared__ double2 s_red[RD_WARPS][8];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), ncta = (int)cl.num_blocks();
  const int job = (int)(blockIdx.x / ncta), c = job >> 1;
  const bool right = job & 1;
  const int N = T.chain_N[c], s0 = T.chain_site0[c], B0 = T.chain_lam0[c];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double2* out = (right ? Rbuf : Lbuf) + (size_t)c * (n_max + 1) * ld;
  if (tid == 0) {
    const double2 v0 = right ? cmk(1, 0) : cmk(T.lam_ptr[B0][0], 0);
    s_vec[0] = v0;
    if (rank == 0) out[right ? (size_t)N * ld : 0] = v0;
  }
  cl.sync();                               // every CTA's buffers exist before the first remote store
  for (int i = 0; i < N; ++i) {
    const int n = right ? N - 1 - i : i;
    const int chl = T.lam_chi[B0 + n], chr = T.lam_chi[B0 + n + 1];
    const double* lam = T.lam_ptr[B0 + n + 1];
    const double2* V = Mbuf + moff[s0 + n] + (size_t)4 * chl * chr;
    const double2* x = s_vec + (i & 1) * ld;
    double2* y = s_vec + ((i + 1) & 1) * ld;
    double2* yo = out + (size_t)(right ? n : n + 1) * ld;
    auto put = [&](int e, double2 v) {
      for (int q = 0; q < ncta; ++q) *cl.map_shared_rank(y + e, q) = v;
      yo[e] = v;
    };
    if (!right) {
      // eight columns r per CTA and turn: lanes 8 r x 4 l, warps over l, V's rows read along r
      for (int r0 = rank * 8; r0 < chr; r0 += ncta * 8) {
        const int r = r0 + (lane & 7);
        double2 a0 = cmk(0, 0), a1 = cmk(0, 0);
        if (r < chr) {
          int l = warp * 4 + (lane >> 3);
          for (; l + 32 < chl; l += 64) {
            a0 = cfma(x[l], V[(size_t)l * chr + r], a0);
            a1 = cfma(x[l + 32], V[(size_t)(l + 32) * chr + r], a1);
          }
          if (l < chl) a0 = cfma(x[l], V[(size_t)l * chr + r], a0);
        }
        a0 = cadd(a0, a1);
#pragma unroll
        for (int o = 8; o <= 16; o <<= 1) {
          a0.x += __shfl_xor_sync(0xffffffffu, a0.x, o);
          a0.y += __shfl_xor_sync(0xffffffffu, a0.y, o);
        }
        if (lane < 8) s_red[warp][lane] = a0;
        __syncthreads();
        if (tid < 8 && r0 + tid < chr) {
          double2 v = s_red[0][tid];
#pragma unroll
          for (int w = 1; w < RD_WARPS; ++w) v = cadd(v, s_red[w][tid]);
          put(r0 + tid, cscale(v, lam[r0 + tid]));
        }
        __syncthreads();
      }
    } else {
      // one row l per warp and turn, lanes along r
      for (int l = rank * RD_WARPS + warp; l < chl; l += ncta * RD_WARPS) {
        double2 a = cmk(0, 0);
        for (int r = lane; r < chr; r += 32) a = cfma(V[(size_t)l * chr + r], cscale(x[r], lam[r]), a);
        a.x = wsum(a.x);
        a.y = wsum(a.y);
        if (lane == 0) put(l, a);
      }
    }
    cl.sync();                             // y is complete in every CTA; x may be overwritten
  }
}

// Clusters of four CTAs, one per Liouville index p: blockIdx.x = p, y = site, z = chain
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(RD_THREADS)
    k_observe_sites(Tables T, const double2* ops, int n_ops, int n_max, double2* obs, double2* trace, int n_chains,
                    const double2* Lbuf, const double2* Rbuf, int ld, int use_history, const double2* Mbuf,
                    const size_t* moff) {
  __shared__ double2 s_e[4];
  __shared__ double s_red[2][RD_WARPS];
  cg::cluster_group cl = cg::this_cluster();
  auto started = cl.barrier_arrive();      // CTA 0 runs before another one stores into its shared memory
  const int p = blockIdx.x, n = blockIdx.y, c = blockIdx.z;
  const int N = T.chain_N[c];
  const bool live = n < N;                 // the same for the whole cluster
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = *T.step, B0 = T.chain_lam0[c];
  const double2* Lp = Lbuf + (size_t)c * (n_max + 1) * ld;
  const double2* Rs = Rbuf + (size_t)c * (n_max + 1) * ld;
  if (live) {
    const int chl = T.lam_chi[B0 + n], chr = T.lam_chi[B0 + n + 1];
    const double* lam = T.lam_ptr[B0 + n + 1];
    const double2* M = Mbuf + moff[T.chain_site0[c] + n] + (size_t)p * chl * chr;
    double2 part = cmk(0, 0);
    for (int r = lane; r < chr; r += 32) {
      double2 a = cmk(0, 0);
      for (int l = warp; l < chl; l += RD_WARPS) a = cfma(Lp[(size_t)n * ld + l], M[(size_t)l * chr + r], a);
      part = cfma(a, cscale(Rs[(size_t)(n + 1) * ld + r], lam[r]), part);
    }
    part.x = wsum(part.x);
    part.y = wsum(part.y);
    if (lane == 0) {
      s_red[0][warp] = part.x;
      s_red[1][warp] = part.y;
    }
    __syncthreads();
  }
  cl.barrier_wait(std::move(started));
  if (live && tid == 0) {
    double2 e = cmk(0, 0);
#pragma unroll
    for (int w = 0; w < RD_WARPS; ++w) e = cadd(e, cmk(s_red[0][w], s_red[1][w]));
    *cl.map_shared_rank(&s_e[p], 0) = e;
  }
  cl.sync();
  if (!live || p != 0) return;
  double lognorm = 0.0;                    // fixed summation order
  if (tid <= n_ops)
    for (int b = 0; b <= N; ++b) lognorm += T.lam_lognorm[B0 + b];
  if (tid < n_ops) {
    const double2* o = ops + tid * 4;
    double2 v = cmk(0, 0);
#pragma unroll
    for (int q = 0; q < 4; ++q) v = cfma(o[q], s_e[q], v);
    double2* dst = obs + (use_history ? (size_t)k * n_chains * n_max * n_ops : 0);
    dst[((size_t)c * n_max + n) * n_ops + tid] = cscale(v, exp(lognorm));
  } else if (tid == n_ops && n == 0) {
    trace[(use_history ? (size_t)k * n_chains : 0) + c] = cscale(Lp[(size_t)N * ld], exp(lognorm));
  }
}

void launch_observe(const Tables& T, int n_chains, int n_max, int gx_m, const double2* ops, int n_ops, double2* obs,
                    double2* trace, double2* Lbuf, double2* Rbuf, int ld, int use_history, double2* Mbuf,
                    const size_t* moff, cudaStream_t st) {
  k_observe_m<<<dim3(gx_m, n_chains, n_max), RD_THREADS, 0, st>>>(T, n_chains, Mbuf, moff);
  const int cl = ld >= RD_SMALL ? RD_CLUSTER : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cl * 2 * n_chains, 1, 1);
  cfg.blockDim = dim3(RD_THREADS, 1, 1);
  cfg.dynamicSmemBytes = 2 * sizeof(double2) * (size_t)ld;      // at most 16 KB: init takes no bond above 512 (4 chi <= 2048)
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_observe_pass, T, n_chains, n_max, Lbuf, Rbuf, ld, (const double2*)Mbuf, moff);
  k_observe_sites<<<dim3(4, n_max, n_chains), RD_THREADS, 0, st>>>(T, ops, n_ops, n_max, obs, trace, n_chains, Lbuf,
                                                                  Rbuf, ld, use_history, Mbuf, moff);
}

}  // namespace ptk
