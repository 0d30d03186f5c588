// Batched complex GEMM on the tensor cores with an FP64-class result, for the large products of
// the fast path's bond SVD (App. A.2): the randomized range finder's sketches D Omega and
// D^H Q, the projection Q^H D, and the singular vectors of D built from those of the small factor.
//
//   C_i = opA(A_i) opB(B_i)        (M_i x N_i, inner dimension K_i; op = as stored, T or H)
//
// for a list of items whose live dims sit in device memory: a plan kernel writes the list from the
// bonds' info words, so one CUDA graph replays every step unchanged.
//
// Arithmetic (the error-free splitting of Ozaki, Ogita, Oishi and Rump, as in the theta GEMM):
// every row of opA(A) and every column of opB(B) is scaled by a power of two 2^-e so its entries
// lie in (-1, 1), then cut into six BF16 fixed-point slices a_s 2^(-7(s+1)) with integer
// |a_s| <= 2^7. Slice products are exact in FP32, and K is accumulated in chunks of 512 so that the
// level-0 and level-1 sums of a chunk stay integers below 2^24: the tensor cores' FP32 accumulation
// is exact there, the deeper levels carry only their own rounding, and the chunks are added in
// FP64 in the output. Products of slice
// pairs (s, t) accumulate in TMEM by level min(s + t, 3), real and imaginary parts separately
// (Re = Ar Br - Ai Bi via the MMA's negate-A bit, Im = Ar Bi + Ai Br); the epilogue adds the
// levels as 64-bit integers and applies 2^(e_row + e_col). The result is accurate to ~1e-12 of the scale
// of the rows and columns it combines (per 512-long chunk of K).
//
// Data flow: one preparation launch (row exponents, then the 12 slice planes in the tcgen05
// K-major no-swizzle layout: A in 128-row tiles, B in 64-column tiles, one 16-element K step per
// block, so one cp.async.bulk stages each), then one persistent GEMM launch (one CTA per SM) that
// walks the live 128 x 64 output tiles of all items with a two-stage bulk-copy / MMA pipeline.
// Every mbarrier wait is bounded: on expiry the kernel records ST_TIMEOUT in *status, waits
// (bounded) for its copies and MMAs in flight, frees its TMEM and returns.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "kernels.h"
#include "tc_common.cuh"

namespace ptk {

using namespace tcx;

namespace {

constexpr int ZNS = 6;                        // BF16 slices per value
constexpr int ZBITS = 7;                      // slice width
constexpr int ZKC_STEPS = 32;                 // K steps (16 each) per exact accumulation chunk: K = 512
using ZG = Geo<true>;                         // BF16 geometry: 16-element K steps

__host__ __device__ __forceinline__ PackCap zcap(const ZGemmItem& it, int which) {
  return which == 0 ? pack_cap(it.cap_m, it.cap_k, TMA, ZG::KSTEP, ZNS)
                    : pack_cap(it.cap_n, it.cap_k, TNB, ZG::KSTEP, ZNS);
}

__device__ __forceinline__ bool item_live(const ZGemmItem& it) { return it.M > 0 && it.N > 0 && it.K > 0; }

__device__ __forceinline__ bool item_fits(const ZGemmItem& it) {
  return it.M <= it.cap_m && it.N <= it.cap_n && it.K <= it.cap_k;
}

}  // namespace

// Operand preparation, both passes in one launch: a block takes PREP_ROWS rows of opA(A) (blockIdx.x < n_a) or
// columns of opB(B) of one item, finds each one's exponent e (max |entry| < 2^e), then writes the 12 slice
// planes: one thread per (row, 8-element K group), 16 bytes per plane, eight consecutive rows in consecutive
// 16-byte slots. The second read of the block's rows comes from L1 or L2.
// Bound by the integer pipes and the planes' writes (24 bytes per element). Integer arithmetic throughout
// (tc_common.cuh): with the slices cut by FP64 rint and ldexp in a launch per operand after another for the
// exponents, the preparation of ten 1120 x 160 x 1120 products took 4.75 ms; the whole product, this kernel
// and the GEMM with its FP64-free epilogue included, went from 5.68 to 0.93 ms (21 products of 16384 x 64
// x 64: 7.67 to 1.54 ms).
// mode 0: B, and A unless the item marks it as packed; mode 1: A alone, marked or not.
// grid: (x: n_a + n_b row blocks, y: items)
constexpr int PREP_ROWS = 8, PREP_THREADS = 256;

__global__ void __launch_bounds__(PREP_THREADS) k_zg_prep(const ZGemmItem* items, int n_items, int n_a, int mode,
                                                          int* status) {
  const int i = blockIdx.y;
  if (i >= n_items) return;
  const ZGemmItem it = items[i];
  const int which = (int)blockIdx.x < n_a ? 0 : 1;
  const int blk = which == 0 ? blockIdx.x : blockIdx.x - n_a, nblk = which == 0 ? n_a : gridDim.x - n_a;
  if (!item_live(it) || (which == 0 && it.skip_a > 0 && mode == 0)) return;
  if (!item_fits(it)) {
    if (blk == 0 && threadIdx.x == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  const int rows = which == 0 ? it.M : it.N, tr = which == 0 ? TMA : TNB;
  const PackCap cp = zcap(it, which);
  unsigned char* out = which == 0 ? it.TA : it.TB;
  int* ex = (int*)(out + cp.exp_off);
  const int n_ks = cdiv(it.K, ZG::KSTEP), n_grp = 2 * n_ks;
  const int padded = cdiv(rows, tr) * tr;
  const bool k_contiguous = which == 0 ? it.opA != ZOP_N : it.opB == ZOP_N;
  const bool conj_op = (which == 0 ? it.opA : it.opB) == ZOP_C;
  const double2* src = which == 0 ? it.A : it.B;
  const size_t ld = which == 0 ? it.lda : it.ldb;
  __shared__ unsigned long long part[PREP_THREADS / PREP_ROWS][PREP_ROWS];
  __shared__ int s_e[PREP_ROWS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int r0 = blk * PREP_ROWS; r0 < padded; r0 += nblk * PREP_ROWS) {
    if (k_contiguous) {
      // one warp per row, lanes along K
      const int r = r0 + warp;
      unsigned long long m = 0;
      if (r < rows) {
        const double2* p = src + (size_t)((which == 1 && it.bcol) ? it.bcol[r] : r) * ld;
        for (int k = lane; k < it.K; k += 32) {
          const double2 v = p[k];
          m = max(m, max(mag_bits(v.x), mag_bits(v.y)));
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) s_e[warp] = row_exponent(__longlong_as_double((long long)m));
    } else {
      // rows contiguous: eight rows by 32 columns per pass of the block
      const int r = r0 + (tid % PREP_ROWS);
      unsigned long long m = 0;
      if (r < rows) {
        const int c = (which == 1 && it.bcol) ? it.bcol[r] : r;
        for (int k = tid / PREP_ROWS; k < it.K; k += PREP_THREADS / PREP_ROWS) {
          const double2 v = src[c + (size_t)k * ld];
          m = max(m, max(mag_bits(v.x), mag_bits(v.y)));
        }
      }
      part[tid / PREP_ROWS][tid % PREP_ROWS] = m;
      __syncthreads();
      if (tid < PREP_ROWS) {
        unsigned long long v = 0;
#pragma unroll
        for (int j = 0; j < PREP_THREADS / PREP_ROWS; ++j) v = max(v, part[j][tid]);
        s_e[tid] = row_exponent(__longlong_as_double((long long)v));
      }
    }
    __syncthreads();
    if (tid < PREP_ROWS) ex[r0 + tid] = s_e[tid];
    const int rt = r0 / tr, m0 = r0 % tr;
    unsigned char* tile = out + (size_t)rt * cp.ksteps * (2 * ZNS) * cp.plane_bytes;
    for (int idx = tid; idx < PREP_ROWS * n_grp; idx += PREP_THREADS) {
      const int rr = idx % PREP_ROWS, grp = idx / PREP_ROWS;
      const int r = r0 + rr, k0 = grp * ZG::KG, e = s_e[rr];
      const int c = (r < rows && which == 1 && it.bcol) ? it.bcol[r] : r;
      const double2* p = k_contiguous ? src + (size_t)c * ld + k0 : src + c + (size_t)k0 * ld;
      const size_t st = k_contiguous ? 1 : ld;
      uint32_t pr[ZNS][4], pi[ZNS][4];       // 8 BF16 per plane, two per word
#pragma unroll
      for (int j = 0; j < ZG::KG; j += 2) {
        double2 v[2];
#pragma unroll
        for (int q = 0; q < 2; ++q)
          v[q] = (r < rows && k0 + j + q < it.K) ? p[(size_t)(j + q) * st] : make_double2(0.0, 0.0);
        uint32_t a0[ZNS], a1[ZNS];
        int_slices<ZNS>(v[0].x, e, ZBITS, a0);
        int_slices<ZNS>(v[1].x, e, ZBITS, a1);
#pragma unroll
        for (int s = 0; s < ZNS; ++s) pr[s][j >> 1] = pair_bf16(a0[s], a1[s]);
        int_slices<ZNS>(conj_op ? -v[0].y : v[0].y, e, ZBITS, a0);
        int_slices<ZNS>(conj_op ? -v[1].y : v[1].y, e, ZBITS, a1);
#pragma unroll
        for (int s = 0; s < ZNS; ++s) pi[s][j >> 1] = pair_bf16(a0[s], a1[s]);
      }
      unsigned char* base = tile + (size_t)(grp >> 1) * (2 * ZNS) * cp.plane_bytes +
                            ((size_t)(grp & 1) * tr + m0 + rr) * 16;
#pragma unroll
      for (int s = 0; s < ZNS; ++s) {
        *(uint4*)(base + (size_t)s * cp.plane_bytes) = make_uint4(pr[s][0], pr[s][1], pr[s][2], pr[s][3]);
        *(uint4*)(base + (size_t)(ZNS + s) * cp.plane_bytes) = make_uint4(pi[s][0], pi[s][1], pi[s][2], pi[s][3]);
      }
    }
    __syncthreads();
  }
}

// The GEMM: persistent, one CTA per SM over the live 128 x 64 tiles of every item. K runs in chunks
// of 512 (32 MMA steps): each chunk's four levels accumulate exactly enough in TMEM, and the
// epilogue adds the chunk to C in FP64 (the first chunk writes C, or C - product for acc < 0).
__global__ void __launch_bounds__(TC_THREADS, 1) k_zgemm(const ZGemmItem* items, int n_items, int* status) {
  constexpr uint32_t A_PLANE = TMA * ROW_BYTES, B_PLANE = TNB * ROW_BYTES;
  constexpr uint32_t A_STAGE = 2 * ZNS * A_PLANE, B_STAGE = 2 * ZNS * B_PLANE, STAGE = A_STAGE + B_STAGE;
  constexpr int STAGES = Stages<ZNS>::value;
  constexpr int NLEV = 4;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint64_t bar_full[MAX_STAGES], bar_empty[MAX_STAGES];
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  __shared__ int col_exp[TNB];
  __shared__ int tile_off[MAX_ITEMS + 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (n_items > MAX_ITEMS) {
    if (blockIdx.x == 0 && tid == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  for (int i = tid; i < n_items; i += blockDim.x) {
    const ZGemmItem& it = items[i];
    tile_off[i + 1] = (item_live(it) && item_fits(it)) ? cdiv(it.M, TMA) * cdiv(it.N, TNB) : 0;
  }
  if (tid == 0) {
    tile_off[0] = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&bar_full[s], 1);
      mbar_init(&bar_empty[s], 1);
    }
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (tid == 0)
    for (int i = 0; i < n_items; ++i) tile_off[i + 1] += tile_off[i];
  __syncthreads();
  const int total = tile_off[n_items];
  if ((int)blockIdx.x >= total) return;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base_s))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base_s;
  const uint32_t idesc = instr_desc(1u, TMA, TNB);
  constexpr uint32_t LBO_A = TMA * 16, LBO_B = TNB * 16, SBO = 128;
  uint32_t g = 0;                 // K steps processed by this CTA (stage = g % STAGES)
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    int lo = 0, hi = n_items - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (tile_off[mid] <= t) lo = mid;
      else hi = mid - 1;
    }
    const ZGemmItem& it = items[lo];
    const PackCap ca = zcap(it, 0), cb = zcap(it, 1);
    const int nt_b = cdiv(it.N, TNB);
    const int rt = (t - tile_off[lo]) / nt_b, ct = (t - tile_off[lo]) % nt_b;
    const int n_ks = cdiv(it.K, ZG::KSTEP);
    if (tid < TNB) col_exp[tid] = ((const int*)(it.TB + cb.exp_off))[ct * TNB + tid];
    const unsigned char* gA = it.TA + (size_t)rt * ca.ksteps * A_STAGE;
    const unsigned char* gB = it.TB + (size_t)ct * cb.ksteps * B_STAGE;
    const int m = rt * TMA + warp * 32 + lane;
    const int e_m = ((const int*)(it.TA + ca.exp_off))[m];
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    bool bad = false;
    for (int ks0 = 0; ks0 < n_ks; ks0 += ZKC_STEPS) {
      const int nk = min(ZKC_STEPS, n_ks - ks0);
      if (tid == 0) {
        auto load = [&](int ks, uint32_t gg) {
          unsigned char* st = smem + (gg % STAGES) * STAGE;
          uint64_t* bar = &bar_full[gg % STAGES];
          mbar_expect_tx(bar, STAGE);
          bulk_g2s(st, gA + (size_t)(ks0 + ks) * A_STAGE, A_STAGE, bar);
          bulk_g2s(st + A_STAGE, gB + (size_t)(ks0 + ks) * B_STAGE, B_STAGE, bar);
        };
        auto par = [](uint32_t gg) { return (gg / STAGES) & 1u; };
        bool ok = true;
        uint32_t loaded = g, waited = g, committed = 0;
        bool any_commit = false;
        bool init[NLEV] = {false, false, false, false};
        // prologue: the chunk's first STAGES - 1 steps (their stages were freed by the last wait)
        for (int ks = 0; ks < nk && ks < STAGES - 1; ++ks) {
          load(ks, g + ks);
          loaded = g + ks + 1;
        }
        for (int ks = 0; ks < nk && ok; ++ks) {
          const uint32_t gg = g + ks;
          ok = mbar_wait(&bar_full[gg % STAGES], par(gg));
          if (!ok) break;
          waited = gg + 1;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const unsigned char* sa = smem + (gg % STAGES) * STAGE;
          const unsigned char* sb = sa + A_STAGE;
#pragma unroll
          for (int s = 0; s < ZNS; ++s) {
#pragma unroll
            for (int u = 0; u < ZNS - s; ++u) {
              const int L = (s + u) < NLEV - 1 ? (s + u) : NLEV - 1;
              const uint32_t dre = tmem + (2 * L) * TNB, dim = dre + TNB;
              const uint64_t ar = smem_desc(sa + s * A_PLANE, LBO_A, SBO);
              const uint64_t ai = smem_desc(sa + (ZNS + s) * A_PLANE, LBO_A, SBO);
              const uint64_t br = smem_desc(sb + u * B_PLANE, LBO_B, SBO);
              const uint64_t bi = smem_desc(sb + (ZNS + u) * B_PLANE, LBO_B, SBO);
              mma<true>(dre, ar, br, idesc, init[L]);
              mma<true>(dre, ai, bi, idesc | NEG_A, true);
              mma<true>(dim, ar, bi, idesc, init[L]);
              mma<true>(dim, ai, br, idesc, true);
              init[L] = true;
            }
          }
          mma_commit(&bar_empty[gg % STAGES]);
          committed = gg;
          any_commit = true;
          const int nx = ks + STAGES - 1;
          if (nx < nk) {
            if (ks >= 1) ok = mbar_wait(&bar_empty[(gg - 1) % STAGES], par(gg - 1));
            if (!ok) break;
            load(nx, g + nx);
            loaded = g + nx + 1;
          }
        }
        if (ok && any_commit) ok = mbar_wait(&bar_empty[committed % STAGES], par(committed));
        if (!ok) {
          atomicOr(status, ST_TIMEOUT);
          abort_s = 1;
          for (uint32_t q = waited; q < loaded; ++q) mbar_wait(&bar_full[q % STAGES], par(q));
          if (any_commit) mbar_wait(&bar_empty[committed % STAGES], par(committed));
        }
      }
      g += nk;
      __syncthreads();
      if (abort_s) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // epilogue of the chunk: thread = row m of the tile, 8 columns per TMEM load
      const bool first = ks0 == 0;
      for (int c0 = 0; c0 < TNB; c0 += 8) {
        long long re[8], im[8];
        uint32_t nonfin = 0;
        {
          float x[NLEV][8], y[NLEV][8];
#pragma unroll
          for (int L = 0; L < NLEV; ++L) {
            tmem_ld8_nowait(tmem + lane_base + (2 * L) * TNB + c0, x[L]);
            tmem_ld8_nowait(tmem + lane_base + (2 * L + 1) * TNB + c0, y[L]);
          }
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const bool f = level_sum(x[0][j], x[1][j], x[2][j], x[3][j], &re[j]) &
                           level_sum(y[0][j], y[1][j], y[2][j], y[3][j], &im[j]);
            if (!f) nonfin |= 1u << j;
          }
        }
        if (m < it.M) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int n = ct * TNB + c0 + j;
            if (n >= it.N) continue;
            const int e = e_m + col_exp[c0 + j];
            double2 v = make_double2(fixed_to_double(it.acc < 0 ? -re[j] : re[j], e),
                                     fixed_to_double(it.acc < 0 ? -im[j] : im[j], e));
            if (nonfin >> j & 1u) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
            double2* cp = it.C + m + (size_t)n * it.ldc;
            if (!first || it.acc < 0) {
              const double2 o = *cp;
              v = make_double2(o.x + v.x, o.y + v.y);
            }
            bad |= mag_bits(v.x) != ((unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull) ||
                   mag_bits(v.y) != ((unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull);
            *cp = v;
          }
        }
      }
      // TMEM reads complete before the next chunk's MMAs overwrite the accumulators
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (abort_s) break;
    if (bad && it.flag) *it.flag = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

size_t zgemm_pack_bytes(int rows_cap, int k_cap, int which) {
  return pack_cap(std::max(1, rows_cap), std::max(1, k_cap), which == 0 ? TMA : TNB, ZG::KSTEP, ZNS).total;
}

int zgemm_max_items() { return MAX_ITEMS; }

int zgemm_tile_cap(int m_cap, int n_cap) { return cdiv(std::max(1, m_cap), TMA) * cdiv(std::max(1, n_cap), TNB); }

namespace {
constexpr int ZMAX_DEV = 64;
bool g_zattr_done[ZMAX_DEV] = {};
}  // namespace

void launch_zgemm_pack_a(const ZGemmItem* items, int n_items, int m_cap_max, int* status, cudaStream_t st) {
  if (n_items <= 0) return;
  const int n_a = std::min(2048, cdiv(cdiv(std::max(1, m_cap_max), TMA) * TMA, PREP_ROWS));
  k_zg_prep<<<dim3(n_a, n_items), PREP_THREADS, 0, st>>>(items, n_items, n_a, 1, status);
}

void launch_zgemm(const ZGemmItem* items, int n_items, int tile_cap, int m_cap_max, int n_cap_max, int* status,
                  cudaStream_t st) {
  if (n_items <= 0) return;
  const int n_a = std::min(2048, cdiv(cdiv(std::max(1, m_cap_max), TMA) * TMA, PREP_ROWS));
  const int n_b = std::min(2048, cdiv(cdiv(std::max(1, n_cap_max), TNB) * TNB, PREP_ROWS));
  k_zg_prep<<<dim3(n_a + n_b, n_items), PREP_THREADS, 0, st>>>(items, n_items, n_a, 0, status);
  const size_t smem = (size_t)Stages<ZNS>::value * 2 * ZNS * (TMA + TNB) * ROW_BYTES + 1024;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (dev >= 0 && dev < ZMAX_DEV && !g_zattr_done[dev]) {
    cudaFuncSetAttribute(k_zgemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    g_zattr_done[dev] = true;
  }
  const int grid = std::max(1, std::min(sms > 0 ? sms : 152, tile_cap));
  k_zgemm<<<grid, TC_THREADS, smem, st>>>(items, n_items, status);
}

}  // namespace ptk
