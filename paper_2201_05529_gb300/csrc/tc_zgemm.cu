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
// pairs (s, t) accumulate in TMEM by level min(s + t, 3), real and imaginary parts side by side
// (B's planes as (-Bi, Br, Bi): Ar (Br, Bi) and Ai (-Bi, Br), one MMA each); the epilogue adds the
// levels as 64-bit integers and applies 2^(e_row + e_col). The result is accurate to ~1e-12 of the scale
// of the rows and columns it combines (per 512-long chunk of K); where the terms of an entry add up coherently, in the
// slices too (constant operands), the FP32 accumulation of the deeper levels truncates to 1.2e-10 of K times that scale.
//
// Data flow: one preparation launch (row exponents, then the slice planes in the tcgen05
// K-major layout with the 32-byte swizzle: A in 128-row tiles, B in 64-column tiles, one 16-element K step per
// block, so one cp.async.bulk stages each), then one persistent GEMM launch (one CTA per SM) that
// walks the live 128 x 64 output tiles of all items with a two-stage bulk-copy / MMA pipeline.
// Every mbarrier wait is bounded: on expiry the kernel records ST_TIMEOUT in *status, waits
// (bounded) for its copies and MMAs in flight, frees its TMEM and returns.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <climits>
#include <mutex>

#include "kernels.h"
#include "tc_common.cuh"

namespace ptk {

using namespace tcx;

namespace {

constexpr int ZBITS = 7;                      // slice width
// The two precisions. Z6: six slices, 42 bits; levels 0..2 alone and 3..5 together fill TMEM with 64 columns (4 x
// 2 x 64); chunks of K = 512. Z9: nine slices, 63 bits, for products that stand in for FP64 ones (the blocked
// QR's updates): levels 0..6 alone and 7, 8 together (8 x 2 x 32 columns), every sum that counts exact for K <= 256 (7
// 2^13 K <= 2^24 for level 4). What forced each: the tensor cores truncate when they accumulate inexactly (levels
// 5..7 together: 1.3e-15 of max|row| max|column| for K = 256), and a reflector's unit entry sets the scale of a
// vector whose other entries are ~0.05 (eight slices: QR residuals 9e-15, nine 1e-15, FP64 kernel 8e-16).
struct Z6 {
  static constexpr int NS = 6, NLEV = 4, TN = TNB, KC = 32;
  static __device__ __forceinline__ double value(const float (&f)[NLEV][8], int j, int e, bool neg) {
    // the last level as it stands in FP32: its multiples of 2^-49
    const long long n = level_sum<0, 3, 49, 49, NS, 2 * 16 * KC>(f, j);
    return fixed_to_double(neg ? -n : n, e, 49);
  }
};
struct Z9 {
  static constexpr int NS = 9, NLEV = 8, TN = 32, KC = Z9_KSTEPS;
  // two words: levels 0..3 in units of 2^-35, the rest in units of 2^-70, one FP64 addition
  static __device__ __forceinline__ double value(const float (&f)[NLEV][8], int j, int e, bool neg) {
    const long long h = level_sum<0, 3, 35, 0, NS, 2 * 16 * KC>(f, j), l = level_sum<4, 7, 70, 65, NS, 2 * 16 * KC>(f, j);
    return fixed_to_double(neg ? -h : h, e, 35) + fixed_to_double(neg ? -l : l, e, 70);
  }
};
using ZG = Geo<true>;                         // BF16 geometry: 16-element K steps

template <class Z>
__host__ __device__ __forceinline__ PackCap zcap(const ZGemmItem& it, int which) {
  return which == 0 ? pack_cap(it.cap_m, it.cap_k, TMA, ZG::KSTEP, Z::NS)
                    : pack_cap(it.cap_n, it.cap_k, Z::TN, ZG::KSTEP, Z::NS, 3 * Z::NS);
}

__device__ __forceinline__ bool item_live(const ZGemmItem& it) { return it.M > 0 && it.N > 0 && it.K > 0; }

__device__ __forceinline__ bool item_fits(const ZGemmItem& it) {
  return it.M <= it.cap_m && it.N <= it.cap_n && it.K <= it.cap_k;
}

}  // namespace

// Operand preparation, both passes in one launch: a block takes PREP_ROWS rows of opA(A) (blockIdx.x < n_a) or
// columns of opB(B) of one item, finds each one's exponent e (max |entry| < 2^e), then writes the slice planes
// (A: 2 per slice, B: 3): one thread per (row, 8-element K group), 16 bytes per plane, consecutive rows in consecutive
// 16-byte slots. Eight rows per block, or 32 where K is at most 64 (a block of eight would have work for 64 threads). The second read of the block's rows comes from L1 or L2.
// Bound by the integer pipes and the planes' writes (24 bytes per element of A, 36 of B). Integer arithmetic throughout
// (tc_common.cuh): with the slices cut by FP64 rint and ldexp in a launch per operand after another for the
// exponents, the preparation of ten 1120 x 160 x 1120 products took 4.75 ms of the call's 5.68; now ~0.16 of 0.58.
// mode 0: B, and A unless the item marks it as packed; mode 1: A alone, marked or not.
// grid: (x: n_a + n_b row blocks, y: items)
constexpr int PREP_THREADS = 256;

template <class Z, int PREP_ROWS>
__global__ void __launch_bounds__(PREP_THREADS) k_zg_prep(const ZGemmItem* items, int n_items, int n_a, int mode,
                                                          int* status) {
  const int i = blockIdx.y;
  if (i >= n_items) return;
  const ZGemmItem it = items[i];
  const int which = (int)blockIdx.x < n_a ? 0 : 1;
  const int blk = which == 0 ? blockIdx.x : blockIdx.x - n_a, nblk = which == 0 ? n_a : gridDim.x - n_a;
  constexpr int ZNS = Z::NS;
  if (!item_live(it) || (which == 0 && it.skip_a > 0 && mode == 0)) return;
  if (!item_fits(it)) {
    if (blk == 0 && threadIdx.x == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  const int rows = which == 0 ? it.M : it.N, tr = which == 0 ? TMA : Z::TN;
  const PackCap cp = zcap<Z>(it, which);
  unsigned char* out = which == 0 ? it.TA : it.TB;
  int* ex = (int*)(out + cp.exp_off);
  const int n_ks = cdiv(it.K, ZG::KSTEP), n_grp = 2 * n_ks;
  // rows beyond the matrix in its last tile only reach product entries that are never written
  const int padded = cdiv(rows, PREP_ROWS) * PREP_ROWS;
  const bool k_contiguous = which == 0 ? it.opA != ZOP_N : it.opB == ZOP_N;
  const bool conj_op = (which == 0 ? it.opA : it.opB) == ZOP_C;
  const double2* src = which == 0 ? it.A : it.B;
  const size_t ld = which == 0 ? it.lda : it.ldb;
  // the first entry of row r of opA(A) (rows from a_split on come from A2) or column r of opB(B)
  auto row_ptr = [&](int r) {
    const double2* base = src;
    if (which == 0 && it.A2 && r >= it.a_split) {
      base = it.A2;
      r -= it.a_split;
    } else if (which == 1 && it.bcol) {
      r = it.bcol[r];
    }
    return base + (size_t)r * (k_contiguous ? ld : 1);
  };
  __shared__ unsigned long long part[PREP_THREADS / PREP_ROWS][PREP_ROWS];
  __shared__ int s_e[PREP_ROWS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int r0 = blk * PREP_ROWS; r0 < padded; r0 += nblk * PREP_ROWS) {
    if (k_contiguous) {
      // one warp per row, lanes along K
#pragma unroll
      for (int rr = warp; rr < PREP_ROWS; rr += PREP_THREADS / 32) {
        const int r = r0 + rr;
        unsigned long long m = 0;
        if (r < rows) {
          const double2* p = row_ptr(r);
          for (int k = lane; k < it.K; k += 32) {
            const double2 v = p[k];
            m = max(m, max(mag_bits(v.x), mag_bits(v.y)));
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) s_e[rr] = row_exponent(__longlong_as_double((long long)m));
      }
    } else {
      // rows contiguous: the block's rows by 256 / rows columns per pass
      const int r = r0 + (tid % PREP_ROWS);
      unsigned long long m = 0;
      if (r < rows) {
        const double2* p = row_ptr(r);
        for (int k = tid / PREP_ROWS; k < it.K; k += PREP_THREADS / PREP_ROWS) {
          const double2 v = p[(size_t)k * ld];
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
    const int planes = which == 0 ? 2 * ZNS : 3 * ZNS;
    unsigned char* tile = out + (size_t)rt * cp.ksteps * planes * cp.plane_bytes;
    for (int idx = tid; idx < PREP_ROWS * n_grp; idx += PREP_THREADS) {
      const int rr = idx % PREP_ROWS, grp = idx / PREP_ROWS;
      const int r = r0 + rr, k0 = grp * ZG::KG, e = s_e[rr];
      const size_t st = k_contiguous ? 1 : ld;
      const double2* p = row_ptr(min(r, rows - 1)) + (size_t)k0 * st;
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
      unsigned char* base = tile + (size_t)(grp >> 1) * planes * cp.plane_bytes + sw32_offset(m0 + rr, grp & 1);
      auto put = [&](int plane, const uint32_t* v, uint32_t flip) {
        *(uint4*)(base + (size_t)plane * cp.plane_bytes) = make_uint4(v[0] ^ flip, v[1] ^ flip, v[2] ^ flip, v[3] ^ flip);
      };
#pragma unroll
      for (int s = 0; s < ZNS; ++s) {
        if (which == 0) {
          put(s, pr[s], 0);
          put(ZNS + s, pi[s], 0);
        } else {                                 // (-Bi, Br, Bi)
          put(3 * s, pi[s], 0x80008000u);
          put(3 * s + 1, pr[s], 0);
          put(3 * s + 2, pi[s], 0);
        }
      }
    }
    __syncthreads();
  }
}

// The GEMM: persistent, one CTA per SM over the live 128 x TN tiles of every item. K runs in chunks
// of KC MMA steps: each chunk's levels accumulate exactly enough in TMEM, and the
// epilogue adds the chunk to C in FP64 (the first chunk writes C, or C - product for acc < 0). An item with a
// split stride has its chunks as separate units of work, chunk c written to C + c split (the caller adds them).
//
// Warps 0 .. 7 read the accumulators back (32 rows and half of the columns each), warp 8 copies the operands'
// planes in (two stages), warp 9 issues the MMAs; the copies run ahead of the MMAs and through the epilogues. One thread that issued both, the copy of a step
// after the MMAs of the step before, left the tensor cores idle for the copy: 9200 cycles per K step of Z6. With the
// roles apart, B's planes stacked and the entries' sums on eight warps the calls went from 0.93 to 0.58 ms (ten
// 1120 x 160 x 1120 products, GEMM 0.91 -> 0.42 ms), 1.54 to 0.72 (21 of 16384 x 64 x 64) and 0.24 to 0.15 (three
// of 300 x 70 x 530). What is left there: an MMA of 128 x 128 x 16 takes 66 cycles (53 up to 64 columns), the epilogue.
constexpr int EPI_WARPS = 8, GEMM_THREADS = 32 * (EPI_WARPS + 2);

template <class Z>
__global__ void __launch_bounds__(GEMM_THREADS, 1) k_zgemm(const ZGemmItem* items, int n_items, int* status) {
  constexpr int ZNS = Z::NS, TN = Z::TN, KC = Z::KC, NLEV = Z::NLEV, STAGES = 2;
  constexpr uint32_t A_PLANE = TMA * ROW_BYTES, B_PLANE = TN * ROW_BYTES;
  constexpr uint32_t A_STAGE = 2 * ZNS * A_PLANE, B_STAGE = 3 * ZNS * B_PLANE, STAGE = A_STAGE + B_STAGE;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint64_t bar_full[STAGES], bar_empty[STAGES], bar_acc, bar_read;
  __shared__ uint32_t tmem_base_s;
  __shared__ int tile_off[MAX_ITEMS + 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (n_items > MAX_ITEMS) {
    if (blockIdx.x == 0 && tid == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  auto chunk_ks = [](const ZGemmItem& it) { return it.split_ks > 0 ? min(it.split_ks, KC) : KC; };
  auto n_chunks = [&](const ZGemmItem& it) { return it.split > 0 ? cdiv(cdiv(it.K, ZG::KSTEP), chunk_ks(it)) : 1; };
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  for (int i = tid; i < n_items; i += blockDim.x) {
    const ZGemmItem& it = items[i];
    tile_off[i + 1] = (item_live(it) && item_fits(it)) ? cdiv(it.M, TMA) * cdiv(it.N, TN) * n_chunks(it) : 0;
  }
  if (tid == 0) {
    tile_off[0] = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&bar_full[s], 1);
      mbar_init(&bar_empty[s], 1);
    }
    mbar_init(&bar_acc, 1);
    mbar_init(&bar_read, EPI_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp == 0) {
    // inclusive prefix of the unit counts
    int run = 0;
    for (int i0 = 0; i0 < n_items; i0 += 32) {
      int v = i0 + lane < n_items ? tile_off[i0 + lane + 1] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
      }
      if (i0 + lane < n_items) tile_off[i0 + lane + 1] = run + v;
      run += __shfl_sync(0xffffffffu, v, 31);
    }
  }
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
  // unit t: its item, tile and K steps
  struct Unit {
    const ZGemmItem* it;
    int rt, ct, ks_from, ks_to, chunk;
  };
  auto unit_of = [&](int t) {
    int lo = 0, hi = n_items - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (tile_off[mid] <= t) lo = mid;
      else hi = mid - 1;
    }
    Unit U;
    U.it = items + lo;
    const int nt_b = cdiv(U.it->N, TN), nch = n_chunks(*U.it), unit = t - tile_off[lo], tile = unit / nch;
    U.chunk = unit - tile * nch;
    U.rt = tile / nt_b;
    U.ct = tile % nt_b;
    const int n_ks = cdiv(U.it->K, ZG::KSTEP);
    U.ks_from = U.it->split > 0 ? U.chunk * chunk_ks(*U.it) : 0;
    U.ks_to = U.it->split > 0 ? min(n_ks, U.ks_from + chunk_ks(*U.it)) : n_ks;
    return U;
  };
  bool ok = true;
  if (warp == EPI_WARPS) {
    if (lane == 0) {
      uint32_t g = 0;
      for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
        const Unit U = unit_of(t);
        const PackCap ca = zcap<Z>(*U.it, 0), cb = zcap<Z>(*U.it, 1);
        const unsigned char* gA = U.it->TA + (size_t)U.rt * ca.ksteps * A_STAGE;
        const unsigned char* gB = U.it->TB + (size_t)U.ct * cb.ksteps * B_STAGE;
        for (int ks = U.ks_from; ks < U.ks_to && ok; ++ks, ++g) {
          const uint32_t st = g % STAGES;
          if (g >= STAGES) ok = mbar_wait(&bar_empty[st], (g / STAGES - 1) & 1u);
          if (!ok) break;
          unsigned char* dst = smem + st * STAGE;
          mbar_expect_tx(&bar_full[st], STAGE);
          bulk_g2s(dst, gA + (size_t)ks * A_STAGE, A_STAGE, &bar_full[st]);
          bulk_g2s(dst + A_STAGE, gB + (size_t)ks * B_STAGE, B_STAGE, &bar_full[st]);
        }
      }
      // the copies in flight land before the CTA leaves (after a failure nobody else waits for them)
      for (uint32_t q = g > STAGES ? g - STAGES : 0; q < g; ++q) ok &= mbar_wait(&bar_full[q % STAGES], (q / STAGES) & 1u);
    }
  } else if (warp == EPI_WARPS + 1) {
    // the whole warp, one lane of which issues
    const bool one = elect_one();
    const uint32_t idesc = instr_desc(1u, TMA, 2 * TN);
    uint32_t g = 0, c = 0;
    for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
      const Unit U = unit_of(t);
      for (int ks0 = U.ks_from; ks0 < U.ks_to && ok; ks0 += KC, ++c) {
        if (c > 0) ok = __all_sync(0xffffffffu, mbar_wait(&bar_read, (c - 1) & 1u));     // the accumulators have been read
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int nk = min(KC, U.ks_to - ks0);
        for (int ks = 0; ks < nk; ++ks, ++g) {
          const uint32_t st = g % STAGES;
          ok = __all_sync(0xffffffffu, mbar_wait(&bar_full[st], (g / STAGES) & 1u));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const unsigned char* sa = smem + st * STAGE;
          mma_slices_stacked<ZNS, NLEV, TN, A_PLANE, B_PLANE>(one, tmem, smem_desc_sw32(sa), smem_desc_sw32(sa + A_STAGE),
                                                              idesc, ks > 0);
          if (one) mma_commit(&bar_empty[st]);
          __syncwarp();
        }
        if (ok && one) mma_commit(&bar_acc);
        __syncwarp();
      }
    }
    // MMAs in flight end before TMEM is freed
    if (!ok && g > 0) mbar_wait(&bar_empty[(g - 1) % STAGES], ((g - 1) / STAGES) & 1u);
  } else {
    uint32_t c = 0;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;      // a warp reads the lanes of its number mod 4
    const int c_from = (warp >> 2) * (TN / 2), c_to = c_from + TN / 2;
    for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
      const Unit U = unit_of(t);
      const ZGemmItem& it = *U.it;
      const PackCap ca = zcap<Z>(it, 0), cb = zcap<Z>(it, 1);
      double2* const C = it.C + (size_t)U.chunk * it.split;
      const int* col_exp = (const int*)(it.TB + cb.exp_off) + U.ct * TN;
      const int m = U.rt * TMA + (warp & 3) * 32 + lane;
      const int e_m = ((const int*)(it.TA + ca.exp_off))[m];
      bool bad = false;
      for (int ks0 = U.ks_from; ks0 < U.ks_to; ks0 += KC, ++c) {
        ok = mbar_wait(&bar_acc, c & 1u);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // thread = row m of the tile, 8 columns per TMEM load
        const bool add = ks0 > U.ks_from || it.acc < 0;
        for (int c0 = c_from; c0 < c_to; c0 += 8) {
          // the entries that the product is added to, on their way while the levels are read and added
          double2 o[8], v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int n = U.ct * TN + c0 + j;
            o[j] = (add && m < it.M && n < it.N) ? C[m + (size_t)n * it.ldc] : make_double2(0.0, 0.0);
          }
          float x[NLEV][8];
#pragma unroll
          for (int part = 0; part < 2; ++part) {
#pragma unroll
            for (int L = 0; L < NLEV; ++L) tmem_ld8_nowait(tmem + lane_base + (2 * L + part) * TN + c0, x[L]);
            tmem_wait_ld();
            if (part == 1 && c0 + 8 >= c_to) {
              // the last read of the chunk: the next chunk's MMAs may start
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0) mbar_arrive(&bar_read);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              double y = Z::value(x, j, e_m + col_exp[c0 + j], it.acc < 0);
              // a NaN or an infinity of an operand is a NaN in its slice 0, so in level 0
              if (!(fabsf(x[0][j]) < 1e30f)) y = __longlong_as_double(0x7ff8000000000000ll);
              (part ? v[j].y : v[j].x) = y;
            }
          }
          if (m < it.M) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int n = U.ct * TN + c0 + j;
              if (n >= it.N) continue;
              if (add) v[j] = make_double2(o[j].x + v[j].x, o[j].y + v[j].y);
              if (it.flag) bad |= !(isfinite(v[j].x) && isfinite(v[j].y));
              C[m + (size_t)n * it.ldc] = v[j];
            }
          }
        }
      }
      if (bad && it.flag) *it.flag = 1;
    }
  }
  if (!ok) atomicOr(status, ST_TIMEOUT);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

size_t zgemm_pack_bytes(int rows_cap, int k_cap, int which) {
  return pack_cap(std::max(1, rows_cap), std::max(1, k_cap), which == 0 ? TMA : Z6::TN, ZG::KSTEP, Z6::NS,
                  which == 0 ? 0 : 3 * Z6::NS).total;
}

size_t zgemm9_pack_bytes(int rows_cap, int k_cap, int which) {
  return pack_cap(std::max(1, rows_cap), std::max(1, k_cap), which == 0 ? TMA : Z9::TN, ZG::KSTEP, Z9::NS,
                  which == 0 ? 0 : 3 * Z9::NS).total;
}


int zgemm_max_items() { return MAX_ITEMS; }

int zgemm_tile_cap(int m_cap, int n_cap) { return cdiv(std::max(1, m_cap), TMA) * cdiv(std::max(1, n_cap), Z6::TN); }

namespace {
constexpr int ZMAX_DEV = 64;
std::once_flag g_zattr[ZMAX_DEV][2];        // the shared-memory limit is set once per device

template <class Z>
void launch_prep(const ZGemmItem* items, int n_items, int m_cap_max, int n_cap_max, int k_cap_max, int mode, int* status,
                 cudaStream_t st) {
  const int rows = k_cap_max <= 64 ? 32 : 8;
  const int n_a = std::min(2048, cdiv(std::max(1, m_cap_max), rows));
  const int n_b = mode == 1 ? 0 : std::min(2048, cdiv(std::max(1, n_cap_max), rows));
  const dim3 grid(n_a + n_b, n_items);
  if (rows == 32) k_zg_prep<Z, 32><<<grid, PREP_THREADS, 0, st>>>(items, n_items, n_a, mode, status);
  else k_zg_prep<Z, 8><<<grid, PREP_THREADS, 0, st>>>(items, n_items, n_a, mode, status);
}

template <class Z>
void launch_gemm(const ZGemmItem* items, int n_items, long long unit_cap, int* status, cudaStream_t st) {
  const size_t smem = (size_t)2 * Z::NS * (2 * TMA + 3 * Z::TN) * ROW_BYTES + 1024;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (dev >= 0 && dev < ZMAX_DEV)
    std::call_once(g_zattr[dev][Z::NS == 9], [smem] {
      cudaFuncSetAttribute(k_zgemm<Z>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
  const int grid = (int)std::max<long long>(1, std::min<long long>(sms > 0 ? sms : 152, unit_cap));
  k_zgemm<Z><<<grid, GEMM_THREADS, smem, st>>>(items, n_items, status);
}
}  // namespace

void launch_zgemm_pack_a(const ZGemmItem* items, int n_items, int m_cap_max, int* status, cudaStream_t st) {
  if (n_items <= 0) return;
  launch_prep<Z6>(items, n_items, m_cap_max, 0, INT_MAX, 1, status, st);
}

void launch_zgemm(const ZGemmItem* items, int n_items, int tile_cap, int m_cap_max, int n_cap_max, int* status,
                  cudaStream_t st, int k_cap_max) {
  if (n_items <= 0) return;
  launch_prep<Z6>(items, n_items, m_cap_max, n_cap_max, k_cap_max, 0, status, st);
  launch_gemm<Z6>(items, n_items, tile_cap, status, st);
}

void launch_zgemm9(const ZGemmItem* items, int n_items, long long unit_cap, int m_cap_max, int n_cap_max, int k_cap_max,
                   int* status, cudaStream_t st) {
  if (n_items <= 0) return;
  launch_prep<Z9>(items, n_items, m_cap_max, n_cap_max, k_cap_max, 0, status, st);
  launch_gemm<Z9>(items, n_items, unit_cap, status, st);
}

}  // namespace ptk
