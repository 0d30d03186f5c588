// Whole-GPU one-sided Jacobi SVD for all bond matrices of one layer (App. A.2).
//
// What bounds it: GB300 issues one FP64 instruction per warp every 64 cycles and sub-partition, whatever the
// number of active lanes (measured; 19 cycles per SM with all four busy), with a latency of 64 cycles, and a
// grid barrier costs ~2400 cycles. A rotation's scalars (one lane's chain of ~30 FP64 operations) and the
// barriers therefore cost as much as the arithmetic on columns of a few hundred rows. So:
//   * the columns are grouped in blocks of b and a round-robin tournament runs over the blocks: one CTA holds
//     a pair of blocks (2 b columns) in shared memory and runs its b x b cross pairs (in the first round of a
//     sweep also the pairs inside the blocks) in sub-rounds of b disjoint pairs;
//   * a task waits for its two blocks only: each block carries the number of rounds it has been through
//     (BondWork::rounds), stored after its columns and polled by the next task that needs it. A grid barrier per round
//     instead, with its column transfers, took 8000 of the 14000 cycles of a round with b = 2; grid barriers remain
//     at the end of a sweep;
//   * the scalars of a sub-round's pairs are computed by the lanes of one extra warp at the same time. Columns
//     carry a real scale (column = d x stored column, q = d^2), so that neither a square root nor a division is
//     needed: with rho = tan / |gamma| (in FP32 and integers: a rotation by an angle that is 1e-7 off is still
//     unitary and leaves 1e-7 of the pair's inner product to the next sweep) the stored columns become
//     x - conj(mu) y and y + nu x, mu = rho q_y g, nu = rho q_x g, g = x^H y of the stored columns, and
//     q_x, q_y are multiplied by cos^2 = 1 / (1 + tan^2). That is 9 FP64 operations before the columns can be
//     rotated; the new norms and scales are formed while they are. A row costs 8 FP64 operations, not 12;
//   * inner products are summed over lanes and warps in 64-bit fixed point (to_fixed below): the butterflies were six of
//     the eighteen FP64 instructions that a warp with one row per lane issues per pair;
//   * a CTA has two such task slots of 8 + 1 warps (named barriers), so one's scalars overlap the other's
//     columns; tasks fill one slot of every SM before the second;
//   * b is chosen on the device from the live dims by a cost model of these terms (choose_block), and CTAs that
//     no round can use leave at once, so small layers pay for small barriers.
// Before (one 512-thread CTA per SM, b = 2, columns in L2, each pair's scalars on one lane in FP64 with two sqrt /
// rsqrt chains, 5800 cycles; now 1900) -> with a grid barrier per round -> with the blocks' own counters and a pair's two
// norms, scales and factors on two lanes -> with fixed-point sums, no divisions and a fitted choice of b: two 256 x 256
// SVDs without QRs before them 112 ms (clusters) -> 31.6 -> 27.9 -> 27; the five-site chain's first eight steps 219 -> 180
// -> 150 -> (with the new pivoted QR 131) 117 ms, the 16 chains' first four 300 -> 177 -> 176 -> (138) 118 ms, the 21-site
// chain's first four on the tensor-core path 990 -> 451 -> 438 -> (417) 414 ms. A sweep now: 64 x 64 0.16 ms, two 136 x
// 136 0.48, 64 of 80 x 80 0.72, two 256 x 256 with V 1.3.
//
// Sums are combined in a fixed order, so results are bitwise reproducible. Every barrier wait has a time
// limit: on expiry the kernel records ST_TIMEOUT, raises an abort flag that releases every other CTA, and
// returns.
//
// on_b = 1: the matrix is R^H left by the pivoted QR (qrcp.cu); only its left vectors are wanted there, so
// the right factor is not accumulated. on_b = 2: R^H of the l x l triangular factor R in G64 of the fast path's
// randomized range finder (rsvd.cu), formed in V: its columns (R's rows) are graded and close to orthogonal, so ~40%
// fewer pairs rotate than on R (CPU emulation, bonds of a nine-site chain), and the other factor follows from R and
// the left vectors. on_b = 0: the matrix in A (the standalone SVD).
#include <algorithm>

#include "grid_sync.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace ptk {

namespace {

constexpr int JG = 2;                      // task slots per CTA
constexpr int JW = 8;                      // column warps of a slot: JW / b per pair
constexpr int JT = 32 * (JW + 1);          // threads of a slot: the last warp computes the scalars
constexpr int CT = JG * JT, CW = CT / 32;  // threads and warps per CTA
constexpr int JB = 8;                      // largest block
constexpr int MAX_ITEMS = 1024;
constexpr double UNIT = 1.1102230246251565e-16;

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the 32 lanes of two values at once (a reduce-scatter butterfly): lane 0 ends with the
// total of a, lane 16 with the total of b; 5 shuffles and 5 adds instead of 10 and 10.
__device__ __forceinline__ double wsum2(double a, double b, int lane) {
  const bool hi = (lane & 16) != 0;
  double keep = hi ? b : a;
  keep += __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, o);
  return keep;
}

__device__ __forceinline__ void item_shape(const BondWork& W, int* Ma, int* Na) {
  const int mD = W.info[0], nD = W.info[1];
  const bool tr = W.info[2] != 0;
  *Ma = (mD > 0 && nD > 0) ? (tr ? nD : mD) : 0;
  *Na = (mD > 0 && nD > 0) ? (tr ? mD : nD) : 0;
}

__device__ __forceinline__ void slot_sync(int grp) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(JT) : "memory");
}

__device__ __forceinline__ double2* mat_of(const BondWork& W, int on_b) {
  return on_b == 0 ? W.A : (on_b == 1 ? W.G64 : W.V);
}

__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// the first 24 bits of a positive double's significand as a float in [1, 2), and its exponent
__device__ __forceinline__ float significand(double x, int* e) {
  const int hi = __double2hiint(x);
  *e = ((hi >> 20) & 0x7ff) - 1023;
  return __int_as_float(0x3f800000 | (hi & 0xfffff) << 3 | (int)((unsigned)__double2loint(x) >> 29));
}

// Sums over the lanes and warps as 64-bit fixed-point numbers. With E = pair_exponent, |x| |y| < 2^E for the stored
// columns, so by Cauchy-Schwarz every partial inner product is below 2^E too and so are sums of their magnitudes: at 57
// fractional bits below 2^E the sums need no further headroom, their error (2^-57 of |x| |y| per lane) is below that of
// FP64 sums, and 5 bits remain for norms that are off (closed forms between two exact ones).
__device__ __forceinline__ int exponent_of(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1023; }

__device__ __forceinline__ int pair_exponent(double al, double be, double qx, double qy) {
  return (exponent_of(al) + exponent_of(be) - exponent_of(qx) - exponent_of(qy) + 3) >> 1;
}

// Squared norms, inner products and thresholds of an item are in units of 2^norm_exponent(||A||_F^2), so that |gamma|^2 and
// norm^2 stay in range whatever the matrix' scale (without, columns of norm 1e-76 or 1e76 were left as they were)
__device__ __forceinline__ int norm_exponent(double fro2) { return max(-1022, min(1022, exponent_of(fro2))); }
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }       // |e| <= 1022

// x in units of 2^(E - 57), truncated; 0 if not finite or out of range
__device__ __forceinline__ long long to_fixed(double x, int E) {
  const long long b = __double_as_longlong(x);
  const int e = exponent_of(x), sh = e - E + 5;
  long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
  m = sh >= 0 ? m << min(sh, 63) : m >> min(-sh, 63);
  if (sh > 9 || e < -1022 || e > 1023) m = 0;
  return b < 0 ? -m : m;
}

// the sum of v over the lanes, in every lane: 21 + 21 + 22 bits by the integer reduction of a warp
__device__ __forceinline__ long long lane_sum(long long v) {
  const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)v & 0x1fffffu);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 21) & 0x1fffffu);
  const int l2 = (int)__reduce_add_sync(0xffffffffu, (unsigned)(int)(v >> 42));
  return (long long)l0 + ((long long)l1 << 21) + ((long long)l2 << 42);
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// f 2^k, f in [1, 2), 0 for k below -60 (k <= 1)
__device__ __forceinline__ float scale_pow2(float f, int k) {
  return k < -60 ? 0.f : __int_as_float(__float_as_int(f) + (k << 23));
}

// shared-memory tables of a launch over n items
__host__ __device__ constexpr int header_bytes(int n) { return (48 * n + 4 * (5 * n + 1) + 15) & ~15; }

__device__ __forceinline__ int load_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void store_relaxed(int* p, int v) {
  asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

constexpr int MIN_SCALE_HI = (1023 - 64) << 20;    // below 2^-64 a squared scale is multiplied into its column

// columns per block: the b in {1, 2, 4, 8} that fits cols_max columns and whose sweep is shortest by the cost of
// its terms in cycles: per sub-round the scalars and reductions (2000 cycles, shared by the tasks of an SM) and 13.5
// cycles per FP64 warp instruction of the SM's tasks; per round the waits and lookups (6100) and the transfer of a task's
// columns (2.6 per row). The constants are fitted to the time of a sweep at every b, measured for 16 x 16, two 32 x 32, 64 x
// 64 (1 and 24), 100 x 100 (2), 136 x 136 (2), 80 x 80 (64), 160 x 160 (10) and, with V, 128 x 128 and 256 x 256 (2): the
// model finds the shortest one in each. An estimate from the issue rate alone (19 cycles, 2500 and 3500) took b = 2 for
// ten 160 x 160 (1.31 ms a sweep, 0.75 at b = 8) and for one 64 x 64 (0.19, 0.16 at b = 4).
// One warp computes it; every lane gets the result.
__device__ int choose_block(const int* s_Na, const int* s_Ma, int n_work, int slots, int sms, int cols_max,
                            bool with_v, int lane) {
  int best = 1;
  float best_t = 3e38f;
  for (int b = 1; b <= JB && 2 * b <= cols_max; b <<= 1) {
    int tasks = 0, rounds = 0, rows = 0, len = 0, most_nb = 0;
    for (int w = lane; w < n_work; w += 32) {
      if (s_Na[w] < 2) continue;
      const int nb = (s_Na[w] + b - 1) / b, nbp = nb + (nb & 1);
      most_nb = max(most_nb, nb);
      tasks += nbp / 2;
      rounds = max(rounds, nbp - 1);
      // FP64 operations per pair: 4 per row for the inner product, 8 per row (and row of V) for the rotation
      rows = max(rows, 12 * s_Ma[w] + (with_v ? 8 * s_Na[w] : 0));
      len = max(len, s_Ma[w] + (with_v ? s_Na[w] : 0));
    }
    tasks = __reduce_add_sync(0xffffffffu, tasks);
    rounds = __reduce_max_sync(0xffffffffu, rounds);
    rows = __reduce_max_sync(0xffffffffu, rows);
    len = __reduce_max_sync(0xffffffffu, len);
    most_nb = __reduce_max_sync(0xffffffffu, most_nb);
    if (tasks == 0) return 1;
    const float per_sm = (float)((tasks + sms - 1) / sms), waves = (float)((tasks + slots - 1) / slots);
    const float fp = 13.5f * b * (float)rows * (1.f / 32.f);
    const float sub = fmaxf(waves * 2000.f + fp, per_sm * fp + 2000.f);
    const float move = waves * 6100.f + per_sm * b * (float)len * 2.6f;
    // one block only: no cross pairs
    const float t = most_nb < 2 ? (b - 1) * sub : rounds * ((float)b * sub + move) + (b - 1) * sub;
    if (t < best_t) {
      best_t = t;
      best = b;
    }
  }
  return best;
}

}  // namespace

// One-sided Jacobi over all matrices of a layer in FP64. with_v: accumulate the right factor V from V = I.
// tol_scale: a pair rotates while |a_i^H a_j| > tol_scale * unit roundoff * |a_i| |a_j| (0: the row count m).
// Columns whose squared norm is at floor2 ||A||_F^2 or below are not rotated: they cannot become orthogonal
// relative to their own norm and carry no information at that precision. Squared column norms (in the item's unit) live
// in aux, squared scales in sig, rotation counters in info[4..5], sweeps go to info[3]. SM: the columns fit in shared memory (cols_max
// of them); otherwise a pair's columns are read from and written to L2 (b = 1).
template <bool SM>
__global__ void __launch_bounds__(CT, 1)
    k_jacobi_grid(const BondWork* work, int n_work, int max_sweeps, GridSync gs, int* status, int on_b, int with_v,
                  double tol_scale, double floor2, int n_grp, int dyn_bytes) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  // of one task slot
  struct Slot {
    double part[JW][2];
    double rot[JB][4];                     // mu, nu of each pair
    double nrm[2 * JB], q[2 * JB];         // squared norms and squared scales of the task's columns
    int flag[JB];                          // rotate
    int redo[JB];                          // recompute the pair's norms from its columns
    int rotc[2 * JB];                      // the column changed in this task
    int cnt, renorm[2], lost[2];
  };
  __shared__ Slot s_slot[JG];
  __shared__ int s_b, s_rounds, s_fit, s_most, s_cols;
  __shared__ long long s_limit;            // wait limit: the launch's, and what a sweep can take
  const int ctid = threadIdx.x, grp = ctid / JT, tid = ctid % JT, lane = tid & 31, wid = tid >> 5, cwid = ctid >> 5;
  Slot& S = s_slot[grp];
  if (n_work > MAX_ITEMS) {
    if (blockIdx.x == 0 && ctid == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  double* s_fro = (double*)s_raw;                    // ||A||_F^2 per item, in units of 2^s_exp
  double2** s_A = (double2**)(s_fro + n_work);       // the items' buffers (the work list itself is behind two loads)
  double2** s_V = s_A + n_work;
  double** s_aux = (double**)(s_V + n_work);
  double** s_sig = s_aux + n_work;
  int** s_ver = (int**)(s_sig + n_work);
  int* s_Na = (int*)(s_ver + n_work);                // columns that are rotated
  int* s_Ma = s_Na + n_work;                         // rows
  int* s_off = s_Ma + n_work;                        // [n_work + 1] prefix of the sweep's tasks per round
  int* s_act = s_off + n_work + 1;
  int* s_exp = s_act + n_work;                       // norm_exponent of ||A||_F^2
  const int hdr = header_bytes(n_work);
  const int slot_bytes = (dyn_bytes - hdr) / n_grp & ~15;
  double2* s_col = (double2*)(s_raw + hdr + (size_t)grp * slot_bytes);
  for (int w = ctid; w < n_work; w += CT) {
    int Ma, Na;
    item_shape(work[w], &Ma, &Na);
    // on_b = 1: B = R^H of the pivoted QR (G64), Na rows and k = info[8] columns (the QR's rank);
    // on_b = 2: R^H of the range finder's small square factor (in V), l = info[9] rows and columns
    const int kq = on_b == 1 ? max(0, min(work[w].info[8], Na)) : (on_b == 2 ? max(0, min(work[w].info[9], Na)) : Na);
    s_Na[w] = kq;
    s_Ma[w] = on_b == 1 ? Na : (on_b == 2 ? kq : Ma);
    s_act[w] = kq >= 2;
    s_A[w] = mat_of(work[w], on_b);
    s_V[w] = work[w].V;
    s_aux[w] = work[w].aux;
    s_sig[w] = work[w].sig;
    s_ver[w] = work[w].rounds;
  }
  __syncthreads();
  if (cwid == 0) {
    int rows = 0;
    for (int w = lane; w < n_work; w += 32) rows = max(rows, s_Ma[w] + (with_v ? s_Na[w] : 0));
    rows = __reduce_max_sync(0xffffffffu, rows);
    const int fit = SM ? (rows > 0 ? slot_bytes / (16 * rows) : 2) : 2;
    const int b = SM ? choose_block(s_Na, s_Ma, n_work, n_grp * gridDim.x, gridDim.x, fit, with_v != 0, lane) : 1;
    int most = 0, cols = 0, nbs = 0;
    for (int w = lane; w < n_work; w += 32) {
      const int nb = (s_Na[w] + b - 1) / b, nbp = nb + (nb & 1);
      if (s_Na[w] >= 2) most += nbp / 2;
      cols += s_Na[w];
      nbs = max(nbs, nbp);
    }
    most = __reduce_add_sync(0xffffffffu, most);
    cols = __reduce_add_sync(0xffffffffu, cols);
    nbs = __reduce_max_sync(0xffffffffu, nbs);
    if (lane == 0) {
      s_fit = fit;
      s_b = b;
      s_most = most;
      s_cols = cols;
      // a CTA without tasks (its items have converged) waits for a whole sweep of the others: rounds x a slot's tasks x up
      // to 2 b sub-rounds of b pairs, at most 64 cycles per row and pair (twelve FP64 instructions of two slots at the issue
      // rate are 24, columns from memory 15) and what does not depend on the rows
      const long long turns = most / (n_grp * (int)gridDim.x) + 1;
      s_limit = gs.limit + nbs * turns * 2 * b * (64LL * b * rows + 20000);
    }
  }
  __syncthreads();
  if (s_fit < 2) {                         // the host sized the buffer for the capacities: cannot happen
    if (blockIdx.x == 0 && ctid == 0) atomicOr(status, ST_CAPACITY);
    return;
  }
  const int b = s_b, lb = __ffs(b) - 1, wpp = JW >> lb, lw = __ffs(wpp) - 1;      // warps per pair; logarithms
  // CTAs that take part: as many as a round has tasks (and the passes over all columns can use)
  const int G = max(1, min((int)gridDim.x, max(s_most, min((s_cols + 15) / 16, 152))));
  if ((int)blockIdx.x >= G) return;
  auto barrier = [&]() { return grid_barrier(GridSync{gs.count, gs.abort, s_limit}, status, G); };
  // V = I, zero counters, unit scales, column norms
  {
    const int gt = blockIdx.x * CT + ctid, ngt = G * CT;
    const int gwarp = cwid * G + blockIdx.x, ngwarp = G * CW;
    int base = 0;
    for (int w = 0; w < n_work; ++w) {
      const BondWork& W = work[w];
      const int Ma = s_Ma[w], Na = s_Na[w];
      if (with_v)
        for (size_t idx = gt; idx < (size_t)Na * Na; idx += ngt)
          __stcg(W.V + idx, make_double2((idx % Na) == (idx / Na) ? 1.0 : 0.0, 0.0));
      if (gt == 0) {
        W.info[4] = 0;
        W.info[5] = 0;
      }
      double2* A = mat_of(W, on_b);
      for (int c = gwarp - base; c < Na; c += ngwarp) {
        if (c < 0) continue;
        double2* a = A + (size_t)c * Ma;
        double s2 = 0;
        for (int r = lane; r < Ma; r += 32) {
          double2 x = make_double2(0.0, 0.0);
          if (on_b != 2) {
            x = __ldcg(a + r);
          } else {
            if (r >= c) {
              const double2 y = __ldcg(W.G64 + c + (size_t)r * Ma);
              x = make_double2(y.x, -y.y);
            }
            __stcg(a + r, x);
          }
          s2 = fma(x.x, x.x, fma(x.y, x.y, s2));
        }
        s2 = wsum(s2);
        if (lane == 0) {
          __stcg(W.aux + c, s2);
          __stcg(W.sig + c, 1.0);
          __stcg(W.rounds + c, 0);         // of block c (blocks are fewer than columns)
        }
      }
      base = (base + Na) % ngwarp;
    }
  }
  if (!barrier()) return;
  // ||A||_F^2 per item, summed in the same fixed order by every CTA
  for (int w = cwid; w < n_work; w += CW) {
    double acc = 0;
    for (int k = lane; k < s_Na[w]; k += 32) acc += __ldcg(work[w].aux + k);
    acc = wsum(acc);
    if (lane == 0) {
      const int e = norm_exponent(acc);
      s_fro[w] = acc * pow2(-e);
      s_exp[w] = e;
    }
  }
  // the rounds of the next sweep, the longest tournament among the active items (0: all converged), and the prefix of
  // the active items' task counts
  auto set_rounds = [&]() {
    if (cwid != 0) return;
    int rounds = 0, run = 0;
    for (int w0 = 0; w0 < n_work; w0 += 32) {
      const int w = w0 + lane;
      int v = 0;
      if (w < n_work && s_act[w]) {
        const int nb = (s_Na[w] + b - 1) / b, nbp = nb + (nb & 1);
        rounds = max(rounds, nbp - 1);
        v = nbp / 2;
      }
      int inc = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
      }
      if (w < n_work) s_off[w] = run + inc - v;
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
    rounds = __reduce_max_sync(0xffffffffu, rounds);
    if (lane == 0) {
      s_off[n_work] = run;
      s_rounds = rounds;
    }
  };
  set_rounds();
  __syncthreads();
  int sweep = 0;
  while (s_rounds > 0 && sweep < max_sweeps) {
    const int par = sweep & 1, rounds = s_rounds;
    if (blockIdx.x == 0)
      for (int w = ctid; w < n_work; w += CT) work[w].info[4 + (par ^ 1)] = 0;
    const int total = s_off[n_work];
    bool gone = false;                     // a wait ran out (this slot or another CTA): to the barrier, which fails
    for (int round = 0; round < rounds && !gone; ++round) {
      for (int t = grp < n_grp ? grp * G + (int)blockIdx.x : total; t < total; t += n_grp * G) {
        int lo = 0, hi = n_work - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (s_off[mid] <= t) lo = mid;
          else hi = mid - 1;
        }
        const int w = lo, q = t - s_off[w];
        const int Ma = s_Ma[w], Na = s_Na[w], Vr = with_v ? Na : 0, ld = Ma + Vr;
        const int nb = (Na + b - 1) >> lb, nbp = nb + (nb & 1), m1 = nbp - 1;
        if (round >= m1) continue;    // this item's tournament is over
        int bi, bj;
        if (q == 0) { bi = nbp - 1; bj = round; }
        else {                             // (round +- q) mod (nbp - 1); a division takes as long as an inner product
          bi = round + q < m1 ? round + q : round + q - m1;
          bj = round >= q ? round - q : round - q + m1;
        }
        double2 *A = s_A[w], *V = s_V[w];
        double *aux = s_aux[w], *sig = s_sig[w];
        const int ex = s_exp[w];
        const double unit = pow2(-ex);
        // local column c: global column of block bi (c < b) or bj; -1 beyond the matrix
        auto gcol = [&](int c) {
          const int g = (c < b ? bi * b + c : bj * b + c - b);
          return g < Na ? g : -1;
        };
        // both blocks have been through the rounds before this one
        const int need = sweep * (nbp - 1) + round;
        int* ver = s_ver[w];
        if (wid == JW && lane < 2) {
          const int blk = lane == 0 ? bi : bj;
          bool lost = false;
          if (blk < nb && need > 0) {
            const long long t0 = clock64();
            for (int it = 1; load_acquire(ver + blk) < need; ++it) {
              if ((it & 63) != 0) continue;
              if (*(volatile int*)gs.abort) lost = true;
              else if (clock64() - t0 > s_limit) {
                atomicOr(status, ST_TIMEOUT);
                atomicExch(gs.abort, 1);
                lost = true;
              }
              if (lost) break;
            }
          }
          S.lost[lane] = lost;
        }
        slot_sync(grp);
        gone = S.lost[0] || S.lost[1];
        if (gone) break;
        if (tid < 2 * b) {
          const int g = gcol(tid);
          S.nrm[tid] = g >= 0 ? __ldcg(aux + g) : 0.0;
          S.q[tid] = g >= 0 ? __ldcg(sig + g) : 1.0;
          S.rotc[tid] = 0;
        }
        if (tid == 0) S.cnt = 0;
        // the column warps share the 2 b columns evenly: JW / 2b warps per column, or two columns per warp
        const int lc = max(0, lw - 1), wpc = 1 << lc, c0 = wid >> lc, rc0 = (wid & (wpc - 1)) * 32 + lane;
        if (SM) {
          for (int c = c0; c < 2 * b && wid < JW; c += JW) {
            const int g = gcol(c);
            if (g < 0) continue;
            const double2* a = A + (size_t)g * Ma;
            const double2* v = V + (size_t)g * Na - Ma;
            double2* dst = s_col + (size_t)c * ld;
#pragma unroll 4
            for (int r = rc0; r < ld; r += 32 * wpc) cp16(dst + r, (r < Ma ? a : v) + r);
          }
          asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
        }
        slot_sync(grp);
        if (round == 0) {
          // once a sweep the norms from the columns (2 b of them, wpc warps or half a warp's turn each): a closed-form
          // norm keeps the rounding error of the norms it came from, which a column that has shrunk by several
          // rotations to the level of rounding does not bear
          double na = 0, nb2 = 0;
          if (wid < JW) {
            const int g0 = gcol(c0), g1 = wpp > 1 ? -1 : gcol(c0 + JW);
            auto norm2 = [&](int c, int g) {
              const double2* a = SM ? s_col + (size_t)c * ld : A + (size_t)g * Ma;
              double v = 0;
              for (int r = rc0; r < Ma; r += 32 * wpc) {
                const double2 u = SM ? a[r] : __ldcg(a + r);
                v = fma(u.x, u.x, fma(u.y, u.y, v));
              }
              return v;
            };
            if (g0 >= 0) na = norm2(c0, g0);
            if (g1 >= 0) nb2 = norm2(c0 + JW, g1);
            __syncwarp();
            const double s = wsum2(na, nb2, lane);
            if ((lane & 15) == 0) S.part[wid][lane >> 4] = s;
          }
          slot_sync(grp);
          if (tid < 2 * b) {
            double s = 0;
            if (wpp > 1)
              for (int k = 0; k < wpc; ++k) s += S.part[tid * wpc + k][0];
            else
              s = S.part[tid & (JW - 1)][tid / JW];
            S.nrm[tid] = s * unit * S.q[tid];
          }
          slot_sync(grp);
        }
        // noise floor as the bits of a non-negative double; significand and exponent of the squared threshold
        const long long fl2 = __double_as_longlong(floor2 * s_fro[w]);
        const double tol = (tol_scale > 0 ? tol_scale : (double)Ma) * UNIT;
        int et;
        const float tm = significand(tol * tol, &et);
        const int n_inner = round == 0 ? b - 1 : 0;
        const int n_cross = bi < nb && bj < nb ? b : 0;       // none against the padding block
        for (int sr = 0; sr < n_inner + n_cross; ++sr) {
          const int p = wid >> lw, gw = wid & (wpp - 1);
          // pair p's local columns: inside a block (round-robin over its b columns) or across the two
          auto pair_of = [&](int pp, int* i, int* j) {
            if (sr < n_inner) {
              const int h = b >> 1, blk = pp >= h, x = pp - blk * h;
              int u, v;
              if (x == 0) { u = b - 1; v = sr; }
              else {
                u = sr + x < b - 1 ? sr + x : sr + x - (b - 1);
                v = sr >= x ? sr - x : sr - x + b - 1;
              }
              *i = blk * b + min(u, v);
              *j = blk * b + max(u, v);
            } else {
              *i = pp;
              *j = b + ((pp + sr - n_inner) & (b - 1));
            }
          };
          int li = 0, lj = 0;
          double2 *x = nullptr, *y = nullptr;
          auto load = [](const double2* s) { return SM ? *s : __ldcg(s); };
          auto store = [](double2* s, double2 v) {
            if (SM) *s = v;
            else __stcg(s, v);
          };
          const int r0 = gw * 32 + lane, step = wpp * 32;
          if (wid < JW) {
            pair_of(p, &li, &lj);
            const int gi = gcol(li), gj = gcol(lj);
            x = SM ? s_col + (size_t)li * ld : A + (size_t)max(gi, 0) * Ma;
            y = SM ? s_col + (size_t)lj * ld : A + (size_t)max(gj, 0) * Ma;
            if (gi >= 0 && gj >= 0) {
              double gr = 0, gim = 0;
              for (int r = r0; r < Ma; r += step) {
                const double2 u = load(x + r), v = load(y + r);
                gr = fma(u.x, v.x, fma(u.y, v.y, gr));
                gim = fma(u.x, v.y, fma(-u.y, v.x, gim));
              }
              const int E = pair_exponent(S.nrm[li], S.nrm[lj], S.q[li], S.q[lj]) + ex;
              __syncwarp();
              const long long sr_ = lane_sum(to_fixed(gr, E)), si_ = lane_sum(to_fixed(gim, E));
              if (lane < 2) S.part[wid][lane] = __longlong_as_double(lane == 0 ? sr_ : si_);
            }
            slot_sync(grp);
          } else {
            // lanes 2 k + comp take column warp k's partial sum; the lanes of a pair compute the same
            const int pp = min(lane >> (1 + lw), b - 1);
            int i, j;
            pair_of(pp, &i, &j);
            const bool first = ((lane >> 1) & (wpp - 1)) == 0 && lane < 2 * JW;
            const bool lead = first && (lane & 1) == 0, lead_odd = first && (lane & 1) != 0;
            const double al = S.nrm[i], be = S.nrm[j], qx = S.q[i], qy = S.q[j];
            const double h = be - al, qq = qx * qy;
            const int pe = pair_exponent(al, be, qx, qy);
            int ea, eb, eh;
            const float am = significand(al, &ea), bm = significand(be, &eb), hm = significand(h, &eh);
            // rotate unless |gamma| <= tol sqrt(alpha beta), or a column is at the noise floor (compared as
            // integers; a NaN fails below)
            bool go = gcol(i) >= 0 && gcol(j) >= 0 &&
                      min(__double_as_longlong(al), __double_as_longlong(be)) > max(fl2, 0x0010000000000000ll - 1);
            if (lane == 0) S.renorm[sr & 1] = 0;
            // computed here, while the column warps form the inner products, not after the barrier
            asm volatile("" ::"d"(h), "d"(qq), "f"(am), "f"(bm), "f"(hm), "r"(ea + eb + et), "r"(eh), "r"(pe),
                         "r"((int)go));
            slot_sync(grp);
            long long vf = lane < 2 * JW ? __double_as_longlong(S.part[lane >> 1][lane & 1]) : 0ll;
            for (int o = 2; o < 2 * wpp; o <<= 1) vf += __shfl_xor_sync(0xffffffffu, vf, o);
            const double v = tcx::fixed_to_double(vf, pe, 57);
            const double other = __shfl_xor_sync(0xffffffffu, v, 1);
            const double gr = (lane & 1) ? other : v, gm = (lane & 1) ? v : other;
            const double g2 = qq * fma(gr, gr, gm * gm);             // |gamma|^2
            int eg;
            const float gs = significand(g2, &eg);
            const int dt = et + ea + eb - eg;
            go = go && eg > -1000 && eg < 1000 && ea < 1000 && eb < 1000 &&
                 (dt < -4 || (dt < 4 && gs > tm * am * bm * __int_as_float((127 + max(dt, -8)) << 23)));
            // rho = 2 sign(h) / (|h| + sqrt(h^2 + 4 |gamma|^2)), h = beta - alpha, on values scaled by 2^-E
            const int E = max(eh, (eg + 1) >> 1);
            const float hf = eh > -1023 ? scale_pow2(hm, eh - E) : 0.f, gf = scale_pow2(gs, eg - 2 * E);
            const float rf = __fdividef(2.0f, hf + sqrt_approx(fmaf(hf, hf, 4.0f * gf)));
            const int rb = __float_as_int(rf);
            const double rho = __hiloint2double(((rb >> 3) + ((1023 - 127 - E) << 20)) | (__double2hiint(h) & 0x80000000),
                                                rb << 29);
            // the even lanes form mu and then column i's norm and scale, the odd lanes nu and column j's
            const bool odd = lane & 1;
            const double own = odd ? qy : qx, f = rho * (odd ? qx : qy);
            if (lead || lead_odd) {
              if (go) {
                S.rot[pp][odd ? 2 : 0] = f * gr;
                S.rot[pp][odd ? 3 : 1] = f * gm;
              }
              if (lead) S.flag[pp] = go;
            }
            slot_sync(grp);
            // while the columns rotate: the squared norms after a rotation by any angle, unless they cancel below a
            // quarter (then recomputed from the columns), and the squared scales times cos^2
            int redo = 0;
            if ((lead || lead_odd) && go) {
              const double rg = rho * g2, t2 = rho * rg, a1 = 1.0 + t2;
              const double c2 = inverse(a1);
              const double mine = odd ? be : al, his = odd ? al : be;
              const double nrm = c2 * fma(t2, his, fma(odd ? 2.0 : -2.0, rg, mine));
              // a quarter: two less in the exponent field
              redo = __double2hiint(nrm) < __double2hiint(mine) - (2 << 20);
              const int at = odd ? j : i;
              S.nrm[at] = nrm;
              S.q[at] = own * c2;
              S.rotc[at] = 1;
              if (lead) atomicAdd(&S.cnt, 1);
            }
            redo |= __shfl_xor_sync(0xffffffffu, redo, 1);
            if (first && redo) S.renorm[sr & 1] = 1;
            if (lead) S.redo[pp] = redo;
          }
          if (wid < JW) slot_sync(grp);
          if (wid < JW && S.flag[p]) {
            const double mr = S.rot[p][0], mi = S.rot[p][1], nr = S.rot[p][2], ni = S.rot[p][3];
            // x <- x - conj(mu) y, y <- y + nu x
            auto rotate = [&](double2* u, double2* v, int r) {
              const double2 a = load(u + r), c = load(v + r);
              double2 na, nc;
              na.x = fma(-mr, c.x, fma(-mi, c.y, a.x));
              na.y = fma(-mr, c.y, fma(mi, c.x, a.y));
              nc.x = fma(nr, a.x, fma(-ni, a.y, c.x));
              nc.y = fma(nr, a.y, fma(ni, a.x, c.y));
              store(u + r, na);
              store(v + r, nc);
            };
            if (SM) {
              for (int r = r0; r < ld; r += step) rotate(x, y, r);
            } else {
              for (int r = r0; r < Ma; r += step) rotate(x, y, r);
              for (int r = r0; r < Vr; r += step)
                rotate(V + (size_t)gcol(li) * Na, V + (size_t)gcol(lj) * Na, r);
            }
          }
          slot_sync(grp);
          if (S.renorm[sr & 1]) {
            // uniform in the CTA: pairs whose closed-form norms cancel get them from their columns
            if (wid < JW && S.redo[p]) {
              double na = 0, nb2 = 0;
              for (int r = r0; r < Ma; r += step) {
                const double2 u = load(x + r), v = load(y + r);
                na = fma(u.x, u.x, fma(u.y, u.y, na));
                nb2 = fma(v.x, v.x, fma(v.y, v.y, nb2));
              }
              const double s = wsum2(na, nb2, lane);
              if ((lane & 15) == 0) S.part[wid][lane >> 4] = s;
            }
            slot_sync(grp);
            if (wid < JW && S.redo[p] && gw == 0 && lane == 0) {
              double sa = 0, sb = 0;
              for (int k = 0; k < wpp; ++k) {
                sa += S.part[p * wpp + k][0];
                sb += S.part[p * wpp + k][1];
              }
              S.nrm[li] = sa * unit * S.q[li];
              S.nrm[lj] = sb * unit * S.q[lj];
            }
            slot_sync(grp);
          }
        }
        // changed columns, norms and scales back; a small scale is multiplied into its column
        for (int c = c0; c < 2 * b && wid < JW; c += JW) {
          const int g = gcol(c);
          if (g < 0 || !S.rotc[c]) continue;
          const bool fold = __double2hiint(S.q[c]) < MIN_SCALE_HI;
          double2* a = A + (size_t)g * Ma;
          double2* v = V + (size_t)g * Na - Ma;
          const double2* from = s_col + (size_t)c * ld;
          if (SM && !fold) {
#pragma unroll 4
            for (int r = rc0; r < ld; r += 32 * wpc) __stcg((r < Ma ? a : v) + r, from[r]);
          } else if (fold) {
            const double f = sqrt(S.q[c]);
            for (int r = rc0; r < ld; r += 32 * wpc) {
              double2* dst = (r < Ma ? a : v) + r;
              double2 val = SM ? from[r] : __ldcg(dst);
              val.x *= f;
              val.y *= f;
              __stcg(dst, val);
            }
          }
        }
        if (tid < 2 * b && gcol(tid) >= 0 && (round == 0 || S.rotc[tid])) {
          const int g = gcol(tid);
          __stcg(aux + g, S.nrm[tid]);
          __stcg(sig + g, __double2hiint(S.q[tid]) < MIN_SCALE_HI ? 1.0 : S.q[tid]);
        }
        slot_sync(grp);
        if (tid == 0) {
          if (S.cnt) atomicAdd(work[w].info + 4 + par, S.cnt);
          __threadfence();                 // the slot's columns, norms and scales (thread 0 has them through the barrier)
          if (bi < nb) store_relaxed(ver + bi, need + 1);
          if (bj < nb) store_relaxed(ver + bj, need + 1);
        }
      }
    }
    if (!barrier()) return;                // every rotation of the sweep has been counted
    // sweep done: retire converged items (every CTA reads the same counters)
    for (int w = ctid; w < n_work; w += CT)
      if (s_act[w] && *(volatile int*)(work[w].info + 4 + par) == 0) {
        s_act[w] = 0;
        if (blockIdx.x == 0) work[w].info[3] = sweep + 1;
      }
    __syncthreads();
    set_rounds();
    ++sweep;
    if (!barrier()) return;
  }
  if (s_rounds > 0 && blockIdx.x == 0 && ctid == 0) {
    atomicOr(status, ST_SVD_NOCONV);
    for (int w = 0; w < n_work; ++w)
      if (s_act[w]) work[w].info[3] = -sweep;
  }
  // singular values: column norms times the scales; normalised columns (left vectors) and V with its scales
  {
    const int gwarp = cwid * G + blockIdx.x, ngwarp = G * CW;
    int base = 0;
    for (int w = 0; w < n_work; ++w) {
      const BondWork& W = work[w];
      const int Ma = s_Ma[w], Na = s_Na[w];
      for (int c = gwarp - base; c < Na; c += ngwarp) {
        if (c < 0) continue;
        double2* a = mat_of(W, on_b) + (size_t)c * Ma;
        const double q = __ldcg(W.sig + c), d = q == 1.0 ? 1.0 : sqrt(q);
        double s2 = 0;
        for (int r = lane; r < Ma; r += 32) {
          const double2 x = __ldcg(a + r);
          s2 = fma(x.x, x.x, fma(x.y, x.y, s2));
        }
        const double nrm = sqrt(wsum(s2)), sg = nrm * d;
        __syncwarp();
        if (lane == 0) __stcg(W.sig + c, sg);
        if (nrm > 0.0) {
          const double inv = 1.0 / nrm;
          for (int r = lane; r < Ma; r += 32) {
            double2 x = __ldcg(a + r);
            x.x *= inv;
            x.y *= inv;
            __stcg(a + r, x);
          }
        }
        if (with_v && d != 1.0) {
          double2* v = W.V + (size_t)c * Na;
          for (int r = lane; r < Na; r += 32) {
            double2 x = __ldcg(v + r);
            x.x *= d;
            x.y *= d;
            __stcg(v + r, x);
          }
        }
        if (lane == 0 && !(sg == sg)) {
          atomicOr(status, ST_NAN);
          atomicOr(W.info + 6, FAULT_SIGMA_NAN);
        }
      }
      base = (base + Na) % ngwarp;
    }
  }
  // on_b: the columns of D beyond the QR's rank have singular value 0
  const int gt = blockIdx.x * CT + ctid, ngt = G * CT;
  auto full = [&](int w) { return on_b == 1 ? s_Ma[w] : s_Na[w]; };
  if (on_b == 1)
    for (int w = 0; w < n_work; ++w)
      for (int c = s_Na[w] + gt; c < full(w); c += ngt) __stcg(work[w].sig + c, 0.0);
  if (!barrier()) return;
  for (int w = 0; w < n_work; ++w) {
    const int Na = full(w);
    const double* sig = work[w].sig;
    for (int c = gt; c < Na; c += ngt) {
      // order by the values' bits (sign and magnitude are those of a non-negative number); a NaN ranks below
      // every number so the ranks stay a permutation (perm indexes columns downstream)
      auto key = [&](int k) {
        const long long v = __double_as_longlong(__ldcg(sig + k));
        return (v & 0x7fffffffffffffffll) > 0x7ff0000000000000ll ? -1ll : v;
      };
      const long long sc = key(c);
      int rk = 0;
      for (int k = 0; k < Na; ++k) {
        const long long sk = key(k);
        rk += (sk > sc) || (sk == sc && k < c);
      }
      work[w].perm[rk] = c;
    }
  }
}

namespace {
// dynamic shared memory of a launch over n_work items with columns of at most `rows` rows (V included), and the
// task slots it holds (two if each has room for b = 2); the header alone: the columns stay in L2
int jacobi_smem(int n_work, int rows, int* n_grp) {
  constexpr long long MAX = 220 * 1024;          // 227 KB per SM less the static arrays
  const int hdr = header_bytes(n_work);
  const long long col = 16LL * rows;
  *n_grp = JG;
  if (hdr + JG * 4 * col <= MAX) return (int)std::min(MAX, hdr + JG * 2 * JB * col);
  *n_grp = 1;
  if (hdr + 2 * col <= MAX) return (int)std::min(MAX, hdr + 2 * JB * col);
  *n_grp = JG;
  return hdr;
}
}  // namespace

int jacobi_grid_blocks() {
  int dev = 0, sms = 0, a = 0, b = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaFuncSetAttribute(k_jacobi_grid<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
  cudaFuncSetAttribute(k_jacobi_grid<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, header_bytes(MAX_ITEMS));
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_jacobi_grid<true>, CT, 220 * 1024);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_jacobi_grid<false>, CT, 32 * 1024);
  cudaGetLastError();
  return a >= 1 && b >= 1 ? sms : 0;
}

cudaError_t launch_jacobi_grid(const BondWork* work, int n_work, int blocks, int rows_cap, int max_sweeps, unsigned* sync3,
                        int* status, cudaStream_t st, int on_b, int with_v, double tol_scale, double floor2,
                        long long wait_cycles) {
  // the barrier's arrival counter and the abort flag start at zero for every launch
  cudaMemsetAsync(sync3, 0, 3 * sizeof(unsigned), st);
  GridSync gs{sync3, (int*)(sync3 + 2), wait_cycles > 0 ? wait_cycles : GRID_WAIT_LIMIT_CYCLES};
  int n_grp = 1;
  const int hdr = jacobi_smem(n_work, 1 << 20, &n_grp), smem = jacobi_smem(n_work, rows_cap, &n_grp);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks, 1, 1);
  cfg.blockDim = dim3(CT, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, smem > hdr ? k_jacobi_grid<true> : k_jacobi_grid<false>, work, n_work, max_sweeps, gs,
                     status, on_b, with_v, tol_scale, floor2, n_grp, smem);
}

// Whole GPU against one cluster per matrix: two 256 x 256 matrices 113 ms in two 16-CTA clusters (32 of 152 SMs),
// see the head of this file; the cluster kernel takes what one launch of this one does not, and what is left of a device
// that cannot hold all of its CTAs at once (a context with fewer SMs than the device says).
void launch_svd_jacobi(const BondWork* items, int batch, int Ma, int Na, int max_sweeps, int* status, unsigned* sync3,
                       cudaStream_t st, const JacobiTune& tune) {
  const int blocks = batch <= MAX_ITEMS ? jacobi_grid_blocks() : 0;
  if (blocks > 0) {
    const bool clean = cudaPeekAtLastError() == cudaSuccess;
    const cudaError_t e = launch_jacobi_grid(items, batch, tune.ctas > 0 ? tune.ctas : blocks, Ma + Na, max_sweeps, sync3,
                                             status, st, /*on_b=*/0, /*with_v=*/1, 0.0, JACOBI_FLOOR2, tune.wait_cycles);
    if (e != cudaErrorCooperativeLaunchTooLarge || !clean) return;
    cudaGetLastError();                    // this launch's, refused before anything ran
  }
  const int cl = jacobi_cluster_size(std::max(1, std::min(16, (Na / 2 + 7) / 8)));
  launch_jacobi_cluster(items, batch, cl, max_sweeps, status, st);
}

}  // namespace ptk
