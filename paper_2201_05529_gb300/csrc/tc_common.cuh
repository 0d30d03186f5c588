// tcgen05 building blocks shared by the tensor-core GEMMs of the fast path (tc_theta.cu, tc_zgemm.cu):
// mbarrier waits with an iteration limit, bulk global -> shared copies, shared-memory and instruction
// descriptors, the MMA and the TMEM load, the packed-operand geometry, and the splitting of an FP64
// value into TF32/BF16 pieces (natural split) or fixed-point BF16 slices (Ozaki, Ogita, Oishi and
// Rump's error-free splitting of matrix products).
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"

namespace ptk {
namespace tcx {

constexpr int TMA = 128;            // A tile rows
constexpr int TNB = 64;             // B tile rows (columns of the product) = output tile columns
constexpr int TC_THREADS = 128;
constexpr int MAX_STAGES = 3;     // shared-memory stages of the K pipeline (2 for six slices: 227 KB)
template <int NS> struct Stages { static constexpr int value = NS >= 6 ? 2 : MAX_STAGES; };
constexpr int MAX_ITEMS = 1024;
constexpr uint32_t ROW_BYTES = 32;  // one K step of one row: 8 tf32 or 16 bf16 (two 16-byte K groups)
constexpr long long SPIN_LIMIT = 20000000;  // mbarrier polls before giving up
constexpr uint32_t NEG_A = 1u << 13;        // instruction descriptor: negate matrix A

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// true when the phase with the given parity has completed; false after SPIN_LIMIT polls
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (long long it = 0; it < SPIN_LIMIT; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// shared memory matrix descriptor: K-major, no swizzle, LBO = K-group stride, SBO = 8-row stride
__device__ __forceinline__ uint64_t smem_desc(const void* p, uint32_t lbo, uint32_t sbo) {
  const uint64_t a = smem_u32(p);
  uint64_t d = 0;
  d |= (a >> 4) & 0x3FFFull;
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;          // descriptor version for sm_100-class tcgen05
  return d;                        // base offset 0, layout type 0 = SWIZZLE_NONE
}

// the same for rows of 32 bytes (one K step) in the 32-byte swizzle: eight rows of 32 bytes per 256-byte atom
// (SBO), the two 16-byte halves of rows 4 .. 7 exchanged
__device__ __forceinline__ uint64_t smem_desc_sw32(const void* p) {
  return smem_desc(p, 16, 256) | (uint64_t)6 << 61;
}
// byte offset of half h (16 bytes) of row m in that layout
__device__ __forceinline__ uint32_t sw32_offset(int m, int h) {
  return (uint32_t)(m * 32 + ((h ^ (m >> 2 & 1)) * 16));
}

// instruction descriptor for kind::tf32 (ab_fmt = 2) or kind::f16 with bf16 inputs (ab_fmt = 1):
// FP32 accumulator, K-major A and B, N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ uint32_t instr_desc(uint32_t ab_fmt, int M, int N) {
  uint32_t d = 0;
  d |= 1u << 4;                    // D format F32
  d |= ab_fmt << 7;                // A format
  d |= ab_fmt << 10;               // B format
  d |= (uint32_t)(N >> 3) << 17;
  d |= (uint32_t)(M >> 4) << 24;
  return d;
}

// slice pairs (s, u), s + u < NS, by accumulator level L = min(s + u, NLEV - 1): pair i of level L
__host__ __device__ constexpr int pair_count(int L, int NS, int NLEV) {
  int n = 0;
  for (int t = L; t < (L == NLEV - 1 ? NS : L + 1); ++t) n += t + 1;
  return n;
}
__host__ __device__ constexpr int pair_s(int L, int i) {
  while (i > L) i -= ++L;          // the deeper levels that share the last accumulator
  return i;
}
__host__ __device__ constexpr int pair_u(int L, int i) {
  while (i > L) i -= ++L;
  return L - i;
}

template <bool BF16>
__device__ __forceinline__ void mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, bool acc) {
  const uint32_t en = acc ? 1u : 0u;
  if (BF16) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(en)
        : "memory");
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(en)
        : "memory");
  }
}

// The MMAs of one K step of a complex product of NS x NS slices (Re += Ar Br - Ai Bi, Im += Ar Bi + Ai Br) into the
// accumulators dre = tmem + 2 L TN, dim = dre + TN of the levels.
template <bool BF16, int NS, int NLEV, int TN, uint32_t A_PLANE, uint32_t B_PLANE>
__device__ __forceinline__ void mma_slices(uint32_t tmem, uint64_t a0, uint64_t b0, uint32_t idesc, bool acc) {
  constexpr int MOST = pair_count(NLEV - 1, NS, NLEV);
  auto a = [&](int plane) { return a0 + (uint64_t)(plane * (A_PLANE >> 4)); };
  auto b = [&](int plane) { return b0 + (uint64_t)(plane * (B_PLANE >> 4)); };
#pragma unroll
  for (int i = 0; i < MOST; ++i)
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int L = NLEV - 1; L >= 0; --L) {
        if (i >= pair_count(L, NS, NLEV)) continue;
        const int s = pair_s(L, i), u = pair_u(L, i);
        const uint32_t dre = tmem + (2 * L) * TN, dim = dre + TN;
        const bool en = acc || i > 0 || r > 0;
        if (r == 0) {
          mma<BF16>(dre, a(s), b(u), idesc, en);
          mma<BF16>(dim, a(s), b(NS + u), idesc, en);
        } else {
          mma<BF16>(dre, a(NS + s), b(NS + u), idesc | NEG_A, en);
          mma<BF16>(dim, a(NS + s), b(u), idesc, en);
        }
      }
}

// The same with B's planes as (-Bi, Br, Bi) per slice, adjacent: one MMA of 2 TN columns forms Ar Br and Ar Bi, another
// -Ai Bi and Ai Br, so half as many MMAs. An MMA of 128 rows costs 53 cycles at up to 64 columns, whatever the
// accumulators of its neighbours, and 66 at 128 (measured; the operands' layout does not matter).
// The whole warp runs it and `one` lane issues: the descriptors then stay in uniform registers (issued by a branch
// of one lane, every operand is moved there first and an MMA takes ~110 cycles).
__device__ __forceinline__ void mma_bf16_one(bool one, uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %4, 0;\n setp.ne.u32 q, %5, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc ? 1u : 0u), "r"(one ? 1u : 0u)
      : "memory");
}

template <int NS, int NLEV, int TN, uint32_t A_PLANE, uint32_t B_PLANE>
__device__ __forceinline__ void mma_slices_stacked(bool one, uint32_t tmem, uint64_t a0, uint64_t b0, uint32_t idesc,
                                                   bool acc) {
  constexpr int MOST = pair_count(NLEV - 1, NS, NLEV);
  auto a = [&](int plane) { return a0 + (uint64_t)(plane * (A_PLANE >> 4)); };
  auto b = [&](int plane) { return b0 + (uint64_t)(plane * (B_PLANE >> 4)); };
#pragma unroll
  for (int i = 0; i < MOST; ++i)
#pragma unroll
    for (int L = NLEV - 1; L >= 0; --L) {
      if (i >= pair_count(L, NS, NLEV)) continue;
      const int s = pair_s(L, i), u = pair_u(L, i);
      const uint32_t d = tmem + 2 * L * TN;
      mma_bf16_one(one, d, a(s), b(3 * u + 1), idesc, acc || i > 0);
      mma_bf16_one(one, d, a(NS + s), b(3 * u), idesc, true);
    }
}

// one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  uint32_t one;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(one));
  return one != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// the same load without its wait, and the wait for every load before it
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, float* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// packed operand geometry: one K step per chunk, 32 bytes of each row
template <bool BF16> struct Geo {
  static constexpr int EB = BF16 ? 2 : 4;       // element bytes
  static constexpr int KG = 16 / EB;            // elements per 16-byte K group
  static constexpr int KSTEP = 2 * KG;          // K per MMA instruction (8 tf32, 16 bf16)
};

__host__ __device__ __forceinline__ int cdiv(int a, int b) { return (a + b - 1) / b; }

// capacity layout of one packed operand: [row tile][K step][plane][K group][rows][16 B],
// then one int exponent per (padded) row
struct PackCap {
  int tiles, ksteps;
  size_t plane_bytes, exp_off, total;
};

// planes: per K step and row tile, 2 ns unless given
__host__ __device__ __forceinline__ PackCap pack_cap(int rows_cap, int k_cap, int tile_rows, int kstep, int ns,
                                                     int planes = 0) {
  if (planes == 0) planes = 2 * ns;
  PackCap c;
  c.tiles = cdiv(rows_cap, tile_rows);
  c.ksteps = cdiv(k_cap, kstep);
  c.plane_bytes = (size_t)tile_rows * ROW_BYTES;
  c.exp_off = (size_t)c.tiles * c.ksteps * planes * c.plane_bytes;
  c.total = c.exp_off + sizeof(int) * (size_t)c.tiles * tile_rows;
  return c;
}

// the NS pieces of x (already scaled by 2^-e for slices) as TF32 or BF16 bit patterns
template <bool BF16, int NS, bool SLICE>
__device__ __forceinline__ void pieces(double x, int b, uint32_t* out) {
  if (SLICE) {
    // fixed-point slices: a_i = rint(r 2^b), r <- r 2^b - a_i; slice value a_i 2^(-b(i+1))
    double r = x;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const double t = ldexp(r, b);
      const double a = rint(t);
      r = t - a;
      const float s = (float)ldexp(a, -b * (i + 1));      // exact: |a| <= 2^b <= 2^8
      out[i] = BF16 ? (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(s)) : __float_as_uint(s);
    }
  } else {
    double r = x;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const float f = (float)r;
      if (BF16) {
        const __nv_bfloat16 h = __float2bfloat16_rn(f);
        out[i] = (uint32_t)__bfloat16_as_ushort(h);
        r -= (double)__bfloat162float(h);
      } else {
        uint32_t hb;
        asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hb) : "f"(f));
        out[i] = hb;
        r -= (double)__uint_as_float(hb);
      }
    }
  }
}

// ---- the slices and their sums in integer arithmetic. GB300 issues an FP64 instruction per warp every 64
// cycles and sub-partition (measured; 19 per SM) against one integer or FP32 instruction per cycle, so
// neither the cut into slices nor the addition of the level sums runs on the FP64 pipe.

// BF16 bit patterns (in the upper half of each word) of the NS fixed-point slices of x 2^-e, |x| < 2^e: x is
// rounded to NS * b fractional bits and cut into signed digits |a_i| <= 2^b, slice value a_i 2^(-b(i+1)) (NS a multiple
// of three, NS b <= 63). A NaN or an infinity becomes a NaN in slice 0 (every sum it enters comes out NaN).
template <int NS>
__device__ __forceinline__ void int_slices(double x, int e, int b, uint32_t* out) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int ex = (int)((hi >> 20) & 0x7ff);
  const uint64_t mant = ((uint64_t)((hi & 0xfffffu) | (ex ? 0x100000u : 0u)) << 32) | lo;
  // |x| = mant 2^(max(ex, 1) - 1075); F = round(|x| 2^(NS b - e)) < 2^(NS b): a shift to the right by 53 - NS b or more,
  // except in a row of subnormals, whose e lies below the exponent of the smallest normal number
  const int sh = 1075 + e - NS * b - max(ex, 1);
  uint64_t F = 0;
  if (sh > 0 && sh < 64) F = (mant + (1ull << (sh - 1))) >> sh;
  else if (sh <= 0 && sh > -53) F = mant << -sh;
  // 32-bit parts of three digits, the last part first; the sign goes onto the digits
  constexpr int P = NS / 3;
  const int pb = 3 * b;
  const uint32_t sign = hi & 0x80000000u;
  const int rnd = 1 << (b - 1);
#pragma unroll
  for (int h = P - 1; h >= 0; --h) {
    int v;
    if (h > 0) {
      const uint64_t up = (F + (1ull << (pb - 1))) >> pb;
      v = (int)((long long)F - (long long)(up << pb));
      F = up;
    } else {
      v = (int)F;
    }
#pragma unroll
    for (int i = 2; i >= 0; --i) {
      const int next = i > 0 ? (v + rnd) >> b : 0;
      const int a = i > 0 ? v - (next << b) : v;
      v = next;
      // 1.5 2^(23 - b s) + a 2^(-b s): adding a to the last bits of the constant's pattern
      const int s = h * 3 + i + 1;
      const uint32_t magic = (uint32_t)(127 + 23 - b * s) << 23 | 0x400000u;
      out[h * 3 + i] = __float_as_uint(__uint_as_float(magic + (uint32_t)a) - __uint_as_float(magic)) ^ sign;
    }
  }
  if (ex == 0x7ff) out[0] = 0x7fc00000u;
}

// two slices' BF16 patterns in one word: first in the low half
__device__ __forceinline__ uint32_t pair_bf16(uint32_t first, uint32_t second) {
  return __byte_perm(first, second, 0x7632);
}

// |x| as an integer, 0 for a NaN or an infinity (integer order = order of the magnitudes)
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  const unsigned long long m = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
  return m < 0x7ff0000000000000ull ? m : 0ull;
}

// n 2^(e - lsb) as a double, n the 64-bit fixed-point sum of a product's levels
__device__ __forceinline__ double fixed_to_double(long long n, int e, int lsb) {
  if (n == 0) return 0.0;
  const unsigned long long a = n < 0 ? (unsigned long long)(-n) : (unsigned long long)n;
  const int lz = __clzll((long long)a);
  // the top 53 bits, rounded to nearest (ties away; a carry moves into the exponent)
  const unsigned long long m = ((a << lz) >> 10) + 1ull;      // 53 bits and the rounding bit
  const int bexp = 63 - lz - lsb + e + 1023;                  // biased exponent of the leading bit
  if (bexp > 1 && bexp < 2046) {
    const unsigned long long r = (m >> 1) + ((unsigned long long)(bexp - 1) << 52);   // the implicit bit adds one
    return __longlong_as_double((long long)(r | (n < 0 ? 0x8000000000000000ull : 0ull)));
  }
  return ldexp((double)n, e - lsb);
}

// the largest sum of a level's slice pairs over `terms` products, in units of 2^(-7 (L + 2)): |a_0| <= 2^7, |a_i| <= 2^6
__host__ __device__ constexpr long long level_max(int L, int NS, long long terms) {
  long long n = 0;
  for (int s = 0; s <= L; ++s)
    if (s < NS && L - s < NS) n += (s == 0 ? 128 : 64) * (s == L ? 128 : 64);
  return n * terms;
}
// the same of levels L .. NS - 1 together, in units of 2^-u
__host__ __device__ constexpr double levels_max(int L, int NS, long long terms, int u) {
  double n = 0;
  for (int t = L; t < NS; ++t) {
    double v = (double)level_max(t, NS, terms);
    for (int q = 7 * (t + 2); q < u; ++q) v *= 2;
    for (int q = u; q < 7 * (t + 2); ++q) v /= 2;
    n += v;
  }
  return n;
}

// the sum of levels FROM .. TO of an entry's accumulators (slice width 7) as an integer multiple of 2^-LSB: level L holds
// integer multiples of 2^(-7 (L + 2)), of TERMS products a pair. LAST > 0: the last level, shared by several, is rounded to
// multiples of 2^-LAST. A 32-bit conversion clamps, so it is taken only where the digits' largest sum fits (entries of
// coherent operands come near it; the 64-bit one costs 1 % of a 300 x 70 x 530 or 16384 x 64 x 64 product).
template <int FROM, int TO, int LSB, int LAST, int NS, int TERMS, int NLEV>
__device__ __forceinline__ long long level_sum(const float (&f)[NLEV][8], int j) {
  static_assert(levels_max(FROM, NS, TERMS, LSB) < 9e18, "the sum fits 63 bits");
  long long n = 0;
#pragma unroll
  for (int L = FROM; L <= TO; ++L) {
    const bool last = LAST > 0 && L == TO;
    const int u = last ? LAST : 7 * (L + 2);
    const float x = f[L][j] * __uint_as_float((uint32_t)(127 + u) << 23);
    const double most = last ? levels_max(L, NS, TERMS, u) : (double)level_max(L, NS, TERMS);
    // less 2^12 for what the accumulation's own rounding adds
    n += (most < 2147483648.0 - 4096.0 ? (long long)__float2int_rn(x) : __float2ll_rn(x)) * (1ll << (LSB - u));
  }
  return n;
}

// slice width: the level-0 sum over K of 2 products of |a| <= 2^b stays below 2^24
__device__ __forceinline__ int slice_bits(int K) { return K <= 512 ? 7 : (K <= 2048 ? 6 : 5); }

// exponent e with max |x| < 2^e (0 for an all-zero row)
__device__ __forceinline__ int row_exponent(double m) {
  if (!(m > 0.0)) return 0;
  int e;
  frexp(m, &e);          // m = f 2^e, f in [0.5, 1)
  return e;
}

}  // namespace tcx
}  // namespace ptk
