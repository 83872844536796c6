// Building blocks of the digit-product kernels (zgemm_digits.cu, qr_tensor.cu): mbarriers with
// bounded waits, bulk copies, tcgen05 kind::f16 on K-major tiles without swizzle, the split of an
// FP64 number into seven signed base-256 digits and the reassembly of the level sums.
#pragma once
#include "fp64_util.cuh"
#include "tdmrg_internal.cuh"

namespace tdmrg {
namespace dig {

constexpr int ND = 7;                         // digits of an operand
constexpr int NL = 8;                         // levels i + j of digit pairs kept
constexpr int E_NONFINITE = 1 << 20;          // scale of a row that holds an Inf or a NaN
constexpr long long WAIT_CYCLES = 4000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait (about 2 s); gives up at once when another role of the CTA has
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* fail,
                                          int* status, int code) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try(bar, parity)) {
    if (*fail) return false;
    if (clock64() - t0 > WAIT_CYCLES) {
      *fail = 1;
      atomicExch(status, code);
      return false;
    }
  }
  return true;
}
// 16-byte aligned copy into shared memory, counted on `bar`
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// K-major operand without swizzle: 8-row x 16-byte core matrices, `lbo` bytes between the two of
// a 16-deep k step, `sbo` bytes between row groups
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo = 128) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}
// D f32, A and B fp16, both K-major, M = 128
__host__ __device__ constexpr uint32_t idesc(int negA, int n) {
  return (1u << 4) | ((uint32_t)negA << 13) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t id,
                                        uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}
// Groups of levels: group g holds the levels lo(g) .. lo(g + 1) - 1 (PACK: four bits each).  The
// order of tcgen05.mma instructions into TMEM columns they share is defined only where accumulator
// and shape are the same, so every instruction of a group writes all of its columns: digit i of A
// meets the digits lo(g) - i .. lo(g + 1) - 1 - i of B, and those outside 0 .. ND - 1 are blocks of
// zeros in shared memory, LEAD of them before each run of ND digits (the one behind a run is the
// next run's first).  Fewer, wider groups need fewer instructions (each reads the 4 KB of A again)
// and a longer lead.
template <int N, unsigned PACK>
struct Groups {
  static constexpr int n = N;
  __host__ __device__ static constexpr int lo(int g) { return (int)(PACK >> (4 * g)) & 15; }
  __host__ __device__ static constexpr int lead() {
    int l = 1;
    for (int g = 0; g < N; ++g) {
      const int i = lo(g + 1) - 1 < ND - 1 ? lo(g + 1) - 1 : ND - 1;     // the last digit of A
      if (i - lo(g) > l) l = i - lo(g);
    }
    return l;
  }
};
// One 16-deep k step: d (re levels; im levels `im` columns further) += A B, QT columns per level.
// A: digit 0 of re at `a` (im `apart`, the next digit `adig` bytes further).  B: digit 0 of re at
// `b`, its runs of ND digits `pitch` bytes apart: re k half 0, re k half 1, im, im.
// conj: conj(A) B (re = ArBr + AiBi, im = ArBi - AiBr).  first: the levels start from zero.
template <class G, int QT>
__device__ __forceinline__ void mma_levels(uint32_t d, uint32_t im, uint32_t a, uint32_t lbo,
                                           uint32_t sbo, uint32_t apart, uint32_t adig, uint32_t b,
                                           uint32_t pitch, bool first, bool conj) {
#pragma unroll
  for (int i = 0; i < ND; ++i) {
    const uint64_t ar = sdesc(a + i * adig, lbo, sbo), ai = sdesc(a + apart + i * adig, lbo, sbo);
    const uint32_t acc = (!first || i > 0) ? 1u : 0u;
#pragma unroll
    for (int g = 0; g < G::n; ++g) {
      if (i >= G::lo(g + 1)) continue;
      const int n = QT * (G::lo(g + 1) - G::lo(g));
      const uint32_t w = b + (G::lo(g) - i) * (QT * 16), dr = d + G::lo(g) * QT, di = dr + im;
      const uint64_t br = sdesc(w, pitch), bi = sdesc(w + 2 * pitch, pitch);
      mma_f16(dr, ar, br, idesc(0, n), acc);
      mma_f16(di, ar, bi, idesc(0, n), acc);
      mma_f16(dr, ai, bi, idesc(conj ? 0 : 1, n), 1u);
      mma_f16(di, ai, br, idesc(conj ? 1 : 0, n), 1u);
    }
  }
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// x (negated if neg) in units of 2^(E - 55), E = emax - 1022 and |x| < 2^E, rounded, plus 128 in
// each of its seven base-256 digits: digit l (l = 0 the highest) is bits 48 - 8 l .. of it, less
// 128.  emax >= 1.
__device__ __forceinline__ unsigned long long digits_of(double x, int emax, bool neg, bool bad) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(bits >> 52) & 0x7ff;
  unsigned long long mant = bits & 0xfffffffffffffULL;
  if (ex) mant |= 1ULL << 52;
  const int sh = max(ex, 1) - emax + 2;
  unsigned long long v;
  if (sh >= 0) v = mant << sh;
  else if (sh >= -54) v = (mant + (1ULL << (-sh - 1))) >> (-sh);
  else v = 0;
  if (bad) v = 0;
  neg = neg != ((bits >> 63) != 0);
  return (neg ? 0ULL - v : v) + 0x0080808080808080ULL;
}
// digit l of two numbers as packed fp16: 0x6400 + u is the fp16 number 1024 + u, less 1152
__device__ __forceinline__ uint32_t digit_pair(unsigned long long a, unsigned long long b, int l) {
  const uint32_t mask = l == 0 ? 0xffffu : 0xffu;
  const uint32_t pk = (0x64006400u + ((uint32_t)(a >> (48 - 8 * l)) & mask)) +
                      (((uint32_t)(b >> (48 - 8 * l)) & mask) << 16);
  uint32_t d;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(d) : "r"(pk), "r"(0x64806480u));
  return d;
}

// One accumulated product sum from its eight level sums (FP32 bits holding integers below 2^25, even
// above 2^24; level l counts units of 2^(E_A + E_B - 14 - 8 l)), rounded to nearest.  General form, with the
// library's scaling where the result leaves the normal range.
static __device__ __noinline__ double from_levels_any(const uint32_t* v, int eA, int eB) {
  if (eA == E_NONFINITE || eB == E_NONFINITE) return __longlong_as_double(0x7ff8000000000000LL);
  long long S[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) S[l] = __float2int_rn(__uint_as_float(v[l]));
  const long long hi = S[0] * 16777216LL + S[1] * 65536LL + S[2] * 256LL + S[3];
  const long long lo = S[4] * 16777216LL + S[5] * 65536LL + S[6] * 256LL + S[7];
  const int sh = min(32, __clzll(hi < 0 ? -hi : hi) - 2);
  const long long T = (long long)((unsigned long long)hi << sh) + (lo >> (32 - sh));
  return scalbn((double)T, eA + eB - 38 - sh);
}

// The same for levels of at most 2^22 and a result in the normal range, in integer arithmetic
// without branches (FP64 conversions run at the FP64 rate, and the float-to-integer conversion at
// a quarter of the rate of the additions used here); sets `rare` where it does not apply.
__device__ __forceinline__ double from_levels(const uint32_t (&v)[NL], int eA, int eB, bool& rare) {
  int S[NL];
  float big = 0.f;
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    const float f = __uint_as_float(v[l]);
    big = fmaxf(big, fabsf(f));
    S[l] = __float_as_int(f + 12582912.f) - 0x4B400000;      // 1.5 * 2^23: integers up to 2^22
  }
  // the sum is hi 2^32 + lo in units of level 7 (|hi| < 2^47, |lo| < 2^48): 62 bits of it, from
  // the top of hi down
  const long long hi = (long long)(S[0] * 256 + S[1]) * 65536 + (S[2] * 256 + S[3]);
  const long long lo = (long long)(S[4] * 256 + S[5]) * 65536 + (S[6] * 256 + S[7]);
  const int sh = min(32, __clzll(hi < 0 ? -hi : hi) - 2);
  const long long T = (long long)((unsigned long long)hi << sh) + (lo >> (32 - sh));
  const unsigned long long u = T < 0 ? 0ULL - (unsigned long long)T : (unsigned long long)T;
  const int lz = __clzll((long long)u) & 63;
  const int be = eA + eB - 38 - sh + 63 - lz + 1023;         // biased exponent
  const unsigned long long m = u << lz;
  const unsigned long long up = (m >> 10) & ((m & 0xbff) != 0 ? 1ULL : 0ULL);
  unsigned long long bits = ((unsigned long long)(be - 1) << 52) + (m >> 11) + up;
  bits |= (unsigned long long)T & (1ULL << 63);
  rare = rare || big > 4194304.f || (u != 0 && (unsigned)(be - 1) > 2044u) ||
         (eA == E_NONFINITE) || (eB == E_NONFINITE);
  return u == 0 ? 0.0 : __longlong_as_double((long long)bits);
}

// Four accumulated sums of one row, and with P = 2 their imaginary parts im columns further: the
// levels of columns c .. c + 3 at taddr + l * ldl.  All 32 lanes call it (lane = TMEM row); eB[c]
// is the scale of column c.
template <int P>
__device__ __forceinline__ void read_levels4(uint32_t taddr, uint32_t ldl, uint32_t im, int eA,
                                             const int (&eB)[4], double (&x)[P][4]) {
  uint32_t v[P][NL][4];
#pragma unroll
  for (int p = 0; p < P; ++p)
#pragma unroll
    for (int l = 0; l < NL; ++l) tmem_ld4(taddr + p * im + l * ldl, v[p][l]);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  bool rare = false;
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int p = 0; p < P; ++p) {
      uint32_t u[NL];
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        asm volatile("" : "+r"(v[p][l][c]));   // the loads are complete: tie the values to the wait
        u[l] = v[p][l][c];
      }
      x[p][c] = from_levels(u, eA, eB[c], rare);
    }
  if (rare) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int p = 0; p < P; ++p) {
        uint32_t u[NL];
#pragma unroll
        for (int l = 0; l < NL; ++l) u[l] = v[p][l][c];
        x[p][c] = from_levels_any(u, eA, eB[c]);
      }
  }
}

}  // namespace dig
}  // namespace tdmrg
