// Complex FP64 GEMM on the tensor cores: both operands are rounded to sums of 8-bit digits, whose
// products are summed in integers (the splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication", with a truncated product sum).
//
// Why: GB300 issues about 2 FP64 FMAs per clock per SM, so a 64 x 64 x 64 complex tile of
// zgemm_kernel holds an SM for ~0.27 ms; its tensor cores take 4096 fp16 multiply-adds per clock.
//
// Split (digit_split_kernel): a row of 128 consecutive k of an operand is scaled by the power of
// two 2^E above its largest component and rounded to a 56-bit integer in units of 2^(E-55), which
// is written as seven signed base-256 digits (-128..128), each an exact fp16.  All of it is integer
// arithmetic.  Re and im parts share E.  The digits are stored as the shared-memory image of the
// tile they will be staged in (8 x 16 byte core matrices), so a stage is one contiguous block.
//
// Product (digit_gemm_kernel): one CTA computes a 128 x 32 (or 128 x 16) tile of C.  Digit i of the
// 128-row operand times digit j of the 32-column operand goes to the accumulator of level i + j <= 7.
// Both the digits in shared memory and the levels in TMEM are contiguous, so one tcgen05.mma
// (kind::f16, FP32 accumulation) takes a digit i with several j at once: a group of levels per
// instruction (Groups in umma.cuh), 4 x 12 instructions per 16-deep k step with 32-column tiles,
// 4 x 7 with 16-column ones, zeros in the place of digits a group does not have.  A digit product is at
// most 2^14; over one chunk of 128 k a level of p pairs sums to an integer of at most p 2^22, exact
// in FP32 up to 2^24.  After each chunk eight warps read the levels back and combine them in
// 64-bit integers; the chunk's result is rounded once to FP64 and the chunks are added in FP64.
//
// Error of a component, per chunk with 2^EA and 2^EB the powers of two above the largest components
// of the row of A and the column of B (|a|_1 = |re| + |im|):
//   operands   sum_k 2^(EA-56) |b|_1 + 2^(EB-56) |a|_1    (entries above 1/8 of 2^E are exact)
//   pairs i + j > 7    2^-60 2^(EA+EB) per k
//   rounding   2^-53 of the chunk's sum, and of the partial sums over the chunks.
// Levels 4 to 7 (five to seven pairs) pass 2^24 only where nearly all digits are near 127 and the
// products of one sign; a chunk can then lose 2^-39 2^(EA+EB), which for such entries is 2^-45 of the
// sum of |a||b| (operands built for it: 2^-55, the rounding of the result).
// So the error is relative to the largest entries of a row and a column, that of FMAs to the sum of
// |a||b|.  The same or less where rows of A and columns of B are even or fall together along k, as in
// a sweep; where one rises as the other falls, by e^s in all, digits lose up to e^s: relative to the
// sum of |a||b|, K = 128, 2e-14 at e^9, 1e-10 at e^18, 2e-6 at e^28 against 2e-16 (falling together
// by e^28: 7e-17 against 1e-15).  Products whose operands are so by their nature, as R and its
// cotangent, take the FMA kernel (capi.cu, QR reverse passes).
//
// Bound: the tensor pipe in the main loop (48 instructions per k step of 128 x 32; narrow ones wait for
// the 4 KB of A that each reads), plus the integer epilogue, which cannot overlap it (eight re and im
// levels of 32 columns fill all 512 TMEM columns).  70 KB per stage from L2, three stages, one CTA per
// SM.  A small product is latency: a launch each for split, product and reduction, set up while the one
// before runs.
//
// Measured on GB300 against the FMA kernel, split and reduction included: 896 x 8192 x 128 0.290
// against 6.2 ms (26 TFLOP/s, tensor pipe 46 %); 8192 x 128 x 128 summed over seven channels 0.342
// against 7.3 ms; 128 x 128 x 8192, seven batches, 0.531 against 34 ms; 64 x 64 x 256, seven
// batches, 26 against 1049 us; 16 x 16 x 4 11 against 21 us.  With the digit pairs of all levels in
// instructions of different width on shared columns (28 a k step, an order that is not promised) the
// first three took 0.255, 0.310 and 0.486 ms.
#include "mix.cuh"
#include "umma.cuh"
#include "workspace.h"

#include <mutex>
#include <type_traits>

namespace tdmrg {

using namespace dig;

namespace {

constexpr int PT = 128;                       // tile rows (operand P)
// tile columns (operand Q): 32, or 16 where the tiles of 32 leave SMs idle
constexpr int KS = 16;                        // k per stage
constexpr int KC = 128;                       // k per chunk (one scale per row and chunk)
constexpr int STEPS = KC / KS;
constexpr int P_BLOCK = 2 * ND * PT * KS * 2; // 57344 bytes per stage
__host__ __device__ constexpr int q_block(int qt) { return 2 * ND * qt * KS * 2; }     // 14336, 7168
// level groups (lead 2 and 6): 16-column tiles have all levels in one, the wider ones as many as
// leave room for three stages
template <int QT>
using LevelsOf = std::conditional_t<QT == 16, Groups<1, 0x80>, Groups<3, 0x8410>>;
template <int QT>
__host__ __device__ constexpr int q_pitch() { return (LevelsOf<QT>::lead() + ND) * QT * 16; }    // between the runs of digits
template <int QT>
__host__ __device__ constexpr int q_stage() { return 4 * q_pitch<QT>() + QT * 16; }              // 18944, 13568
constexpr int NST = 3;
constexpr int GEMM_THREADS = 320;             // TMA warp, MMA warp, eight epilogue warps
constexpr size_t gemm_smem(int qt) {
  return (size_t)NST * (P_BLOCK + (qt == 16 ? q_stage<16>() : q_stage<32>())) + 256 + 128;
}
static_assert(gemm_smem(16) <= 227 * 1024 && gemm_smem(32) <= 227 * 1024, "shared memory");

struct Operand {
  const cplx* p;
  long long rs, ks, sb, sr;   // strides of row, k, batch, reduction term
  int conj;
  int rows, nb;               // rows; batches stored (1 when the batches share the operand)
  int tile;                   // PT, or the width of a Q tile
  int tiles;                  // row tiles
  unsigned char* dig;         // [nb][tiles][steps] blocks
  int* ex;                    // [nb][chunks][tiles * tile]
  // mixed on the fly (mix_start != NULL): p = X, the strides address Y
  const int* mix_start;
  const int2* mix_cu;
  const cplx* mix_val;
  long long xs;
  int dmb, d, b0;             // b0: first batch of a slab
  long long off0;             // offset of the first row of a slab
  int by_red;                 // the channel is the reduction term (else the batch)
};

struct SplitArgs {
  Operand o[2];
  int K, nred, ksteps, chunks;   // k steps and chunks of one reduction term
  int blocks0;                   // blocks of operand 0
  const int* skip;
};

constexpr int SR = 16;                        // rows of a split block
constexpr int S_LD = KC + 1;
constexpr int PER = 4;                        // entries a thread loads at a time
static_assert(SR * KC % (256 * PER) == 0, "split block");

// One block: 16 rows x one chunk of 128 k of one operand.
__global__ void __launch_bounds__(256) digit_split_kernel(SplitArgs A) {
  behind_next();
  behind_wait();
  if (A.skip && *A.skip) return;
  __shared__ cplx s_v[SR * S_LD];
  __shared__ int s_e[SR];
  const bool second = (int)blockIdx.x >= A.blocks0;
  const Operand& o = A.o[second ? 1 : 0];
  int id = blockIdx.x - (second ? A.blocks0 : 0);
  const int tc = A.nred * A.chunks;
  const int chunk = id % tc;
  id /= tc;
  const int groups = o.tiles * (o.tile / SR);
  const int r0 = (id % groups) * SR;
  const int b = id / groups;
  const int red = chunk / A.chunks, c = chunk % A.chunks;
  const int k0 = c * KC, kn = min(KC, A.K - k0);
  const int steps = (kn + KS - 1) / KS;
  const cplx* src = o.p + (long long)b * o.sb + (long long)red * o.sr;
  if (threadIdx.x < SR) s_e[threadIdx.x] = 0;
  // load in the order that is contiguous in memory, PER entries of a thread at a time: their loads
  // (and, mixed on the fly, the chains table row -> term -> X) are in flight together
  const bool kfast = o.ks == 1;
  const int* rows = o.mix_start ? o.mix_start + (o.by_red ? red : b + o.b0) * o.d : nullptr;
#pragma unroll 1
  for (int e0 = threadIdx.x; e0 < SR * KC; e0 += 256 * PER) {
    cplx v[PER];
    const cplx* x[PER];
    int at[PER], end[PER], dst[PER];
    bool more = false;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = e0 + i * 256;
      const int r = kfast ? e / KC : e % SR, k = kfast ? e % KC : e / SR;
      dst[i] = r * S_LD + k;
      v[i] = make_double2(0.0, 0.0);
      x[i] = o.p;
      at[i] = end[i] = 0;
      if (r0 + r < o.rows && k < kn) {
        const long long off = (long long)(r0 + r) * o.rs + (long long)(k0 + k) * o.ks;
        if (!rows) {
          v[i] = src[off];
        } else {
          const int idx = (int)(off + o.off0), sig = (idx / o.dmb) % o.d;
          x[i] = o.p + (idx - sig * o.dmb);
          at[i] = __ldg(rows + sig);
          end[i] = __ldg(rows + sig + 1);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) more = more || at[i] < end[i];
    for (bool first = true; more; first = false) {
      cplx f[PER], z[PER];
      int2 c[PER];
#pragma unroll
      for (int i = 0; i < PER; ++i) {          // (a term that is not wanted: term 0 and X[0])
        const int t = at[i] < end[i] ? at[i] : 0;
        c[i] = __ldg(o.mix_cu + t);
        f[i] = __ldg(o.mix_val + t);
      }
#pragma unroll
      for (int i = 0; i < PER; ++i)
        z[i] = at[i] < end[i] ? x[i][c[i].x * o.xs + (long long)c[i].y * o.dmb] : o.p[0];
      more = false;
#pragma unroll
      for (int i = 0; i < PER; ++i)
        if (at[i] < end[i]) {
          mix_add(v[i], f[i], z[i], first);
          ++at[i];
          more = more || at[i] < end[i];
        }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) s_v[dst[i]] = v[i];
  }
  __syncthreads();
  const int r = threadIdx.x & (SR - 1), g = threadIdx.x / SR;      // row, group of 8 k
  const cplx* mine = s_v + r * S_LD + g * 8;
  int e = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const cplx v = mine[i];
    e = max(e, max(bexp(v.x), bexp(v.y)));
  }
  atomicMax(&s_e[r], e);
  __syncthreads();
  const int em = s_e[r];
  if (g == 0)
    o.ex[((long long)b * tc + chunk) * ((long long)o.tiles * o.tile) + r0 + r] =
        em == 0x7ff ? E_NONFINITE : max(em, 1) - 1022;
  if (g >= 2 * steps) return;
  const int emax = max(em, 1);
  const bool bad = em == 0x7ff;
  const int row = r0 + r, tile = row / o.tile, rt = row % o.tile;
  const int ks = g >> 1, kh = g & 1;
  const long long step = (long long)red * A.ksteps + (long long)c * STEPS + ks;
  const int block = 2 * ND * o.tile * KS * 2;
  unsigned char* dst = o.dig +
      (((long long)b * o.tiles + tile) * ((long long)A.nred * A.ksteps) + step) * block;
  // PT: [part][digit][k half][row group][8 rows][16 B]; Q: [part][k half][digit][row group]...
  const bool wide = o.tile == PT;
  const int group = o.tile * 16;                     // the row groups of one digit and k half
  const int by_digit = wide ? 2 * group : group, by_half = wide ? group : ND * group;
  dst += kh * by_half + (rt >> 3) * 128 + (rt & 7) * 16;
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    unsigned long long w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
      w[i] = digits_of(part == 0 ? mine[i].x : mine[i].y, emax, part == 1 && o.conj != 0, bad);
#pragma unroll
    for (int l = 0; l < ND; ++l) {
      uint32_t h[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) h[q] = digit_pair(w[2 * q], w[2 * q + 1], l);
      *reinterpret_cast<uint4*>(dst + part * 2 * ND * group + l * by_digit) =
          make_uint4(h[0], h[1], h[2], h[3]);
    }
  }
}

struct GemmArgs {
  const unsigned char* pd;
  const unsigned char* qd;
  const int* pe;
  const int* qe;
  long long p_b, q_b;          // bytes between batches (0: shared)
  long long pe_b, qe_b;        // exponents between batches
  int p_rows, q_rows;          // output extent along P and Q
  int p_tiles, q_tiles;
  int ksteps, chunks, nred;    // per reduction term
  int ksplit, per_split;       // chunks (over all terms) of one split
  cplx* C;
  long long cp, cq, sc;        // output strides along P, along Q, between batches
  cplx* part;                  // split-K partials [ksplit][nbatch][p_rows][q_rows] (cp = 1)
  int nbatch;
  cplx alpha, beta;
  int plain;                   // alpha = 1, beta = 0
  int* status;
  const int* skip;
};

template <int QT>
__global__ void __launch_bounds__(GEMM_THREADS, 1) digit_gemm_kernel(const __grid_constant__ GemmArgs A) {
  constexpr int PITCH = q_pitch<QT>(), LEAD = LevelsOf<QT>::lead() * QT * 16;
  constexpr int Q_BLOCK = q_block(QT), STAGE = P_BLOCK + q_stage<QT>();
  constexpr int TMEM_COLS = 2 * NL * QT;
  constexpr int CW = QT / 2;                   // columns of an epilogue warp
  behind_next();
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NST * STAGE);
  uint64_t* empty = full + NST;
  uint64_t* acc_full = empty + NST;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  volatile int* fail = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* issued = fail + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pt = blockIdx.y, qt = blockIdx.x;
  const int bz = blockIdx.z / A.ksplit, sp = blockIdx.z % A.ksplit;
  const int all = A.nred * A.chunks;
  const int cbeg = sp * A.per_split, cend = min(all, cbeg + A.per_split);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 8);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // the zeros around the runs of Q's digits (the copies write only the runs)
  for (int e = threadIdx.x; e < NST * (q_stage<QT>() / 16); e += GEMM_THREADS)
    *reinterpret_cast<uint4*>(smem + e / (q_stage<QT>() / 16) * STAGE + P_BLOCK +
                              e % (q_stage<QT>() / 16) * 16) = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  behind_wait();
  if (A.skip && *A.skip) {
    if (warp == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(TMEM_COLS));
    return;
  }

  if (threadIdx.x == 0) {
    // producer: one contiguous block of each operand per k step
    const long long tsteps = (long long)A.nred * A.ksteps;
    const unsigned char* P = A.pd + bz * A.p_b + (long long)pt * tsteps * P_BLOCK;
    const unsigned char* Q = A.qd + bz * A.q_b + (long long)qt * tsteps * Q_BLOCK;
    int t = 0;
    bool live = true;
    for (int ch = cbeg; ch < cend && live; ++ch) {
      const int red = ch / A.chunks, c = ch % A.chunks;
      const int ns = min(STEPS, A.ksteps - c * STEPS);
      for (int k = 0; k < ns; ++k, ++t) {
        const int s = t % NST;
        if (t >= NST && !mbar_wait(&empty[s], (t / NST - 1) & 1, fail, A.status, 3)) {
          live = false;
          break;
        }
        const long long step = (long long)red * A.ksteps + c * STEPS + k;
        unsigned char* st = smem + s * STAGE;
        mbar_expect_tx(&full[s], P_BLOCK + Q_BLOCK);
        bulk_load(st, P + step * P_BLOCK, P_BLOCK, &full[s]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          bulk_load(st + P_BLOCK + LEAD + u * PITCH, Q + step * Q_BLOCK + u * (Q_BLOCK / 4),
                    Q_BLOCK / 4, &full[s]);
      }
    }
    *issued = t;
  } else if (threadIdx.x == 32) {
    // MMA issuer
    int t = 0;
    bool live = true;
    for (int ch = cbeg; ch < cend && live; ++ch) {
      const int ns = min(STEPS, A.ksteps - (ch % A.chunks) * STEPS);
      const int local = ch - cbeg;
      if (local > 0 && !mbar_wait(acc_empty, (local - 1) & 1, fail, A.status, 3)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int k = 0; k < ns; ++k, ++t) {
        const int s = t % NST;
        if (!mbar_wait(&full[s], (t / NST) & 1, fail, A.status, 3)) {
          live = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t p0 = smem_u32(smem + s * STAGE);
        mma_levels<LevelsOf<QT>, QT>(tmem, NL * QT, p0, PT * 16, 128, ND * (PT * KS * 2),
                                     PT * KS * 2, p0 + P_BLOCK + LEAD, PITCH, k == 0, false);
        mma_commit(&empty[s]);
      }
      if (live) mma_commit(acc_full);
    }
  } else if (warp >= 2) {
    // epilogue: warp w reads TMEM lanes 32 (w mod 4)..; warps 2-5 the first half of every
    // level's columns, warps 6-9 the other
    const int quad = warp & 3, half = (warp - 2) >> 2;
    const int prow = pt * PT + quad * 32 + lane;
    const int qcol0 = qt * QT + half * CW;
    const long long pext = (long long)A.p_tiles * PT, qext = (long long)A.q_tiles * QT;
    const int* pe = A.pe + bz * A.pe_b + prow;
    const int* qe = A.qe + bz * A.qe_b + qcol0;
    const uint32_t base = tmem + ((uint32_t)(quad * 32) << 16) + half * CW;
    double re[CW], im[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) re[c] = im[c] = 0.0;
    bool ok = true;
    for (int ch = cbeg; ch < cend; ++ch) {
      const int local = ch - cbeg;
      // (not __ldg: the split that writes the scales ends after this kernel has started)
      const int ep = __ldcg(pe + ch * pext);
      const int eqv = __ldcg(qe + ch * qext + (lane & (CW - 1)));      // column lane mod CW
      ok = mbar_wait(acc_full, local & 1, fail, A.status, 3);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int blk = 0; blk < CW / 2; ++blk) {     // four columns of re, then of im
        const int c0 = (blk >> 1) * 4;
        const bool imag = blk & 1;
        int eq[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) eq[c] = __shfl_sync(0xffffffffu, eqv, c0 + c);
        double x[1][4];
        read_levels4<1>(base + (imag ? NL * QT : 0) + c0, QT, 0, ep, eq, x);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (imag) im[c0 + c] = local == 0 ? x[0][c] : im[c0 + c] + x[0][c];
          else re[c0 + c] = local == 0 ? x[0][c] : re[c0 + c] + x[0][c];
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    }
    if (ok && prow < A.p_rows) {
      if (A.ksplit > 1) {
        cplx* D = A.part + (((long long)sp * A.nbatch + bz) * A.q_rows) * A.p_rows + prow;
#pragma unroll
        for (int c = 0; c < CW; ++c)
          if (qcol0 + c < A.q_rows) D[(long long)(qcol0 + c) * A.p_rows] = make_double2(re[c], im[c]);
      } else {
        cplx* D = A.C + bz * A.sc + prow * A.cp;
#pragma unroll
        for (int c = 0; c < CW; ++c) {
          if (qcol0 + c < A.q_rows) {
            cplx v = make_double2(re[c], im[c]);
            cplx* d = D + (qcol0 + c) * A.cq;
            if (!A.plain) {
              v = make_double2(A.alpha.x * re[c] - A.alpha.y * im[c],
                               A.alpha.x * im[c] + A.alpha.y * re[c]);
              if (A.beta.x != 0.0 || A.beta.y != 0.0) {
                const cplx o = *d;
                v.x += A.beta.x * o.x - A.beta.y * o.y;
                v.y += A.beta.x * o.y + A.beta.y * o.x;
              }
            }
            *d = v;
          }
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && *fail) {
    // a failed pipeline may still have copies in flight: the last one of each stage lands
    // (bounded) before the shared memory is released
    const int n = *issued;
    for (int s = 0; s < NST; ++s) {
      int last = -1;
      for (int u = s; u < n; u += NST) last = u;
      int none = 0;
      if (last >= 0) mbar_wait(&full[s], (last / NST) & 1, &none, A.status, 3);
    }
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS));
  }
}

// C = alpha sum_s part_s + beta C, splits in order
__global__ void __launch_bounds__(256) digit_reduce_kernel(GemmArgs A) {
  behind_next();
  behind_wait();
  if (A.skip && *A.skip) return;
  const long long mn = (long long)A.p_rows * A.q_rows, total = mn * A.nbatch;
  for (long long e = blockIdx.x * 256LL + threadIdx.x; e < total; e += (long long)gridDim.x * 256) {
    const cplx* p = A.part + e;
    cplx v = p[0];
    for (int s = 1; s < A.ksplit; ++s) {
      const cplx u = p[(long long)s * total];
      v.x += u.x;
      v.y += u.y;
    }
    const long long b = e / mn, r = e % mn;
    cplx* d = A.C + b * A.sc + (r % A.p_rows) * A.cp + (r / A.p_rows) * A.cq;
    if (!A.plain) {
      v = make_double2(A.alpha.x * v.x - A.alpha.y * v.y, A.alpha.x * v.y + A.alpha.y * v.x);
      if (A.beta.x != 0.0 || A.beta.y != 0.0) {
        const cplx o = *d;
        v.x += A.beta.x * o.x - A.beta.y * o.y;
        v.y += A.beta.x * o.y + A.beta.y * o.x;
      }
    }
    *d = v;
  }
}

constexpr size_t ALIGN = 256;
size_t up(size_t x) { return (x + ALIGN - 1) & ~(ALIGN - 1); }

struct Plan {
  int ksteps, chunks, tc;
  size_t row_p, row_q;       // bytes of one 128-row tile of P, one tile of Q (with scales)
};
Plan plan_of(int k, int nred, int qt = 32) {
  Plan p;
  p.ksteps = (k + KS - 1) / KS;
  p.chunks = (k + KC - 1) / KC;
  p.tc = p.chunks * nred;
  p.row_p = (size_t)p.ksteps * nred * P_BLOCK + (size_t)p.tc * PT * sizeof(int);
  p.row_q = (size_t)p.ksteps * nred * q_block(qt) + (size_t)p.tc * qt * sizeof(int);
  return p;
}

}  // namespace

namespace {
constexpr int SMS = 152;                      // of this chip
// Most CTAs with 16-column tiles: one per SM.  They read the 128-row operand twice as often, which
// L2 has room for as long as they run side by side; a second wave would cost more than the shorter
// main loop gives.  448 x 256 x 64 (64 CTAs) 15 against 21 us, 128 x 128 x 128 19 against 27.
constexpr int NARROW = SMS;
// Splits of the chunk loop that fill the GPU when there are few tiles: as many CTAs as leave at most
// four SMs idle where a whole number of splits does (50 tiles take three, 150 CTAs, and not four)
int splits_of(long long ntile, int chunks) {
  const long long ks = (SMS - 4 + ntile - 1) / ntile;
  return (int)(ks < chunks ? ks : chunks);
}
}  // namespace

size_t zgemm_digits_bytes(int m, int n, int k, int nbatch, int nred, int nbA, int nbB) {
  const Plan p = plan_of(k, nred);
  auto need = [&](int pr, int qr, int nbp, int nbq) {
    const size_t tp = (pr + PT - 1) / PT, tq = (qr + 31) / 32;      // (tiles of 16 need no more)
    const int ks = splits_of((long long)(tp * tq) * nbatch, p.tc);
    return tp * nbp * p.row_p + tq * nbq * p.row_q +
           (ks > 1 ? sizeof(cplx) * (size_t)pr * qr * nbatch * ks : 0);
  };
  const size_t a = need(m, n, nbA, nbB), b = need(n, m, nbB, nbA);
  return (a > b ? a : b) + 8 * ALIGN;
}

// C_b = alpha sum_r A_{b,r} B_{b,r} + beta C_b by digit products; *taken = false (and nothing is
// launched) when the workspace cannot hold one tile row of each operand.
cudaError_t zgemm_digits(int m, int n, int k, int nbatch, int nred, cplx alpha, MatRef A, MatRef B,
                         cplx beta, cplx* C, long long ldc, long long sc, const int* skip,
                         const ZgWork& ws, cudaStream_t s, bool* taken) {
  *taken = false;
  static OncePerDevice smem;
  int dev = 0;
  cudaError_t ea = cudaGetDevice(&dev);
  if (ea == cudaSuccess)
    ea = smem.run(dev, cudaErrorInvalidDevice, [] {
      const cudaError_t e = cudaFuncSetAttribute(
          digit_gemm_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem(32));
      return e != cudaSuccess ? e
                              : cudaFuncSetAttribute(digit_gemm_kernel<16>,
                                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)gemm_smem(16));
    });
  if (ea != cudaSuccess) return ea;
  // the 128-row operand P is the side that pads least; on a tie the columns of C, whose stores
  // are then contiguous across the lanes
  auto tiles = [](int a, int t) { return (long long)(a + t - 1) / t; };
  const bool swap = tiles(n, PT) * tiles(m, 32) <= tiles(m, PT) * tiles(n, 32);
  auto operand = [&](const MatRef& M, int rows, long long rs, long long ks) {
    Operand o{};
    o.p = M.p;
    o.rs = rs;
    o.ks = ks;
    o.sb = M.sb;
    o.sr = M.sr;
    o.conj = M.conj;
    o.rows = rows;
    o.nb = M.sb == 0 ? 1 : nbatch;
    if (M.mix) {
      o.mix_start = M.mix->sp_start;
      o.mix_cu = M.mix->sp_cu;
      o.mix_val = M.mix->sp_val;
      o.xs = M.xs;
      o.dmb = M.dmb;
      o.d = M.mix->d;
      o.by_red = M.sr != 0;
    }
    return o;
  };
  const Operand a = operand(A, m, A.rs, A.cs), b = operand(B, n, B.cs, B.rs);
  Operand P = swap ? b : a, Q = swap ? a : b;
  const long long cp = swap ? 1 : ldc, cq = swap ? ldc : 1;
  const int tc = (k + KC - 1) / KC * nred;
  const long long narrow = tiles(P.rows, PT) * tiles(Q.rows, 16) * nbatch;
  const int QT = narrow * splits_of(narrow, tc) <= NARROW ? 16 : 32;
  const Plan pl = plan_of(k, nred, QT);
  P.tile = PT;
  Q.tile = QT;
  const int pt_all = (int)tiles(P.rows, PT), qt_all = (int)tiles(Q.rows, QT);
  // slabs of the batch, then of the rows of P, then of Q, that fit the workspace
  const size_t room = ws.bytes > 8 * ALIGN ? ws.bytes - 8 * ALIGN : 0;
  int nb = nbatch, np = pt_all, nq = qt_all;
  auto fits = [&](int bb, int pp, int qq) {
    return (size_t)pp * (P.nb == 1 ? 1 : bb) * pl.row_p +
               (size_t)qq * (Q.nb == 1 ? 1 : bb) * pl.row_q <= room;
  };
  if (!fits(1, 1, 1)) return cudaSuccess;
  if (!fits(nb, np, nq)) {
    nb = 1;
    while (np > 1 && !fits(1, np, nq)) np = (np + 1) / 2;
    while (nq > 1 && !fits(1, np, nq)) nq = (nq + 1) / 2;
  }
  for (int b0 = 0; b0 < nbatch; b0 += nb)
    for (int p0 = 0; p0 < pt_all; p0 += np)
      for (int q0 = 0; q0 < qt_all; q0 += nq) {
        const int bb = b0 + nb < nbatch ? nb : nbatch - b0;
        Operand p = P, q = Q;
        p.tiles = p0 + np < pt_all ? np : pt_all - p0;
        q.tiles = q0 + nq < qt_all ? nq : qt_all - q0;
        p.rows = P.rows - p0 * PT < p.tiles * PT ? P.rows - p0 * PT : p.tiles * PT;
        q.rows = Q.rows - q0 * QT < q.tiles * QT ? Q.rows - q0 * QT : q.tiles * QT;
        for (Operand* o : {&p, &q}) {
          const long long row0 = o == &p ? (long long)p0 * PT : (long long)q0 * QT;
          if (o->mix_start) {
            o->off0 = row0 * o->rs;
            o->b0 = b0;
          } else {
            o->p += row0 * o->rs + (long long)b0 * o->sb;
          }
        }
        p.nb = P.nb == 1 ? 1 : bb;
        q.nb = Q.nb == 1 ? 1 : bb;
        // carve the workspace
        unsigned char* w = reinterpret_cast<unsigned char*>(
            (reinterpret_cast<uintptr_t>(ws.p) + ALIGN - 1) & ~(uintptr_t)(ALIGN - 1));
        unsigned char* end = static_cast<unsigned char*>(ws.p) + ws.bytes;
        const long long tsteps = (long long)nred * pl.ksteps;
        const size_t pbytes = (size_t)p.tiles * tsteps * P_BLOCK;
        const size_t qbytes = (size_t)q.tiles * tsteps * q_block(QT);
        p.dig = w;
        w += up(pbytes * p.nb);
        q.dig = w;
        w += up(qbytes * q.nb);
        p.ex = reinterpret_cast<int*>(w);
        w += up(sizeof(int) * (size_t)p.nb * pl.tc * p.tiles * PT);
        q.ex = reinterpret_cast<int*>(w);
        w += up(sizeof(int) * (size_t)q.nb * pl.tc * q.tiles * QT);
        SplitArgs sa{};
        sa.o[0] = p;
        sa.o[1] = q;
        sa.K = k;
        sa.nred = nred;
        sa.ksteps = pl.ksteps;
        sa.chunks = pl.chunks;
        sa.skip = skip;
        const long long blk0 = (long long)p.nb * p.tiles * (PT / SR) * pl.tc;
        const long long blk1 = (long long)q.nb * q.tiles * (QT / SR) * pl.tc;
        sa.blocks0 = (int)blk0;
        if (blk0 + blk1 > 0x7fffffffLL) return cudaErrorInvalidValue;
        count_launch();
        cudaError_t e = launch_behind(digit_split_kernel, dim3((unsigned)(blk0 + blk1)), 256, 0, s, sa);
        if (e != cudaSuccess) return e;
        GemmArgs g{};
        g.pd = p.dig;
        g.qd = q.dig;
        g.pe = p.ex;
        g.qe = q.ex;
        g.p_b = p.nb == 1 ? 0 : (long long)pbytes;
        g.q_b = q.nb == 1 ? 0 : (long long)qbytes;
        g.pe_b = p.nb == 1 ? 0 : (long long)pl.tc * p.tiles * PT;
        g.qe_b = q.nb == 1 ? 0 : (long long)pl.tc * q.tiles * QT;
        g.p_rows = p.rows;
        g.q_rows = q.rows;
        g.p_tiles = p.tiles;
        g.q_tiles = q.tiles;
        g.ksteps = pl.ksteps;
        g.chunks = pl.chunks;
        g.nred = nred;
        g.C = C + (long long)b0 * sc + (long long)p0 * PT * cp + (long long)q0 * QT * cq;
        g.cp = cp;
        g.cq = cq;
        g.sc = sc;
        g.nbatch = bb;
        g.alpha = alpha;
        g.beta = beta;
        g.plain = alpha.x == 1.0 && alpha.y == 0.0 && beta.x == 0.0 && beta.y == 0.0;
        g.status = ws.status;
        g.skip = skip;
        // split the chunks when the tiles leave SMs idle
        const long long ntile = (long long)p.tiles * q.tiles * bb;
        int ks = splits_of(ntile, pl.tc);
        const size_t one = sizeof(cplx) * (size_t)p.rows * q.rows * bb;
        while (ks > 1 && w + one * ks > end) --ks;
        g.per_split = (pl.tc + ks - 1) / ks;
        g.ksplit = (pl.tc + g.per_split - 1) / g.per_split;
        g.part = reinterpret_cast<cplx*>(w);
        if ((long long)bb * g.ksplit > 65535 || p.tiles > 65535) return cudaErrorInvalidValue;
        count_launch();
        e = launch_behind(QT == 16 ? digit_gemm_kernel<16> : digit_gemm_kernel<32>,
                          dim3(q.tiles, p.tiles, bb * g.ksplit), GEMM_THREADS, gemm_smem(QT), s, g);
        if (e != cudaSuccess) return e;
        if (g.ksplit > 1) {
          long long blocks = ((long long)p.rows * q.rows * bb + 255) / 256;
          if (blocks > 152 * 8) blocks = 152 * 8;
          count_launch();
          e = launch_behind(digit_reduce_kernel, dim3((unsigned)blocks), 256, 0, s, g);
          if (e != cudaSuccess) return e;
        }
      }
  *taken = true;
  return cudaSuccess;
}

// ------------------------------------------------------------------------------------------
// workspaces
// ------------------------------------------------------------------------------------------
namespace {
// The library's stream-ordered pool, one per device, made at the first use.  It keeps at most
// kPoolKeep bytes between calls (zg_pool_trim gives them back); CUDA's pools are safe with
// several threads, and an allocation freed on one stream is handed to another only after it.
constexpr unsigned long long kPoolKeep = 512ULL << 20;
constexpr int kPoolDevices = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[kPoolDevices];

cudaError_t pool_of(cudaMemPool_t* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kPoolDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  if (!g_pool[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    if ((e = cudaMemPoolCreate(&p, &props)) != cudaSuccess) return e;
    unsigned long long keep = kPoolKeep;
    if ((e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
      cudaMemPoolDestroy(p);
      return e;
    }
    g_pool[dev] = p;
  }
  *out = g_pool[dev];
  return cudaSuccess;
}
}  // namespace

cudaError_t zg_pool_alloc(void** p, size_t bytes, cudaStream_t s) {
  cudaMemPool_t pool = nullptr;
  const cudaError_t e = pool_of(&pool);
  return e != cudaSuccess ? e : cudaMallocFromPoolAsync(p, bytes, pool, s);
}

cudaError_t zg_reserve(ZgWork& w, size_t bytes, cudaStream_t s) {
  if (bytes > w.limit) bytes = w.limit;
  if (w.fixed || bytes <= w.bytes) return cudaSuccess;
  bytes = up(bytes + bytes / 8);      // room to grow without a new allocation
  if (bytes > w.limit) bytes = w.limit;
  const bool pooled = w.pooled;
  const cudaError_t e = grow_block<cudaError_t>(
      w.p, w.bytes, bytes,
      [&](void** q, size_t n) { return pooled ? zg_pool_alloc(q, n, s) : cudaMalloc(q, n); },
      [&](void* q) { pooled ? cudaFreeAsync(q, s) : cudaFree(q); },
      [](cudaError_t r) { return r == cudaErrorMemoryAllocation; });
  if (e == cudaErrorMemoryAllocation) cudaGetLastError();      // the caller goes on with what there is
  return e;
}

void zg_free(ZgWork& w, cudaStream_t s) {
  if (w.p) {
    if (w.pooled) cudaFreeAsync(w.p, s);
    else cudaFree(w.p);
  }
  w.p = nullptr;
  w.bytes = 0;
}

void zg_pool_trim() {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  for (cudaMemPool_t p : g_pool)
    if (p) cudaMemPoolTrimTo(p, 0);
}

}  // namespace tdmrg
