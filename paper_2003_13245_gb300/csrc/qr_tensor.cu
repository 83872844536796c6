// Gauge QR with its projections on the tensor cores: the factorisation, skipping and completion of
// qr_blocked.cu (blocked Gram-Schmidt of 16 columns at a time, deterministic completion) in one
// cooperative launch, with Q^H V, V^H V and Q P taken as digit products (the scheme of
// zgemm_digits.cu) instead of FP64 FMAs.
//
// CTA g owns a slice of at most 128 rows of Y, Q and the working block V (shared memory, FP64).
// Up to 256 columns: the accepted vectors enter the products in tiles of 128.
// The digits of the accepted columns of its slice are kept in global memory in the two operand
// forms the products need (K = rows for Q^H V, K = columns for Q P); both are private to the CTA
// and stream through a two-stage ring of bulk copies.  The first form has one scale per column,
// the second one per row, with a bit to spare: a row that a later column outgrows is written
// again from Q.
//
// Per block of 16 columns a pass is
//  1. digits of V; P = Q^H V (accumulators in TMEM columns 0-255) and V^H V (columns 256-511);
//     cross-CTA sums of both;
//  2. V -= Q P, and P^H P (columns 256-511; every CTA for itself).
// V^H V - P^H P is the Gram matrix of what is left, unless less than 1e-8 of some norm^2 is left:
// then a second pass follows (before it, where next to nothing is left of any column, as with
// dependent columns, their norms alone tell whether all of them are skipped).  Then, as in
// qr_blocked.cu, Gram-Schmidt with skips inside the block in Gram form; the triangular inverse is
// built beside it, so that the new columns are one product V M.  A column that keeps less than 1e-8
// of its norm^2 starts the next block.  Where one kept less than a quarter, the rounding of the first
// round shows: a second round projects the new columns (orthonormal to 1e-8) once more and corrects
// them by the series of the Cholesky factor of 1 + E, without the serial chain.  Graded columns, as
// a center matrix has them, thus take two passes for 16 columns instead of a block for every few.
//
// Completion of skipped positions runs the same blocks over the candidates (columns of E, then
// unit vectors); the first pass rejects every candidate in the span of the accepted columns at
// once (residual^2 = ||e||^2 - |P|^2 <= 1e-4 ||e||^2), so 16 rejections cost one pass.
//
// Bound: latency.  A block of 8192 x 128 takes ~165 us: two to four grid barriers of ~1.3 us a pass,
// two tensor-core products a pass (64 instructions a k step, the ring's copies from L2), reading their
// levels back, the digits, the serial 16-column factorisation (~16 us) and the FP64 product V M
// (3-10 us); the FP64 work per column does not grow with the number of accepted columns.
//
// Measured on GB300 against qr_blocked.cu (FP64 FMAs), us.  "parallel": random columns, nearly
// parallel; "graded": singular values from 1 to e^-9, mixed; "rank 2": all but two columns are
// completed from 7 n candidates of which n lie in the span:
//   m x n        parallel       graded         rank 2
//   64 x 16        87 /   74     257 /   77     676 /  177
//   256 x 32      161 /  194     358 /  198    1546 /  326
//   1024 x 64     336 /  429     706 /  460    3702 /  615
//   256 x 128     803 / 1056    1028 / 1064    7546 / 1362
//   1024 x 128    871 / 1032    1174 / 1193    9628 / 1392
//   2048 x 128   1062 / 1002    1523 / 1057   12481 / 1392
//   8192 x 128   2360 / 1164    3912 / 1330   19450 / 1706
//   8192 x 128 on 76 CTAs (two lanes)  3949 / 1442 (parallel), 6746 / 1644, 25157 / 2204
// The rule goes by size alone, since neither the grading nor the rank is known before the call.  What a
// sweep brings is graded or rank deficient (center matrices of truncated chains): there this kernel is
// at par for 128 columns of few rows and faster elsewhere; columns that are nearly parallel and few
// rows (0.76-0.84 of the FMA kernel's speed) are the price.  Below nine columns the other kernel is the
// faster one at full rank (256 x 4: 55 against 95 us), where such bonds, at the ends of a chain,
// mostly are.  About 32 rows per CTA: fewer rows raise the number of partial sums, more the FP64
// product V M.  With the digit pairs of all levels in 28 instructions of different width on shared
// columns (an order that is not promised) 8192 x 128 took 1114 (graded).
#include "umma.cuh"
#include "workspace.h"

namespace tdmrg {

using namespace dig;

namespace {

constexpr int QB = 16;                          // columns per block
constexpr int QT_THREADS = 256;
constexpr int MAXR = 128;                       // rows of a CTA
constexpr int MAXN = 256;                       // columns
constexpr int TILE = 128;                       // accepted vectors of one product
constexpr int MINN = 9;                         // fewer: qr_blocked.cu (one block, no projection)
constexpr int GROUP = 2 * ND * 2 * 128;         // digits of 8 rows x 16 k: 3584 bytes
constexpr int RING = 16 * GROUP;                // one k step of 128 rows: 57344 bytes
// digits of B (16 columns): four runs (part, k half) per k step, a block of zeros before each and one
// behind the last.  Four level groups (16 x 4 instructions per k step) because they need no longer
// lead: one group (7 x 4) would take 41 KB more shared memory than there is
using Levels = Groups<4, 0x85310>;
constexpr int RUN = (Levels::lead() + ND) * 256;   // one run: 2048 bytes
constexpr int BSTEP = 4 * RUN;                  // 16 columns x 16 k: 8192 bytes
constexpr int LEAD = Levels::lead() * 256;
constexpr int BDIG = 8 * BSTEP + 256;           // 65792 bytes
constexpr int PASSES = 4;                       // projections of a block, at most (and a second round)
// smallest part of a norm^2 that may be left where the rest is taken off in the Gram matrix
// (rounding of 2^-53 is then up to 1e-8 of what is left; the second round takes that out)
constexpr double KEEP = 1e-8;
// a correction whose coefficients are below it is formed in FP32: 16 terms of 2^-32 rounded at 2^-24
constexpr double SMALL = 2.3283064365386963e-10;
constexpr int E_EMPTY = -100000;
constexpr int TMEM_COLS = 512;
constexpr int IM = NL * QB;                     // im levels after the re levels

struct QtArgs {
  int m, n, p;
  QrRef Y, E;
  cplx* Q;
  cplx* R;
  cplx* part;               // [2][G][PS], used in turn
  cplx* fin;                // [PASSES + 1][PS]
  int PS;
  unsigned char* dig;       // per CTA: form 1 then form 2
  long long dig_cta;        // bytes of one CTA
  int rows;                 // rows of a CTA
  unsigned* bar;
  int* status;
  long long wait;
  unsigned char* acc_out;
  int* src_out;
  double rank_tol, complete_tol;
};

__device__ __forceinline__ double wsum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ bool qt_barrier(const QtArgs& A, unsigned& epoch, int* s_ok) {
  const unsigned G = gridDim.x;
  __syncthreads();
  ++epoch;
  if (threadIdx.x == 0) {
    volatile unsigned* vbar = A.bar;
    volatile int* vstat = A.status;
    const unsigned target = epoch * G;
    __threadfence();
    atomicAdd(A.bar, 1u);
    int ok = 1;
    const long long t0 = clock64();
    while (*vbar < target) {
      if (*vstat) { ok = 0; break; }
      if (clock64() - t0 > A.wait) {
        atomicExch(A.status, 1);
        ok = 0;
        break;
      }
    }
    __threadfence();
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

// fin[0..cnt) = sum over the CTAs of part[.][0..cnt) in a fixed order.  Every CTA sums a slice of
// the entries and a second barrier makes all of them readable; where all partial sums are few,
// every CTA sums them itself into its shared copy `own` (the same order, so the same result) and
// the second barrier is left out (a CTA may then still read partial sums when another goes on:
// two sets of them are used in turn).  Without `fin` (few entries) always so.  Returns where to
// read the sums.
constexpr int OWN = 512;                        // entries a CTA may sum for itself
__device__ const cplx* qt_reduce(const QtArgs& A, int cnt, const cplx* part, cplx* fin, cplx* own,
                                 unsigned& ep, int* s_ok) {
  const int G = gridDim.x;
  if (G > 1) {
    if (!qt_barrier(A, ep, s_ok)) return nullptr;
  } else {
    __syncthreads();
  }
  const bool alone = !fin || (cnt <= OWN && cnt * G <= 4096);
  const int per = alone ? cnt : (cnt + G - 1) / G;
  const int lo = alone ? 0 : blockIdx.x * per, hi = min(cnt, lo + per);
  cplx* out = alone ? own : fin;
  // L lanes per entry, so that one round of loads covers the slice where possible
  int L = 32;
  while (L > 1 && (per * L > QT_THREADS || L > G)) L >>= 1;
  const int sub = threadIdx.x & (L - 1);
  for (int e0 = lo; e0 < hi; e0 += QT_THREADS / L) {
    const int e = e0 + threadIdx.x / L;
    double ax = 0.0, ay = 0.0;
    if (e < hi) {
      const cplx* src = part + e;
#pragma unroll 4
      for (int g = sub; g < G; g += L) {
        const cplx u = __ldcg(src + (long long)g * A.PS);
        ax += u.x;
        ay += u.y;
      }
    }
    for (int o = L >> 1; o > 0; o >>= 1) {
      ax += __shfl_xor_sync(0xffffffffu, ax, o);
      ay += __shfl_xor_sync(0xffffffffu, ay, o);
    }
    if (sub == 0 && e < hi) {
      out[e] = make_double2(ax, ay);
      if (alone && fin && blockIdx.x == 0) fin[e] = make_double2(ax, ay);   // R is formed from it
    }
  }
  if (alone) {
    __syncthreads();
    return own;
  }
  return qt_barrier(A, ep, s_ok) ? fin : nullptr;
}

__device__ __forceinline__ cplx qt_load(const QrRef& Y, long long r, long long c) {
  const long long off = r * Y.rs + (c < Y.cb ? c * Y.cs : (c % Y.cb) * Y.cs + (c / Y.cb) * Y.cbs);
  const cplx v = Y.p[off];
  return Y.conj ? make_double2(v.x, -v.y) : v;
}

struct Pipe {
  uint64_t* full;           // [2] ring stages
  uint64_t* empty;          // [2]
  uint64_t* done;           // one GEMM's accumulators
  uint64_t* side;           // Q P: its B^H B, which comes after
  uint32_t it;              // ring steps used so far
  uint32_t gemms;           // GEMMs completed so far
  uint32_t sides;
  volatile int* fail;
  int* status;
};

// Issued by thread 0.  D += sum over S k steps of A_s B_s: A from `src` (step s at s * stride,
// `bytes` of it, at `off` of a stage) through the ring, B in shared memory at bdig + s * BSTEP.
// conj: Q^H V (re = ArBr + AiBi, im = ArBi - AiBr), else Q P (re = ArBr - AiBi, im = ArBi + AiBr).
// gram_steps: also B^H B of the same B tiles into columns 256.. (A = the B tile itself, its rows
// beyond 16 unused): with Q^H V while the first copies are on their way, with Q P behind it, so that
// it runs while V is updated.
__device__ void qt_gemm(Pipe& P, uint32_t tmem, unsigned char* ring, int off,
                        const unsigned char* bdig,
                        const unsigned char* src, long long stride, uint32_t bytes, int S,
                        bool conj, int gram_steps) {
  bool ok = true;
  const uint32_t it0 = P.it;
  int issued = 0;
  auto load = [&](int s) {
    const int st = (it0 + s) & 1;
    mbar_expect_tx(&P.full[st], bytes);
    bulk_load(ring + st * RING + off, src + s * stride, bytes, &P.full[st]);
    ++issued;
  };
  for (int s = 0; s < S && s < 2; ++s) load(s);
  const uint32_t b0 = smem_u32(bdig) + LEAD;
  auto gram = [&] {
    for (int s = 0; s < gram_steps; ++s)
      mma_levels<Levels, QB>(tmem + 2 * IM, IM, b0 + s * BSTEP, RUN, 128, 2 * RUN, 256,
                             b0 + s * BSTEP, RUN, s == 0, true);
  };
  if (conj) gram();
  for (int s = 0; s < S; ++s) {
    const int st = (it0 + s) & 1;
    const uint32_t par = ((it0 + s) >> 1) & 1;
    if (!mbar_wait(&P.full[st], par, P.fail, P.status, 1)) {
      ok = false;
      break;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    mma_levels<Levels, QB>(tmem, IM, smem_u32(ring + st * RING), 128, GROUP, GROUP / 2, 256,
                           b0 + s * BSTEP, RUN, s == 0, conj);
    mma_commit(&P.empty[st]);
    if (s + 2 < S) {
      if (!mbar_wait(&P.empty[st], par, P.fail, P.status, 1)) {
        ok = false;
        break;
      }
      load(s + 2);
    }
  }
  mma_commit(P.done);
  if (!conj && gram_steps > 0) {
    gram();
    mma_commit(P.side);
  }
  P.it += S;
  if (!ok) {
    // copies in flight land (bounded) before the shared memory can be released
    int none = 0;
    for (int s = issued > 2 ? issued - 2 : 0; s < issued; ++s)
      mbar_wait(&P.full[(it0 + s) & 1], ((it0 + s) >> 1) & 1, &none, P.status, 1);
  }
}

// the thread's 8 complex results of one accumulator set: lane = row, columns t0 .. t0 + 7
__device__ __forceinline__ void qt_read(uint32_t addr, int eA, const int* eB, cplx (&out)[8]) {
#pragma unroll
  for (int c0 = 0; c0 < 8; c0 += 4) {
    const int e[4] = {eB[c0], eB[c0 + 1], eB[c0 + 2], eB[c0 + 3]};
    double x[2][4];
    read_levels4<2>(addr + c0, QB, IM, eA, e, x);
#pragma unroll
    for (int c = 0; c < 4; ++c) out[c0 + c] = make_double2(x[0][c], x[1][c]);
  }
}

// 4 consecutive k of one part (re or im) of a row as digits: 8-byte stores, 256 bytes per digit
__device__ __forceinline__ void qt_store(const cplx* x, int stride, int live, int part, int emax,
                                         bool bad, unsigned char* dst) {
  unsigned long long w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    w[i] = i < live ? digits_of(part == 0 ? x[i * stride].x : x[i * stride].y, emax, false, bad)
                    : 0x0080808080808080ULL;
#pragma unroll
  for (int l = 0; l < ND; ++l)
    *reinterpret_cast<uint2*>(dst + l * 256) =
        make_uint2(digit_pair(w[0], w[1], l), digit_pair(w[2], w[3], l));
}

struct Shared {
  cplx G[QB][QB];            // Gram matrix of the block
  cplx R[QB][QB];            // its triangular factor
  cplx M[QB][QB];            // and the inverse
  cplx u[2][QB], y[QB];      // factors of one step (u of alternate steps)
  double inv;
  double ref[QB];            // norm^2 of the column before the last projection
  double hh[8][QB];          // partial sums of |P|^2
  double lim[QB];            // completion: smallest residual norm of a candidate that is taken
  int em[QB];                // largest biased exponent of a column (digit scale)
  int ev[QB];                // its digit scale E
  short idx[MAXN];           // column of Q of every accepted vector, in order of acceptance
  int ec[MAXN];              // form 1: scale of every accepted vector (this CTA's rows)
  int er[MAXR];              // form 2: scale of every row (E_EMPTY: nothing but zeros so far)
  int rnew[MAXR];            // largest biased exponent of a row's new entries
  unsigned char acc[MAXN];   // accepted (main factorisation) or filled (completion)
  int take[QB];
  int src[QB];               // block column of the block's i-th accepted vector
  int drop[QB];              // skipped before the in-block factorisation
  double red[32];
  int ok, fail, done, last, any, near, refine;
  uint32_t tmem;
  uint64_t bar[6];
};

}  // namespace

__global__ void __launch_bounds__(QT_THREADS, 1) gauge_qr_tensor_kernel(QtArgs A) {
  extern __shared__ unsigned char raw[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(raw) + 127) & ~(uintptr_t)127);
  unsigned char* ring = base;                                   // 2 * RING
  unsigned char* bdig = base + 2 * RING;                        // BDIG
  cplx* V = reinterpret_cast<cplx*>(bdig + BDIG);               // [QB][MAXR + 1]
  constexpr int LDV = MAXR + 1;
  cplx* H = reinterpret_cast<cplx*>(ring + RING);               // [TILE][QB], in stage 1
  // sums of a small reduction, behind it: read before the next product's copies are issued
  cplx* own = H + TILE * QB;                                    // [OWN]
  static_assert(sizeof(cplx) * (TILE * QB + OWN) <= RING, "stage 1");
  __shared__ Shared S;

  const int m = A.m, n = A.n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0 = blockIdx.x * A.rows;
  const int nr = max(0, min(m, r0 + A.rows) - r0);
  const int rsteps = (A.rows + 15) / 16, rgroups = (A.rows + 7) / 8;
  const int ngroups = (n + 7) / 8;
  unsigned char* d1 = A.dig + blockIdx.x * A.dig_cta;           // [rstep][column group][GROUP]
  unsigned char* d2 = d1 + (long long)rsteps * ngroups * GROUP; // [column step][row group][GROUP]
  const long long s1 = (long long)ngroups * GROUP, s2 = (long long)rgroups * GROUP;
  const long long pset = (long long)gridDim.x * A.PS;
  const cplx* part = A.part;
  cplx* mypart = A.part + (long long)blockIdx.x * A.PS;
  unsigned ep = 0;
  bool alive = true;

  Pipe P{&S.bar[0], &S.bar[2], &S.bar[4], &S.bar[5], 0, 0, 0, &S.fail, A.status};
  if (tid == 0) {
    for (int i = 0; i < 6; ++i) mbar_init(&S.bar[i], 1);
    S.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&S.tmem)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (blockIdx.x == 0)
    for (int e = tid; e < n * n; e += QT_THREADS) A.R[e] = make_double2(0.0, 0.0);
  for (int i = tid; i < n; i += QT_THREADS) S.acc[i] = 0;
  for (int i = tid; i < MAXR; i += QT_THREADS) S.er[i] = E_EMPTY;
  // the zeros around the runs of bdig (the digits are written over the rest)
  for (int e = tid; e < BDIG / 16; e += QT_THREADS)
    reinterpret_cast<uint4*>(bdig)[e] = make_uint4(0u, 0u, 0u, 0u);
  // ||Y||_F (summed over the CTAs with the first block's Gram matrix)
  {
    double s = 0.0;
    for (long long e = tid; e < (long long)nr * n; e += QT_THREADS) {
      const bool cfast = A.Y.cs == 1;
      const int r = (int)(cfast ? e / n : e % nr), c = (int)(cfast ? e % n : e / nr);
      const cplx y = qt_load(A.Y, r0 + r, c);
      s = fma(y.x, y.x, fma(y.y, y.y, s));
    }
    s = wsum(s);
    if (lane == 0) S.red[warp] = s;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < QT_THREADS / 32; ++w) t += S.red[w];
      mypart[QB * QB] = make_double2(t, 0.0);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = S.tmem;
  double thr = 0.0, thr2 = 0.0;       // known after the first reduction
  int na = 0;               // accepted vectors
  int j0 = 0;               // next column of Y (main) -- n when the factorisation is done
  int open = 0;             // completion: next position to look at
  long long cand = 0;       // completion: next candidate
  bool main_phase = true, started = false;

  while (alive) {
    int bsz;
    if (main_phase) {
      bsz = min(QB, n - j0);
    } else {
      if (na >= n) break;
      const long long left = (long long)A.p + m - cand;
      if (left <= 0) {
        if (tid == 0 && blockIdx.x == 0) atomicExch(A.status, 2);
        break;
      }
      bsz = (int)(left < QB ? left : QB);
    }
    // ---- load the block (missing columns are zero)
    {
      const QrRef& src = main_phase ? A.Y : A.E;
      const long long c0 = main_phase ? j0 : cand;
      const bool rfast = src.rs == 1;
      for (int e = tid; e < QB * nr; e += QT_THREADS) {
        const int t = rfast ? e / nr : e % QB, r = rfast ? e % nr : e / QB;
        cplx v = make_double2(0.0, 0.0);
        if (t < bsz) {
          if (main_phase || c0 + t < A.p) v = qt_load(src, r0 + r, c0 + t);
          else if (c0 + t - A.p == r0 + r) v.x = 1.0;
        }
        V[t * LDV + r] = v;
      }
    }
    if (tid < QB) S.drop[tid] = tid < bsz ? 0 : 1;
    __syncthreads();
    // ---- projection passes
    bool private_r = false;   // some of the sums were not published
    int npass = 0;            // passes of the first round
    bool all_dropped = false;
    bool refine = false;      // second round: one pass over the block's new columns
    bool small = false;       // it changes them by less than SMALL
    for (;;) {
      for (int pass = npass; pass <= PASSES; ++pass) {
        // digits of V, one scale per column (two columns per warp)
        {
          int e2[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int t = 2 * warp + u;
            int e = 0;
            for (int r = lane; r < nr; r += 32) {
              const cplx v = V[t * LDV + r];
              e = max(e, max(bexp(v.x), bexp(v.y)));
            }
            e2[u] = __reduce_max_sync(0xffffffffu, e);
            if (lane == 0) S.ev[t] = e2[u] == 0x7ff ? E_NONFINITE : max(e2[u], 1) - 1022;
          }
          for (int k = lane; k < 16 * rsteps; k += 32) {     // column, part, group of 4 rows
            const int u = k & 1, part = (k >> 1) & 1, q = k >> 2;
            const int t = 2 * warp + u, em = u ? e2[1] : e2[0];
            qt_store(V + t * LDV + q * 4, 1, min(4, nr - q * 4), part, max(em, 1), em == 0x7ff,
                     bdig + LEAD + (q >> 2) * BSTEP + (2 * part + ((q >> 1) & 1)) * RUN + t * 16 +
                         (q & 1) * 8);
          }
        }
        asm volatile("fence.proxy.async;" ::: "memory");
        __syncthreads();
        // P and V^H V, a tile of accepted vectors at a time.  With at most 96 vectors in a tile they
        // sit in its rows 32.., so that the warps of rows 0-31 have the Gram matrix alone.
        for (int i0 = 0; i0 == 0 || i0 < na; i0 += TILE) {
          const int ni = min(TILE, na - i0);
          const bool g0 = i0 == 0;
          const int shift = g0 && ni <= TILE - 32 ? 32 : 0;
          if (tid == 0)
            qt_gemm(P, tmem, ring, shift / 8 * GROUP, bdig, d1 + (long long)(i0 / 8) * GROUP, s1,
                    (uint32_t)((ni + 7) / 8 * GROUP), ni > 0 ? rsteps : 0, true, g0 ? rsteps : 0);
          __syncwarp();
          alive = mbar_wait(P.done, P.gemms & 1, P.fail, A.status, 1);
          ++P.gemms;
          alive = __syncthreads_and(alive ? 1 : 0) != 0;
          if (!alive) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int quad = warp & 3, t0 = (warp >> 2) * 8;
          const int row = quad * 32 + lane - shift;
          const uint32_t addr = tmem + ((uint32_t)(quad * 32) << 16) + t0;
          cplx out[8];
          if (quad * 32 >= shift && quad * 32 - shift < ni) {
            qt_read(addr, S.ec[i0 + min(row, ni - 1)], S.ev + t0, out);
            if (row < ni)
#pragma unroll
              for (int c = 0; c < 8; ++c) mypart[(i0 + row) * QB + t0 + c] = out[c];
          }
          if (g0 && quad == 0) {
            qt_read(addr + 2 * IM, S.ev[lane & 15], S.ev + t0, out);
            if (lane < QB)
#pragma unroll
              for (int c = 0; c < 8; ++c) mypart[na * QB + lane * QB + t0 + c] = out[c];
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          if (i0 + TILE < na) {
            __syncthreads();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
        }
        if (!alive) break;
        cplx* fin = A.fin + (long long)pass * A.PS;
        const int cnt = na * QB + QB * QB + (started ? 0 : 1);
        const cplx* sum = qt_reduce(A, cnt, part, fin, own, ep, &S.ok);
        if (!sum) {
          alive = false;
          break;
        }
        mypart += part == A.part ? pset : -pset;
        part = part == A.part ? A.part + pset : A.part;
        if (sum == own) private_r = true;
        if (!refine) npass = pass + 1;
        auto take_sum = [&](int e) { return sum == own ? own[e] : __ldcg(sum + e); };
        if (!started) {
          started = true;
          const double y2 = take_sum(QB * QB).x;
          if (!(y2 < 1.7976931348623157e308)) {
            // Inf or NaN in Y: every column is skipped
            bsz = n;
            all_dropped = true;
            break;
          }
          thr = A.rank_tol * sqrt(y2);
          thr2 = thr * thr;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        S.G[tid >> 4][tid & 15] = take_sum(na * QB + tid);
        // one tile of P: into shared memory, its |P|^2 and its scale per column
        cplx hreg[TILE / QB];
        double hsum = 0.0;
        auto load_p = [&](int i0) {
          const int t = tid & 15, q = tid >> 4;
          if (tid < QB) S.em[tid] = 0;
#pragma unroll
          for (int k = 0; k < TILE / QB; ++k) {
            const int i = i0 + k * QB + q;
            hreg[k] = i < na ? take_sum(i * QB + t) : make_double2(0.0, 0.0);
          }
          __syncthreads();
          int e = 0;
#pragma unroll
          for (int k = 0; k < TILE / QB; ++k)
            if (i0 + k * QB < na) {
              const cplx h = hreg[k];
              if (i0 + k * QB + q < na) H[(k * QB + q) * QB + t] = h;
              e = max(e, max(bexp(h.x), bexp(h.y)));
            }
          atomicMax(&S.em[t], e);
        };
        auto square_p = [&](int i0) {
#pragma unroll
          for (int k = 0; k < TILE / QB; ++k)
            if (i0 + k * QB < na)
              hsum = fma(hreg[k].x, hreg[k].x, fma(hreg[k].y, hreg[k].y, hsum));
        };
        // what to do with each column; rejections of candidates are wanted before Q P, all else runs
        // while the tensor cores form it
        auto decide = [&] {
          const int t = tid & 15;
          const double s = hsum + __shfl_xor_sync(0xffffffffu, hsum, 16);
          if (lane < 16) S.hh[warp][t] = s;
          __syncthreads();
          if (tid < QB) {
            const double vv = S.G[tid][tid].x;
            double h = 0.0;
            for (int w = 0; w < QT_THREADS / 32; ++w) h += S.hh[w][tid];
            int drop = S.drop[tid];
            if (main_phase) {
              if (!(vv > thr2)) drop = 1;
            } else if (pass == 0) {
              S.lim[tid] = A.complete_tol * sqrt(vv);
              // in the span of the accepted vectors (or zero, or not finite)
              if (!(vv - h > A.complete_tol * A.complete_tol * vv)) drop = 1;
            }
            S.drop[tid] = drop;
            S.ref[tid] = vv;
            // first pass: V^H V - P^H P stands in for the Gram matrix of what is left, where that is
            // not too small a part; later ones: V^H V as it is, where P does not change it
            const bool more = !drop && (pass == 0 ? !(vv - h > KEEP * vv) : h > 6.9e-18 * vv);
            const bool away = !drop && vv - h > 2e-15 * vv;
            const unsigned mm = __ballot_sync(0xffffu, more), dd = __ballot_sync(0xffffu, !drop);
            const unsigned aa = __ballot_sync(0xffffu, away);
            if (tid == 0) {
              S.last = mm == 0;
              S.any = dd != 0;
              S.near = main_phase && pass == 0 && aa == 0;
            }
          }
          __syncthreads();
        };
        const bool first = !refine && pass == 0;
        if (first) {
          for (int i0 = 0; i0 < na; i0 += TILE) {
            load_p(i0);
            square_p(i0);
            if (i0 + TILE < na) __syncthreads();
          }
          decide();
          if (!S.any) {
            all_dropped = true;
            break;
          }
        }
        // V -= Q P, a tile of accepted vectors at a time
        for (int i0 = 0; i0 < na; i0 += TILE) {
          if (!first || na > TILE) {
            load_p(i0);
            __syncthreads();
          }
          const int ni = min(TILE, na - i0), isteps = (ni + 15) / 16;
          {
            const int t = tid & 15;
            const int em = max(S.em[t], 1);
            const bool bad = em == 0x7ff;
            if (tid < QB) S.ev[t] = bad ? E_NONFINITE : em - 1022;
            for (int k = tid >> 4; k < 8 * isteps; k += 16) {     // part, group of 4 columns of Q
              const int part = k & 1, q = k >> 1;
              qt_store(H + q * 4 * QB + t, QB, min(4, ni - q * 4), part, em, bad,
                       bdig + LEAD + (q >> 2) * BSTEP + (2 * part + ((q >> 1) & 1)) * RUN + t * 16 +
                           (q & 1) * 8);
            }
          }
          asm volatile("fence.proxy.async;" ::: "memory");
          __syncthreads();
          // with a single pass also P^H P, which every CTA forms for itself
          const bool corr = first && S.last;
          if (tid == 0)
            qt_gemm(P, tmem, ring, 0, bdig, d2 + (long long)(i0 / 16) * s2, s2, (uint32_t)s2, isteps,
                    false, corr ? isteps : 0);
          __syncwarp();
          if (!first && !refine) {
            square_p(i0);
            if (i0 + TILE >= na) decide();
          }
          alive = mbar_wait(P.done, P.gemms & 1, P.fail, A.status, 1);
          ++P.gemms;
          alive = __syncthreads_and(alive ? 1 : 0) != 0;
          if (!alive) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int quad = warp & 3, t0 = (warp >> 2) * 8;
          if (quad * 32 < nr) {
            cplx out[8];
            const int r = quad * 32 + lane;
            qt_read(tmem + ((uint32_t)(quad * 32) << 16) + t0, S.er[min(r, nr - 1)], S.ev + t0, out);
            if (r < nr)
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                cplx& v = V[(t0 + c) * LDV + r];
                v = make_double2(v.x - out[c].x, v.y - out[c].y);
              }
          }
          if (corr) {
            alive = mbar_wait(P.side, P.sides & 1, P.fail, A.status, 1);
            ++P.sides;
            alive = __syncthreads_and(alive ? 1 : 0) != 0;
            if (!alive) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          if (corr && quad == 0) {
            cplx out[8];
            qt_read(tmem + 2 * IM + t0, S.ev[lane & 15], S.ev + t0, out);
            if (lane < QB)
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                cplx& g = S.G[lane][t0 + c];
                g = make_double2(g.x - out[c].x, g.y - out[c].y);
              }
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncthreads();
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        if (!alive || refine) break;
        if (!S.any) {
          all_dropped = true;
          break;
        }
        if (S.last || npass == PASSES) break;
        if (S.near) {
          // next to nothing is left of any column: their norms tell whether they are skipped, without
          // another projection
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int t = 2 * warp + u;
            double q = 0.0;
            for (int r = lane; r < nr; r += 32) {
              const cplx v = V[t * LDV + r];
              q = fma(v.x, v.x, fma(v.y, v.y, q));
            }
            q = wsum(q);
            if (lane == 0) mypart[t] = make_double2(q, 0.0);
          }
          if (!qt_reduce(A, QB, part, nullptr, own, ep, &S.ok)) {
            alive = false;
            break;
          }
          mypart += part == A.part ? pset : -pset;
          part = part == A.part ? A.part + pset : A.part;
          if (tid < QB) {
            const int drop = S.drop[tid] || !(own[tid].x > thr2);
            S.drop[tid] = drop;
            const unsigned dd = __ballot_sync(0xffffu, !drop);
            if (tid == 0) S.any = dd != 0;
          }
          __syncthreads();
          if (!S.any) {
            all_dropped = true;
            break;
          }
        }
      }
      if (!alive || all_dropped) break;
      if (!refine) {
        // ---- Gram-Schmidt with skips inside the block (Gram form, right-looking), the inverse of
        // the triangular factor beside it.  Thread e holds the pair (a, b), a <= b, numbered by
        // falling b: at step s the pairs with b > s are the first ones.  It carries G_ab until row a
        // is taken (then R_ab), and the inverse's M_ab from then on; both are updated by the same
        // product of a column factor u_a (conj(R_sa) for a > s, M_as for a <= s) and R_sb.
        const int room = n - na;             // completion: positions left
        if (tid == 0) S.refine = 0;
        __syncthreads();
        if (warp < 5) {
          int b = QB - 1, rem = tid;
          while (b >= 0 && rem > b) rem -= b-- + 1;
          const int a = rem;                 // b < 0: no pair
          cplx g = b >= 0 ? S.G[a][b] : make_double2(0.0, 0.0);
          int taken = 0, s = 0;
          for (; s < bsz; ++s) {
            if (a == s && b == s) {
              // positive doubles compare like their bits (a negative rho is below everything):
              // integer comparisons keep the FP64 pipe out of the serial chain
              const double rho = g.x;
              const long long rb = __double_as_longlong(rho);
              int take = 0;
              double inv = 0.0, nrm = 0.0;
              if (!main_phase && taken >= room) take = -1;
              else if (!S.drop[s]) {
                // cancellation inside the block: this column starts the next block
                if (taken > 0 && rb < __double_as_longlong(KEEP * S.ref[s])) take = -1;
                else if (rb > 0) {
                  inv = bexp(rho) > 0 ? rsqrt_series(rho) : rsqrt(rho);
                  nrm = rho * inv;
                  const double lim = main_phase ? thr : S.lim[s];
                  take = __double_as_longlong(nrm) > __double_as_longlong(lim) ? 1 : 0;
                  if (!take) inv = 0.0;
                  // much of it went with the projection or with the block's other columns: what is
                  // left carries their rounding, the second round takes it out
                  else if (rho < 0.25 * S.ref[s]) S.refine = 1;
                }
              }
              S.take[s] = take;
              S.inv = inv;
              if (take >= 0) S.R[s][s] = make_double2(take ? nrm : 0.0, 0.0);
              S.M[s][s] = make_double2(take > 0 ? inv : 0.0, 0.0);
              S.u[s & 1][s] = make_double2(inv, 0.0);
            }
            asm volatile("bar.sync 1, 160;" ::: "memory");
            const int take = S.take[s];
            if (take < 0) break;
            if (take > 0) {
              const double inv = S.inv;
              ++taken;
              if (a == s && b > s) {         // row s of R
                g = make_double2(g.x * inv, g.y * inv);
                S.R[s][b] = g;
                S.y[b] = g;
                S.u[s & 1][b] = make_double2(g.x, -g.y);
                g = make_double2(0.0, 0.0);
              } else if (b == s && a < s) {  // column s of the inverse
                g = make_double2(g.x * inv, g.y * inv);
                S.M[a][s] = g;
                S.u[s & 1][a] = g;
              }
              asm volatile("bar.sync 1, 160;" ::: "memory");
              if (b > s) {
                const cplx u = S.u[s & 1][a], y = S.y[b];
                g.x = fma(-u.x, y.x, g.x);
                g.x = fma(u.y, y.y, g.x);
                g.y = fma(-u.x, y.y, g.y);
                g.y = fma(-u.y, y.x, g.y);
              }
            } else {
              if (a == s && b > s) {
                S.R[s][b] = make_double2(0.0, 0.0);
                g = make_double2(0.0, 0.0);
              } else if (b == s && a < s) {
                S.M[a][s] = make_double2(0.0, 0.0);
              }
              asm volatile("bar.sync 1, 160;" ::: "memory");
            }
          }
          if (tid == 0) S.done = s;
        }
        __syncthreads();
      } else {
        // ---- second round: the columns are orthonormal up to E = V^H V - 1, |E| < 1e-6 (KEEP); the
        // factor 1 + U and its inverse 1 - W, W = U - U^2, to third order (the second-order terms,
        // below 1e-12, in FP32)
        const int a = tid >> 4, b = tid & 15;
        const bool on = a <= b && b < S.done && S.take[a] > 0 && S.take[b] > 0;
        float2* F = reinterpret_cast<float2*>(own);      // U to first order, U, then W
        cplx g = make_double2(0.0, 0.0);
        if (on) {
          g = S.G[a][b];
          if (a == b) g = make_double2(0.5 * (g.x - 1.0), 0.0);
        }
        F[tid] = make_float2((float)g.x, (float)g.y);
        __syncthreads();
        if (on) {
          float2 q = make_float2(0.0f, 0.0f);  // (U^H U)_ab
          for (int k = 0; k <= a; ++k) {
            const float2 x = F[k * QB + a], y = F[k * QB + b];
            q.x = fmaf(x.x, y.x, fmaf(x.y, y.y, q.x));
            q.y = fmaf(x.x, y.y, fmaf(-x.y, y.x, q.y));
          }
          if (a == b) q = make_float2(0.5f * q.x, 0.0f);
          g = make_double2(g.x - q.x, g.y - q.y);
        }
        S.G[a][b] = g;                         // U
        F[256 + tid] = make_float2((float)g.x, (float)g.y);
        __syncthreads();
        cplx w = g;
        if (on) {
          float2 q = make_float2(0.0f, 0.0f);  // (U^2)_ab
          for (int k = a; k <= b; ++k) {
            const float2 x = F[256 + a * QB + k], y = F[256 + k * QB + b];
            q.x = fmaf(x.x, y.x, fmaf(-x.y, y.y, q.x));
            q.y = fmaf(x.x, y.y, fmaf(x.y, y.x, q.y));
          }
          w = make_double2(w.x - q.x, w.y - q.y);
        }
        S.M[a][b] = make_double2((on && a == b ? 1.0 : 0.0) - w.x, -w.y);
        F[512 + tid] = make_float2((float)w.x, (float)w.y);
        small = __syncthreads_and(fabs(w.x) < SMALL && fabs(w.y) < SMALL) != 0;
      }
      const int done = S.done;
      // ---- the new columns q_t = sum_{s <= t} v_s M_st: warp w takes columns w and 15 - w, the
      // lanes the rows (MAXR / 32 rows each).  A second round that changes little: v_t - sum v_s W_st,
      // the sum in FP32
      if (small) {
        const float2* W = reinterpret_cast<const float2*>(own) + 512;
        float2* F = reinterpret_cast<float2*>(ring);       // V, [QB][MAXR + 1]
        for (int e = tid; e < QB * nr; e += QT_THREADS) {
          const int t = e / nr, r = e - t * nr;
          const cplx v = V[t * LDV + r];
          F[t * LDV + r] = make_float2((float)v.x, (float)v.y);
        }
        __syncthreads();
        for (int u = 0; u < 2; ++u) {
          const int t = u == 0 ? warp : QB - 1 - warp;
          if (t >= done || S.take[t] <= 0) continue;
          for (int r = lane; r < nr; r += 32) {
            float2 q = make_float2(0.0f, 0.0f);
            for (int s = 0; s <= t; ++s) {
              const float2 v = F[s * LDV + r], c = W[s * QB + t];
              q.x = fmaf(v.x, c.x, fmaf(-v.y, c.y, q.x));
              q.y = fmaf(v.x, c.y, fmaf(v.y, c.x, q.y));
            }
            cplx& v = V[t * LDV + r];
            v = make_double2(v.x - q.x, v.y - q.y);
          }
        }
        __syncthreads();
      } else {
        cplx q[2][MAXR / 32];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int t = u == 0 ? warp : QB - 1 - warp;
          const bool on = t < done && S.take[t] > 0;
#pragma unroll
          for (int k = 0; k < MAXR / 32; ++k) {
            q[u][k] = make_double2(0.0, 0.0);
            const int r = k * 32 + lane;
            if (on && k * 32 < nr) {
              double x = 0.0, y = 0.0, x2 = 0.0, y2b = 0.0;
              for (int s = 0; s <= t; ++s) {
                if (S.take[s] <= 0) continue;      // (a skipped vector may hold Inf or NaN)
                const cplx v = V[s * LDV + min(r, nr - 1)], c = S.M[s][t];
                x = fma(v.x, c.x, x);
                x2 = fma(-v.y, c.y, x2);
                y = fma(v.x, c.y, y);
                y2b = fma(v.y, c.x, y2b);
              }
              q[u][k] = make_double2(x + x2, y + y2b);
            }
          }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int t = u == 0 ? warp : QB - 1 - warp;
          if (t < done && S.take[t] > 0)
#pragma unroll
            for (int k = 0; k < MAXR / 32; ++k) {
              const int r = k * 32 + lane;
              if (r < nr) V[t * LDV + r] = q[u][k];
            }
        }
        __syncthreads();
      }
      if (refine || !S.refine) break;
      refine = true;
      // skipped and put-off columns take no part in the second round
      for (int e = tid; e < QB * nr; e += QT_THREADS) {
        const int t = e / nr, r = e % nr;
        if (t >= S.done || S.take[t] <= 0) V[t * LDV + r] = make_double2(0.0, 0.0);
      }
      __syncthreads();
    }
    if (!alive) break;
    // rows of the accepted vectors in R's new columns: the sum of the passes' coefficients (the CTAs
    // share the rows where they can all read the sums, else CTA 0 kept them)
    auto write_r = [&](int cols) {
      if (private_r && blockIdx.x != 0) return;
      const int first = private_r ? 0 : blockIdx.x, G = private_r ? 1 : gridDim.x;
      for (int e = first * QT_THREADS + tid; e < na * QB; e += G * QT_THREADS) {
        const int i = e >> 4, t = e & 15;
        cplx r = make_double2(0.0, 0.0);
        for (int q = 0; q < npass; ++q) {
          const cplx h = __ldcg(A.fin + (long long)q * A.PS + e);
          r = make_double2(r.x + h.x, r.y + h.y);
        }
        if (refine)
          for (int s = 0; s <= t; ++s)
            if (S.take[s] > 0) {
              const cplx h = __ldcg(A.fin + (long long)npass * A.PS + i * QB + s), f = S.R[s][t];
              r.x = fma(h.x, f.x, fma(-h.y, f.y, r.x));
              r.y = fma(h.x, f.y, fma(h.y, f.x, r.y));
            }
        if (t < cols) A.R[(long long)S.idx[i] * n + j0 + t] = r;
      }
    };
    if (all_dropped) {
      if (main_phase) {
        write_r(bsz);
        j0 += bsz;
      } else {
        cand += bsz;
      }
    } else {
      const int done = S.done;
      // ---- bookkeeping: S.em[t] = position of column t among the accepted vectors, -1 if none
      if (tid == 0) {
        int a = na, pos = open;
        for (int t = 0; t < QB; ++t) S.em[t] = -1;
        for (int t = 0; t < done; ++t) {
          if (S.take[t] <= 0) continue;
          int col;
          if (main_phase) {
            col = j0 + t;
          } else {
            while (S.acc[pos]) ++pos;
            col = pos;
            if (A.src_out && blockIdx.x == 0) A.src_out[col] = (int)(cand + t);
          }
          S.acc[col] = 1;
          S.idx[a] = (short)col;
          S.src[a - na] = t;
          S.em[t] = a++;
        }
        S.any = a;
        S.last = pos;
      }
      __syncthreads();
      const int na1 = S.any;
      open = S.last;
      // digits of the new columns are wanted while a column or a position is left
      const bool more = na1 < n;
      // form 2 is written two bytes at a time: a k step is cleared when its first column comes
      // (its unused columns must be zero)
      if (more)
        for (int k = (na + 15) / 16; k * 16 < na1; ++k)
          for (int e = tid; e < s2 / 16; e += QT_THREADS)
            reinterpret_cast<uint4*>(d2 + k * s2)[e] = make_uint4(0u, 0u, 0u, 0u);
      // ---- Q in FP64, and its digits in both operand forms
      for (int r = tid; r < nr; r += QT_THREADS) S.rnew[r] = 0;
      if (tid < QB) S.ev[tid] = 0;
      __syncthreads();
      for (int e = tid; e < QB * nr; e += QT_THREADS) {
        const int t = e % QB, r = e / QB;
        const int a = S.em[t];
        if (a >= 0) {
          const cplx v = V[t * LDV + r];
          A.Q[(long long)(r0 + r) * n + S.idx[a]] = v;
          const int ex = max(bexp(v.x), bexp(v.y));
          atomicMax(&S.rnew[r], ex);
          atomicMax(&S.ev[t], ex);
        }
      }
      __syncthreads();
      {
        const int t = tid & 15, g = tid >> 4;
        const int a = S.em[t];
        if (more && a >= 0) {
          const int em = max(S.ev[t], 1);
          if (g == 0) S.ec[a] = em - 1022;
          for (int k = g; k < 8 * rsteps; k += 16) {
            const int part = k & 1, q = k >> 1;
            qt_store(V + t * LDV + q * 4, 1, min(4, nr - q * 4), part, em, em == 0x7ff,
                     d1 + (q >> 2) * s1 + (a >> 3) * GROUP + part * (GROUP / 2) +
                         ((q >> 1) & 1) * 128 + (a & 7) * 16 + (q & 1) * 8);
          }
        }
        for (int r = g; more && r < nr; r += 16) {
          // this row's scale; outgrown: all its columns again (the 16 threads of a row agree)
          int er = S.er[r];
          const int en = S.rnew[r] - 1022;
          const bool grown = S.rnew[r] > 0 && en > er;
          if (grown) er = en + 1;
          const int first = grown ? 0 : na;
          for (int c = first + t; c < na1; c += 16) {
            const cplx v = c < na ? A.Q[(long long)(r0 + r) * n + S.idx[c]]
                                  : V[S.src[c - na] * LDV + r];
            unsigned char* dst = d2 + (c >> 4) * s2 + (r >> 3) * GROUP + ((c >> 3) & 1) * 128 +
                                 (r & 7) * 16 + (c & 7) * 2;
            const unsigned long long wr = digits_of(v.x, er + 1022, false, false);
            const unsigned long long wi = digits_of(v.y, er + 1022, false, false);
#pragma unroll
            for (int l = 0; l < ND; ++l) {
              const uint32_t d = digit_pair(wr, wi, l);
              *reinterpret_cast<unsigned short*>(dst + l * 256) = (unsigned short)d;
              *reinterpret_cast<unsigned short*>(dst + GROUP / 2 + l * 256) =
                  (unsigned short)(d >> 16);
            }
          }
          __syncwarp(0xffffu << (lane & 16));      // the row's 16 threads (the other half may be done)
          if (t == 0) S.er[r] = er;
        }
      }
      // the block's own part of R, a share of it to every CTA
      if (main_phase)
        for (int e = blockIdx.x * 32 + (tid & 31) + (tid >> 5) * 32 * gridDim.x; e < QB * QB;
             e += QT_THREADS * gridDim.x) {
          const int s = e >> 4, t = e & 15;
          if (s > t || t >= done) continue;
          cplx r = S.R[s][t];
          if (refine && S.take[s] > 0)       // (1 + U) R
            for (int k = s; k <= t; ++k)
              if (S.take[k] > 0) {
                const cplx x = S.G[s][k], y = S.R[k][t];
                r.x = fma(x.x, y.x, fma(-x.y, y.y, r.x));
                r.y = fma(x.x, y.y, fma(x.y, y.x, r.y));
              }
          A.R[(long long)(j0 + s) * n + j0 + t] = r;
        }
      if (main_phase) write_r(done);
      na = na1;
      if (main_phase) j0 += done;
      else cand += done;
      asm volatile("fence.proxy.async;" ::: "memory");
      __syncthreads();
    }
    if (main_phase && j0 >= n) {
      main_phase = false;
      if (blockIdx.x == 0)
        for (int i = tid; i < n; i += QT_THREADS) A.acc_out[i] = (unsigned char)S.acc[i];
    }
    __syncthreads();
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS));
  }
}

namespace {
struct QtPlan {
  int G, rows;
  long long dig_cta;
};
// about 32 rows per CTA, at most MAXR
bool qt_plan(int m, int n, int cap, QtPlan& p) {
  if (n > MAXN || n < MINN || cap < 1) return false;
  long long g = ((long long)m + 31) / 32;
  if (g > cap) g = cap;
  p.rows = (int)((m + g - 1) / g);
  if (p.rows > MAXR) return false;
  p.G = (m + p.rows - 1) / p.rows;
  p.dig_cta = ((long long)((p.rows + 15) / 16) * ((n + 7) / 8) +
               (long long)((n + 15) / 16) * ((p.rows + 7) / 8)) * GROUP;
  return true;
}
constexpr size_t QT_SMEM = 2 * (size_t)RING + BDIG + sizeof(cplx) * QB * (MAXR + 1) + 128;
}  // namespace

size_t gauge_qr_tensor_bytes(int m, int n, int sms) {
  if (n > MAXN || n < MINN || m > (long long)MAXR * sms) return 0;
  const long long G = (m + 31) / 32 < sms ? (m + 31) / 32 : sms;
  return (size_t)((m + 16 * G) * ((n + 7) / 8) / 16 + (m + 8 * G) * (long long)((n + 15) / 16) / 8 +
                  32) * GROUP;
}

cudaError_t gauge_qr_tensor(int m, int n, QrRef Y, int p, QrRef E, cplx* Q, cplx* R, cplx* scratch,
                            long long scratch_len, unsigned char* acc, const QrScratch& W,
                            int* status, cudaStream_t s, int gcap, double rank_tol, int* src,
                            bool* taken) {
  *taken = false;
  int cap = W.gmax;
  if (gcap > 0 && gcap < cap) cap = gcap;
  QtPlan pl;
  if (!W.dig || !qt_plan(m, n, cap, pl)) return cudaSuccess;
  const long long PS = (long long)n * QB + QB + QB * QB;
  if ((size_t)pl.G * pl.dig_cta > W.dig_bytes || (2 * (long long)pl.G + PASSES + 1) * PS > scratch_len) return cudaSuccess;
  static OncePerDevice smem;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = smem.run(dev, cudaErrorInvalidDevice, [] {
      return cudaFuncSetAttribute(gauge_qr_tensor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)QT_SMEM);
    });
  if (e != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(W.bar, 0, 2 * sizeof(unsigned), s)) != cudaSuccess) return e;
  QtArgs a{};
  a.m = m; a.n = n; a.p = p;
  a.Y = Y; a.E = p > 0 ? E : Y;
  a.Q = Q; a.R = R;
  a.part = scratch;
  a.fin = scratch + 2 * (long long)pl.G * PS;      // (PASSES + 1) * PS
  a.PS = (int)PS;
  a.dig = W.dig;
  a.dig_cta = pl.dig_cta;
  a.rows = pl.rows;
  a.bar = W.bar;
  a.status = status;
  a.wait = W.wait > 0 ? W.wait : kBarrierWaitCycles;
  a.acc_out = acc;
  a.src_out = src;
  a.rank_tol = rank_tol;
  a.complete_tol = 1e-2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pl.G);
  cfg.blockDim = dim3(QT_THREADS);
  cfg.dynamicSmemBytes = QT_SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch();
  *taken = true;
  return cudaLaunchKernelEx(&cfg, gauge_qr_tensor_kernel, a);
}

}  // namespace tdmrg
