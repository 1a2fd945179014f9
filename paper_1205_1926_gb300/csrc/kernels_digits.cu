// FP64 products with the dense K^+ of a box shape on the tensor cores.
//
// The FP64 pipe of this part issues two FMAs per SM and clock (1.06 TFLOP/s for the whole
// device), so the banded sweeps of the subdomains that share their shape's elastic factor
// are bound by it: 1600 us a pass over 512 boxes of 8^3 elements (2187 dofs, 1158 at the
// boundary), 4750 us over 1728.  Their K^+ apply is a contraction, Y = X K^+ with one row of X
// per subdomain, and BF16 tensor cores run 1800 times faster.  Measured with these kernels: 135
// us for the pass on all dofs of the 512 boxes (split 15, GEMM 102, scatter 18) and 75 us on the
// boundary dofs; the GEMM's 141 GFLOP of digit products run at 1.4 PFLOP/s, bound by the MMAs
// (95 us without copies and without draining the accumulators, 58 us without the MMAs).
//
// FP64 accuracy comes from an error-free splitting of both operands into integer digits (the
// scheme of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its applications",
// Numer. Algorithms 59, 2012): a row of X, scaled by the power of two above its largest entry, is
//     x = 2^(e-7) sum_i d_i 2^(-8 i),  i = 0..6,  integers |d_i| <= 128,
// i.e. 55 bits below 2^e (round to nearest), and likewise every row of K^+.  A digit
// times 2^(-8 i) is exact in BF16.  The products d_i d'_j with i + j = g have weight
// 2^(-8 g); the 28 pairs with i + j <= 6 are formed, the dropped ones lie below 2^-55 of
// the leading one.  Sums over K of the groups g = 0..4 are integers times 2^(-8 g): at
// most 5 x 192 x 2^14 < 2^24 over a chunk of 192 of K, so the FP32 accumulators in TMEM
// hold them exactly; after each chunk they are added, as integers, into a 64-bit sum.
// The groups 5 and 6 carry at most 2^-40 of the leading weight, so they are accumulated in
// FP32 over the whole K range.  The total is an integer in units of 2^-37 and is converted to
// FP64 once.  Against extended precision the product of a 2187-dof box is off by 2.2e-15 (norm),
// a sequential FP64 sum by 2.4e-15 (with four exact groups instead of five: 3.9e-14).
//
// Non-finite entries make the row's scale NaN, so that the whole result of that subdomain
// is NaN, as it is after the banded sweeps.
//
// Tiles: 128 rows of X (subdomains) x 64 rows of K^+ (output dofs) per CTA.  The digits of a
// stage's K^+ tile are stacked as 7 x 64 rows, so the products of digit i of X with the digits
// j = 0..6 - i are one run of 64 (7 - i) columns of accumulators starting at group i: ten MMAs
// of up to 256 columns per 16 columns of K instead of 28 of 64 (a narrow MMA takes about 64
// cycles whatever its width: 28 MMAs of 80, 64, 48 or 32 columns each took 126 us a wave for
// the 2187-dof boxes).  Stages of 16 columns of K, 43 KB, five in flight.  The seven
// accumulators fill 448 of the 512 TMEM columns.
#include <cuda_bf16.h>

#include "async_common.cuh"
#include "dev.h"
#include "dual_common.cuh"

namespace tfeti {

namespace {

constexpr int kM = kDgM, kN = kDgN, kK = 16;     // CTA tile, K columns of a stage (one MMA step)
constexpr int kS = 7;                            // digits per value
constexpr int kExact = 5;                        // digit groups with exact accumulators
constexpr int kChunk = 12;                       // stages per chunk of exact accumulation (K = 192)
constexpr int kUnit = 37;                        // the integer results are in units of 2^-kUnit
constexpr int kStages = 5;
constexpr uint32_t kABytes = kM * kK * 2;        // one digit's tile of X
constexpr uint32_t kBBytes = kS * kN * kK * 2;   // a stage's tile of K^+, all digits
constexpr uint32_t kStageBytes = kS * kABytes + kBBytes;
constexpr uint32_t kTmem = 512;                  // columns: kS x kN rounded up to a power of two
constexpr int kEpiWarps = 8;
constexpr int kGemmThreads = 32 * (kEpiWarps + 2);
// instruction descriptor of kind::f16 without N: D FP32, A and B BF16, K-major, M
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kM >> 4) << 24);
constexpr size_t kGemmSmem = kStages * kStageBytes + (2 * kStages + 3) * sizeof(uint64_t) + 2 * sizeof(uint32_t);
static_assert(kS * kN <= (int)kTmem, "accumulators exceed TMEM");
static_assert(kExact * kChunk * kK * (1 << 14) <= (1 << 24), "a chunk's sums exceed FP32 integers");

// Element offset of (row, col8 x 8) inside a tile of `groups` x 8 rows and kK columns: core
// matrices of 8 rows x 16 bytes, K-major (no swizzle).
__device__ __forceinline__ int tile_off8(int row, int col8, int groups) {
  return (col8 * groups + (row >> 3)) * 64 + (row & 7) * 8;
}

// The digits of a value: t = round(v 2^(55 - e)) in balanced radix 256, from the bits of v
// (integer instructions only; the FP64 pipe is the scarce unit).  emax: the biased exponent
// field of the row's largest entry (at least 1), 2^e = 2^(emax - 1022).
__device__ __forceinline__ void split_digits(double v, int emax, int (&d)[kS]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  int ex = (int)(b >> 52) & 0x7ff;
  unsigned long long mant = b & 0xfffffffffffffULL;
  if (ex) mant |= 1ULL << 52;
  else ex = 1;
  const int sh = emax - ex;   // v = mant 2^(emax - 1075 - sh), t = mant 2^(2 - sh)
  unsigned long long t = 0;
  if (sh <= 2) t = mant << (2 - sh);
  else if (sh <= 56) t = (mant + (1ULL << (sh - 3))) >> (sh - 2);
  long long s = (b >> 63) ? -(long long)t : (long long)t;
#pragma unroll
  for (int i = kS - 1; i > 0; --i) {
    d[i] = (int)(signed char)(s & 0xff);
    s = (s - d[i]) >> 8;
  }
  d[0] = (int)s;
}

// BF16 bits of d 2^(-8 i) for |d| <= 128 (exact).
__device__ __forceinline__ uint32_t digit_bf16(int d, int i) {
  const float f = (float)d * __uint_as_float((uint32_t)(127 - 8 * i) << 23);
  return __float_as_uint(f) >> 16;
}

// Writes the digits of 8 consecutive columns (16 bytes per digit) of a row.
__device__ __forceinline__ void store_digits8(const double* v, int emax, uint4* dst, long long digit_stride16) {
  uint32_t w[kS][4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    int d0[kS], d1[kS];
    split_digits(v[2 * h], emax, d0);
    split_digits(v[2 * h + 1], emax, d1);
#pragma unroll
    for (int i = 0; i < kS; ++i) w[i][h] = digit_bf16(d0[i], i) | (digit_bf16(d1[i], i) << 16);
  }
#pragma unroll
  for (int i = 0; i < kS; ++i) dst[i * digit_stride16] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// 2^(e - 7) with 2^e the power of two above a row's largest entry, emax its biased exponent
// field (the integer product in units of 2^-kUnit times the two rows' scales is the result);
// NaN for a non-finite row.
__device__ __forceinline__ double row_scale(int emax) {
  if (emax >= 0x7ff) return __longlong_as_double(0x7ff8000000000000LL);
  return scalbn(1.0, emax - 1022 - 7);
}

__device__ __forceinline__ int exp_field(double v) {
  return (int)((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ff;
}

// Largest exponent field over the block (at least 1), known to all threads.
__device__ __forceinline__ int block_max_exp(int e) {
  __shared__ int s_max;
  if (threadIdx.x == 0) s_max = 1;
  __syncthreads();
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_max, e);
  __syncthreads();
  return s_max;
}

// Digit tiles of the rows of X, one CTA per row: row blockIdx.x is subdomain list[row] of
// block blk_of[row].  Boundary form (full = 0): X = (B^T lam) at the shape's boundary dofs, 0
// off the interface; full form: X = (src or 0) + sign (B^T lam) on all local dofs, 0 at the
// fixing dofs (K^+ has zero rows there; their values must not set the scale).
__global__ void __launch_bounds__(256) k_dg_split_x(DevMesh M, const DgBlock* __restrict__ blocks,
                                                    const DgRow* __restrict__ rows, int full,
                                                    const double* __restrict__ src, const double* __restrict__ lam,
                                                    double sign, uint4* __restrict__ A, double* __restrict__ sA) {
  extern __shared__ double xs[];
  const DgRow row = rows[blockIdx.x];
  const DgBlock& blk = blocks[row.blk];
  const SubDev& S = M.subs[row.sub];
  const int n = full ? blk.n : blk.n_bd, nk = full ? blk.nk : blk.nk_bd, kcols = nk * kK;
  const int tid = threadIdx.x, nt = blockDim.x;
  constexpr int U = 4;   // copy slots per thread with their B^T gathers in flight together
  if (full) {
    for (int i = tid; i < kcols; i += nt) xs[i] = (src && i < n) ? src[S.dof_off + i] : 0.0;
    __syncthreads();
    if (lam)
      for (int s0 = tid; s0 < S.n_copy; s0 += U * nt) {
        long long sl[U];
        double v[U];
#pragma unroll
        for (int k = 0; k < U; ++k) sl[k] = s0 + k * nt < S.n_copy ? S.copy_off + s0 + k * nt : -1;
        bt_at_slots<U>(M, lam, sl, v);
#pragma unroll
        for (int k = 0; k < U; ++k)
          if (sl[k] >= 0) xs[__ldg(M.slot_ldof + sl[k])] += sign * v[k];
      }
    __syncthreads();
    if (tid < 6) xs[S.fix[tid]] = 0.0;
  } else {
    int fix[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) fix[q] = S.fix[q];
    for (int j0 = tid; j0 < kcols; j0 += U * nt) {
      long long sl[U];
      double v[U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int j = j0 + k * nt;
        const int b = j < n ? __ldg(M.sub_b2s + S.b2s_off + j / 3) : -1;
        const int ld = j < n ? 3 * __ldg(M.shape_bln + S.bnd_off + j / 3) + j % 3 : -1;
        bool fixed = false;   // fixing dofs are boundary dofs; their rows and columns of S are zero
#pragma unroll
        for (int q = 0; q < 6; ++q) fixed |= ld == fix[q];
        sl[k] = b >= 0 && !fixed ? (long long)b + j % 3 : -1;
      }
      bt_at_slots<U>(M, lam, sl, v);
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (j0 + k * nt < kcols) xs[j0 + k * nt] = sl[k] >= 0 ? v[k] : 0.0;
    }
  }
  __syncthreads();
  int e = 0;
  for (int i = tid; i < n; i += nt) e = max(e, exp_field(xs[i]));
  const int emax = block_max_exp(e);
  if (tid == 0) sA[blockIdx.x] = row_scale(emax);
  const int mt = row.local / kM, r = row.local % kM;
  uint4* base = A + ((full ? blk.a_off : blk.a_off_bd) + (long long)mt * nk * kS * (kM * kK)) / 8;
  for (int c = tid; c < nk * (kK / 8); c += nt) {
    const int ks = c / (kK / 8), c8 = c % (kK / 8);
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = xs[ks * kK + c8 * 8 + k];
    store_digits8(v, emax, base + ((long long)ks * kS * (kM * kK) + tile_off8(r, c8, kM / 8)) / 8, kM * kK / 8);
  }
}

// Digit tiles of the rows of K^+ (set-up), one CTA per padded row: row i of the full form is
// column i of the dense kinv (symmetric), of the boundary form its boundary dofs.
__global__ void __launch_bounds__(256) k_dg_split_k(DevMesh M, long long bnd_off, int n, int n_bd, int full,
                                                    const double* __restrict__ kinv, uint4* __restrict__ B,
                                                    double* __restrict__ sB) {
  const int i = blockIdx.x, rows = full ? n : n_bd, nk = (rows + kK - 1) / kK;
  const int tid = threadIdx.x, nt = blockDim.x;
  auto dof = [&](int j) { return full ? j : 3 * M.shape_bln[bnd_off + j / 3] + j % 3; };
  const double* col = i < rows ? kinv + (long long)dof(i) * n : nullptr;
  int e = 0;
  if (col)
    for (int j = tid; j < rows; j += nt) e = max(e, exp_field(col[dof(j)]));
  const int emax = block_max_exp(e);
  if (tid == 0) sB[i] = row_scale(emax);
  const int ntile = i / kN, r = i % kN;
  uint4* base = B + (long long)ntile * nk * kS * (kN * kK) / 8;
  for (int c = tid; c < nk * (kK / 8); c += nt) {
    const int ks = c / (kK / 8), c8 = c % (kK / 8);
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int j = ks * kK + c8 * 8 + k;
      v[k] = (col && j < rows) ? col[dof(j)] : 0.0;
    }
    store_digits8(v, emax, base + ((long long)ks * kS * (kN * kK) + tile_off8(r, c8, kS * kN / 8)) / 8, kN);
  }
}

// ---- tensor-core primitives -------------------------------------------------
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, int n, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(kIdesc | ((uint32_t)(n >> 3) << 17)), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

__device__ __forceinline__ void mbar_init_n(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive accumulator columns of this thread's TMEM lane (issued; wait with tmem_wait).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The MMAs of one stage over the digit groups [g0, g1): digit i of X times the digits
// j = max(0, g0 - i) .. g1 - 1 - i of K^+, i.e. the accumulator columns from group i + j on, in
// pieces of at most 256 columns.  first: the groups' accumulators start from zero (digit 0 of X
// reaches all of them).
template <int g0, int g1>
__device__ __forceinline__ void issue_groups(uint32_t tmem, uint32_t sa, uint32_t sb, bool first) {
#pragma unroll
  for (int i = 0; i < g1; ++i) {
    const int jlo = g0 > i ? g0 - i : 0, cols = (g1 - i - jlo) * kN;
    const int pieces = cols > 256 ? 2 : 1, w = cols / pieces;
    const uint64_t da = smem_desc(sa + i * kABytes, (kM / 8) * 128, 128);
#pragma unroll
    for (int h = 0; h < pieces; ++h) {
      const uint64_t db = smem_desc(sb + (jlo * (kN / 8) + h * (w / 8)) * 128, (kS * kN / 8) * 128, 128);
      mma(tmem + (uint32_t)((i + jlo) * kN + h * w), da, db, w, (first && i == 0) ? 0u : 1u);
    }
  }
}

// One 128 x 64 tile of Y = X K^+ over the stages [ks0, ks1) of its K split, as 64-bit
// integers in units of 2^-kUnit (before the rows' scales), to out + the CTA's offset (row-major,
// pitch ld).  Warp 8: streams the stages; warp 9: issues the MMAs; warps 0..7 read the exact
// accumulators after every chunk (warp w: TMEM lanes 32 (w % 4) .. + 31, columns 32 (w / 4)
// .. + 31) while the MMAs of the low groups go on: the last two stages of a chunk issue their
// exact groups first, the first two of the next chunk their low groups.
__global__ void __launch_bounds__(kGemmThreads, 1) k_dg_gemm(const DgBlock* __restrict__ blocks,
                                                             const DgCta* __restrict__ ctas, int full,
                                                             const unsigned char* __restrict__ A,
                                                             const unsigned char* __restrict__ B,
                                                             long long* __restrict__ out, int* err,
                                                             long long limit) {
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* empty_bar = full_bar + kStages;
  uint64_t* exact_bar = empty_bar + kStages;   // the chunk's exact groups are complete
  uint64_t* drained_bar = exact_bar + 1;       // the epilogue warps have read them
  uint64_t* done_bar = drained_bar + 1;        // all MMAs complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done_bar + 1);
  int* s_fail = reinterpret_cast<int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const DgCta cta = ctas[blockIdx.x];
  const DgBlock& blk = blocks[cta.blk];
  const int nk = full ? blk.nk : blk.nk_bd;
  const int n_ks = cta.ks1 - cta.ks0;
  const int n_chunk = (n_ks + kChunk - 1) / kChunk;
  auto wait = [limit](uint64_t* bar, uint32_t parity) { return limit != 0 && mbar_wait(bar, parity, limit); };

  if (threadIdx.x == 0) {
    for (int q = 0; q < kStages; ++q) {
      mbar_init(&full_bar[q]);
      mbar_init(&empty_bar[q]);
    }
    mbar_init(exact_bar);
    mbar_init_n(drained_bar, kEpiWarps);
    mbar_init(done_bar);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpiWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == kEpiWarps) {
    if (lane == 0) {
      const unsigned char* a = A + 2 * (full ? blk.a_off : blk.a_off_bd) + ((long long)cta.mt * nk + cta.ks0) * kS * kABytes;
      const unsigned char* b = B + 2 * (full ? blk.b_off : blk.b_off_bd) + ((long long)cta.nt * nk + cta.ks0) * kBBytes;
      int issued = 0;
      for (int j = 0; j < n_ks; ++j) {
        const int st = j % kStages, u = j / kStages;
        if (u > 0 && !wait(&empty_bar[st], (uint32_t)((u - 1) & 1))) {
          atomicOr(s_fail, 1);
          break;
        }
        unsigned char* base = smem + st * kStageBytes;
        mbar_expect_tx(&full_bar[st], kStageBytes);
        bulk_copy_tx(base, a + (long long)j * kS * kABytes, kS * kABytes, &full_bar[st]);
        bulk_copy_tx(base + kS * kABytes, b + (long long)j * kBBytes, kBBytes, &full_bar[st]);
        ++issued;
      }
      // every issued copy has landed before the CTA can leave (immediate on the normal path)
      for (int j = issued - 1; j >= 0 && j >= issued - kStages; --j)
        mbar_wait(&full_bar[j % kStages], (uint32_t)((j / kStages) & 1));
    }
  } else if (warp == kEpiWarps + 1) {
    if (lane == 0) {
      bool ok = true;
      auto wait_full = [&](int j) {
        if (!wait(&full_bar[j % kStages], (uint32_t)((j / kStages) & 1))) ok = false;
      };
      auto sa_of = [&](int j) { return smem_addr(smem + (j % kStages) * kStageBytes); };
      for (int j = 0; j < n_ks && ok; j += 2) {
        const int m = min(2, n_ks - j), c = j / kChunk;
        const bool first = j % kChunk == 0, last = (j + 2) % kChunk == 0 || j + 2 >= n_ks;
        if (!first && !last) {
          for (int s = j; s < j + m && ok; ++s) {
            wait_full(s);
            fence_after();
            issue_groups<0, kS>(tmem, sa_of(s), sa_of(s) + kS * kABytes, false);
            mma_commit(&empty_bar[s % kStages]);
          }
          continue;
        }
        for (int s = j; s < j + m && ok; ++s) wait_full(s);
        if (!ok) break;
        fence_after();
        const bool low_first = first && c > 0;
        if (low_first) {
          for (int s = j; s < j + m; ++s) issue_groups<kExact, kS>(tmem, sa_of(s), sa_of(s) + kS * kABytes, false);
          if (!wait(drained_bar, (uint32_t)((c - 1) & 1))) {
            ok = false;
            break;
          }
          fence_after();
        }
        for (int s = j; s < j + m; ++s)
          issue_groups<0, kExact>(tmem, sa_of(s), sa_of(s) + kS * kABytes, first && s == j);
        if (last) mma_commit(exact_bar);
        if (!low_first)
          for (int s = j; s < j + m; ++s) issue_groups<kExact, kS>(tmem, sa_of(s), sa_of(s) + kS * kABytes, s == 0);
        for (int s = j; s < j + m; ++s) mma_commit(&empty_bar[s % kStages]);
      }
      if (!ok) atomicOr(s_fail, 1);
      mma_commit(done_bar);
    }
  } else {
    const int quad = warp & 3, cbeg = (warp >> 2) * (kN / 2);
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
    long long acc[kN / 2];
#pragma unroll
    for (int k = 0; k < kN / 2; ++k) acc[k] = 0;
    bool ok = true;
    for (int c = 0; c < n_chunk && ok; ++c) {
      ok = wait(exact_bar, (uint32_t)(c & 1));
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      fence_after();
#pragma unroll
      for (int c0 = 0; c0 < kN / 2; c0 += 16) {
        uint32_t v[kExact][16];
#pragma unroll
        for (int g = 0; g < kExact; ++g) tmem_ld16(lane_base + (uint32_t)(g * kN + cbeg + c0), v[g]);
        tmem_wait();
#pragma unroll
        for (int k = 0; k < 16; ++k)
#pragma unroll
          for (int g = 0; g < kExact; ++g) {
            // an integer of at most 2^24 times 2^(-8 g)
            const int t = __float2int_rn(__uint_as_float(v[g][k]) * (float)(1LL << (8 * g)));
            acc[c0 + k] += (long long)t * (1LL << (8 * (kExact - 1 - g)));
          }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(drained_bar);
    }
    // also where a wait gave up: no MMA may be in flight when TMEM is freed and the CTA ends
    if (!mbar_wait(done_bar, 0u)) ok = false;
    ok = __all_sync(0xffffffffu, ok);
    if (!ok && lane == 0) atomicOr(s_fail, 1);
    if (ok) {
      fence_after();
      const long long ld = cta.ld;
      long long* dst = out + cta.out_off + (long long)(quad * 32 + lane) * ld + cbeg;
#pragma unroll
      for (int c0 = 0; c0 < kN / 2; c0 += 16) {
        uint32_t v[16], w6[16];
        tmem_ld16(lane_base + (uint32_t)(kExact * kN + cbeg + c0), v);
        tmem_ld16(lane_base + (uint32_t)((kExact + 1) * kN + cbeg + c0), w6);
        tmem_wait();
#pragma unroll
        for (int k = 0; k < 16; k += 2) {
          // units of 2^-kUnit: the exact sum is in units of 2^(-8 (kExact - 1))
          constexpr long long up = 1LL << (kUnit - 8 * (kExact - 1));
          constexpr float lu = (float)(1LL << kUnit);
          longlong2 w;
          w.x = acc[c0 + k] * up + __float2ll_rn((__uint_as_float(v[k]) + __uint_as_float(w6[k])) * lu);
          w.y = acc[c0 + k + 1] * up + __float2ll_rn((__uint_as_float(v[k + 1]) + __uint_as_float(w6[k + 1])) * lu);
          *reinterpret_cast<longlong2*>(dst + c0 + k) = w;
        }
      }
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *s_fail) atomicOr(err, kErrDigits);
  if (warp == kEpiWarps) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmem) : "memory");
  }
}

// The results: row r of the list, y[i] = (sum over the K splits of the integers) x the scales
// of the row of X and of row i of K^+.  Boundary form: to cbuf at the interface slots; full
// form: to dst (nullable) and, at the copy slots, to cbuf (nullable).  One CTA per row.
__global__ void __launch_bounds__(256) k_dg_scatter(DevMesh M, const DgBlock* __restrict__ blocks,
                                                    const DgRow* __restrict__ rows, int full,
                                                    const long long* __restrict__ out, const double* __restrict__ sA,
                                                    const double* __restrict__ sB, double* __restrict__ cbuf,
                                                    double* __restrict__ dst) {
  extern __shared__ double ys[];
  const DgRow row = rows[blockIdx.x];
  const DgBlock& blk = blocks[row.blk];
  const SubDev& S = M.subs[row.sub];
  const int n = full ? blk.n : blk.n_bd, splits = full ? blk.splits : blk.splits_bd;
  const long long ld = full ? blk.ld : blk.ld_bd;
  const long long* o = out + (full ? blk.o_off : blk.o_off_bd) + (long long)row.local * ld;
  const long long zs = (long long)blk.rows_pad * ld;
  const double a = sA[blockIdx.x];
  const double* b = sB + (full ? blk.sb_off : blk.sb_off_bd);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    long long t = o[i];
    for (int z = 1; z < splits; ++z) t += o[i + z * zs];
    const double y = ((double)t * (1.0 / (1LL << kUnit)) * a) * b[i];
    if (!full) {
      const int sl = __ldg(M.sub_b2s + S.b2s_off + i / 3);
      if (sl >= 0) cbuf[(long long)sl + i % 3] = y;
    } else {
      if (dst) dst[S.dof_off + i] = y;
      if (cbuf) ys[i] = y;
    }
  }
  if (full && cbuf) {
    __syncthreads();
    for (int s = threadIdx.x; s < S.n_copy; s += blockDim.x) {
      const long long slot = S.copy_off + s;
      cbuf[slot] = ys[__ldg(M.slot_ldof + slot)];
    }
  }
}

}  // namespace

int dg_nk(int n) { return (n + kK - 1) / kK; }
int dg_chunk_stages() { return kChunk; }
double dg_flops(int rows, int n) { return 2.0 * (kS * (kS + 1) / 2) * (double)rows * n * n; }
long long dg_a_elems(int rows_pad, int n) { return (long long)rows_pad * dg_nk(n) * kK * kS; }
long long dg_b_elems(int n) { return (long long)((n + kN - 1) / kN) * kN * dg_nk(n) * kK * kS; }

void launch_dg_split_k(const DevMesh& M, long long bnd_off, int n, int n_bd, bool full, const double* kinv, void* B,
                       double* sB, cudaStream_t st) {
  const int rows = full ? n : n_bd;
  if (rows <= 0) return;
  k_dg_split_k<<<(unsigned)((rows + kN - 1) / kN * kN), 256, 0, st>>>(M, bnd_off, n, n_bd, full ? 1 : 0, kinv,
                                                                       static_cast<uint4*>(B), sB);
}

int launch_dg_product(const DevMesh& M, const DgArgs& a, const double* src, const double* lam, double sign, double* cbuf,
                      double* dst, cudaStream_t st) {
  if (a.n_rows <= 0) return 0;
  const int full = a.full ? 1 : 0;
  const size_t xsm = sizeof(double) * (size_t)dg_nk(a.max_n) * kK;
  k_dg_split_x<<<a.n_rows, 256, xsm, st>>>(M, a.blocks, a.rows, full, src, lam, sign, static_cast<uint4*>(a.A), a.sA);
  cudaFuncSetAttribute(k_dg_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
  k_dg_gemm<<<a.n_ctas, kGemmThreads, kGemmSmem, st>>>(a.blocks, a.ctas, full,
                                                       static_cast<const unsigned char*>(a.A),
                                                       static_cast<const unsigned char*>(a.B), a.out, a.err, a.wait_limit);
  k_dg_scatter<<<a.n_rows, 256, xsm, st>>>(M, a.blocks, a.rows, full, a.out, a.sA, a.sB, cbuf, dst);
  return 3;
}

}  // namespace tfeti
