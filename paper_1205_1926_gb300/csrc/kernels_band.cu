// Batched banded Cholesky of the regularised subdomain matrices K_rr and the
// generalised-inverse apply K^+ x (Remark 1: fixing dofs replaced by identity
// rows, forward and backward substitution).
//
// Band workspace (per subdomain, n rows, half bandwidth bw, W = bw + 1):
//   band[r*W + k] = K[r][r - bw + k] on input, L[r][r - bw + k] after factorisation.
//
// Factor record written by the factorisation and read by the solves, for row
// blocks b of nb rows (r0 = b nb):
//   panel b : M_b = L_bb^{-1} L_b,off, nb x bw, entry (t, j) = column r0 - bw + j
//   dinv b  : L_bb^{-1}, nb x nb lower triangular
// With L = D (I + N), D = blockdiag(L_bb), N_b = M_b:
//   L^{-1} x = (I + N)^{-1} D^{-1} x   and   L^{-T} y = D^{-T} (I + N)^{-T} y,
// so each step of the forward and backward block recurrences is one GEMV with
// a panel, and the triangular blocks are applied in parallel before and after.
#include <algorithm>
#include <cstdint>

#include "async_common.cuh"
#include "dev.h"
#include "diag_chol.cuh"
#include "dual_common.cuh"

namespace tfeti {

namespace {

constexpr int kThreads = 256;
constexpr int kThreads32 = 512;   // of the FP32 one-CTA solve, whose steps are bound by latency
constexpr int kSolveStages = 6;   // most panels in flight in the one-CTA solve
constexpr int kNB1 = kMaxNB + 1;

// ---------------------------------------------------------------------------
// Factorisation: a cluster of C CTAs per subdomain, right-looking by block
// columns of nb.  Per block column every CTA factors the diagonal block and
// inverts it (identical, deterministic results, no exchange needed); the CTAs
// split the factor-record panel of the block row, the panel TRSM through the
// inverse and the SYRK update of the trailing band.  Two cluster barriers per
// block column order the global-memory band updates between the CTAs.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cluster_sync_all() {
  __threadfence();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}

__global__ void __launch_bounds__(kThreads) k_band_chol(DevMesh M, const int* __restrict__ sub_list,
                                                         const long long* __restrict__ off_list, double* band,
                                                         const long long* __restrict__ fac_list, double* fac_pool,
                                                         int* err) {
  extern __shared__ double sm[];
  double* Dm = sm;                       // [NB][NB+1] diagonal block -> its Cholesky factor
  double* Di = Dm + kMaxNB * kNB1;       // [NB][NB+1] inverse of the factor
  double* Lp = Di + kMaxNB * kNB1;       // [bw][NB+1] panel
  const int C = (int)cluster_size(), q = (int)cluster_rank();
  const int item = blockIdx.x / C;
  const int p = sub_list[item];
  const SubDev S = M.subs[p];
  double* A = band + off_list[item];
  double* fac = fac_pool + fac_list[item];
  double* dinv = fac + (long long)S.nblk * S.rec;
  const int n = S.n_dof, bw = S.bw, W = bw + 1, NB = S.nb;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int j0 = 0, b = 0; j0 < n; j0 += NB, ++b) {
    const int jb = min(NB, n - j0);
    #pragma unroll 4
    for (int idx = tid; idx < jb * jb; idx += nt) {
      const int r = idx / jb, c = idx % jb;
      Dm[r * kNB1 + c] = (c <= r) ? A[(long long)(j0 + r) * W + c - r + bw] : 0.0;
    }
    __syncthreads();
    diag_factor_invert(Dm, Di, jb, err, 1);
    // factor record of block row b (split over the cluster): dinv and M_b = Di * L[b rows][j0-bw .. j0)
    if (q == 0)
      for (int idx = tid; idx < NB * NB; idx += nt) {
        const int t = idx / NB, u = idx % NB;
        dinv[(long long)b * NB * NB + idx] = (t < jb && u < jb && u <= t) ? Di[t * kNB1 + u] : 0.0;
      }
    double* panel = fac + (long long)b * S.rec;
    {
      const int chunk = (S.rec + C - 1) / C;
      const int lo = q * chunk, hi = min(S.rec, lo + chunk);
      for (int idx = lo + tid; idx < hi; idx += nt) {
        double v = 0.0;
        const int t = idx / bw, j = idx % bw;
        const int c = j0 - bw + j;
        if (idx < NB * bw && t < jb && c >= 0) {
          for (int u = 0; u <= t; ++u) {
            const int k = c - (j0 + u) + bw;
            if (k >= 0) v += Di[t * kNB1 + u] * A[(long long)(j0 + u) * W + k];
          }
        }
        panel[idx] = v;
      }
    }
    const int i0 = j0 + jb;
    const int P = min(bw, n - i0);
    if (P > 0) {
      // panel TRSM, rows split over the cluster: L[i][j0+c] = sum_{s<=c} A[i][j0+s] Di[c][s]
      const int rchunk = (P + C - 1) / C;
      const int t0 = q * rchunk, t1 = min(P, t0 + rchunk);
      #pragma unroll 4
      for (int idx = tid; idx < (t1 - t0) * jb; idx += nt) {
        const int t = t0 + idx / jb, c = idx % jb;
        const int i = i0 + t, k = j0 + c - i + bw;
        Lp[t * kNB1 + c] = (k >= 0) ? A[(long long)i * W + k] : 0.0;
      }
      __syncthreads();
      for (int idx = tid; idx < (t1 - t0) * jb; idx += nt) {
        const int t = t0 + idx / jb, c = idx % jb;
        double v = 0.0;
        for (int s2 = 0; s2 <= c; ++s2) v += Lp[t * kNB1 + s2] * Di[c * kNB1 + s2];
        const int i = i0 + t, k = j0 + c - i + bw;
        if (k >= 0) A[(long long)i * W + k] = v;
      }
    }
    cluster_sync_all();
    if (P > 0) {
      #pragma unroll 4
      for (int idx = tid; idx < P * jb; idx += nt) {
        const int t = idx / jb, c = idx % jb;
        const int i = i0 + t, k = j0 + c - i + bw;
        Lp[t * kNB1 + c] = (k >= 0) ? A[(long long)i * W + k] : 0.0;
      }
      __syncthreads();
      // trailing update A[i][i'] -= sum_c L[i][c] L[i'][c], lower triangle split over the cluster
      const int ntri = P * (P + 1) / 2;
      const int tchunk = (ntri + C - 1) / C;
      const int l0 = q * tchunk, l1 = min(ntri, l0 + tchunk);
      for (int L = l0 + tid; L < l1; L += nt) {
        int t = (int)((sqrtf(8.0f * (float)L + 1.0f) - 1.0f) * 0.5f);
        while (t * (t + 1) / 2 > L) --t;
        while ((t + 1) * (t + 2) / 2 <= L) ++t;
        const int tp = L - t * (t + 1) / 2;
        double v = 0.0;
        for (int c = 0; c < jb; ++c) v += Lp[t * kNB1 + c] * Lp[tp * kNB1 + c];
        const int i = i0 + t, ip = i0 + tp;
        A[(long long)i * W + ip - i + bw] -= v;
      }
    }
    cluster_sync_all();
  }
}

// ---------------------------------------------------------------------------
// Subdomain solve: one CTA applies K^+ to up to kMaxRHS subdomains of one
// shape that share a factor record.  Shared memory: a.stages panel buffers
// (nb x bw entries each) filled ahead by bulk copies, the local vectors, one
// mbarrier per buffer.
// ---------------------------------------------------------------------------

// Right-hand sides of an item into vec (stride npad), by all threads of a CTA; ends with a barrier.
template <typename T>
__device__ __forceinline__ void load_rhs(const DevMesh& M, const SolveArgs& a, const SolveItem& item, const SubDev& S0,
                                         T* vec, int npad) {
  const int n = S0.n_dof, R = item.count, tid = threadIdx.x, nt = blockDim.x;
  if (a.in_mode == 2 || a.in_mode == 5) {   // unit vectors at boundary dofs (2) or local dofs (5) item.sub[r]
    for (int r = 0; r < R; ++r)
      for (int i = tid; i < n; i += nt) vec[r * npad + i] = T(0);
    __syncthreads();
    if (tid < R) {
      const int j = item.sub[tid];
      vec[tid * npad + (a.in_mode == 2 ? 3 * M.shape_bln[S0.bnd_off + j / 3] + j % 3 : j)] = T(1);
    }
  }
  const bool unit_in = a.in_mode == 2 || a.in_mode == 5;
  for (int r = 0; r < R && !unit_in; ++r) {
    const SubDev& S = M.subs[item.sub[r]];
    T* x = vec + r * npad;
    if (a.in_mode == 0)
      for (int i = tid; i < n; i += nt) x[i] = T(0);
    else if (a.in_mode == 4)
      for (int i = tid; i < n; i += nt) x[i] = T(a.src[S.dof_off + box_dof(S, i)]);
    else
      for (int i = tid; i < n; i += nt) x[i] = a.src ? T(a.src[S.dof_off + i]) : T(0);
  }
  __syncthreads();
  constexpr int U = 4;   // copy slots per thread with their B^T gathers in flight together
  for (int r = 0; r < R && !unit_in && a.in_mode != 4 && a.lam; ++r) {
    const SubDev& S = M.subs[item.sub[r]];
    T* x = vec + r * npad;
    for (int s0 = tid; s0 < S.n_copy; s0 += U * nt) {
      long long sl[U];
      double v[U];
#pragma unroll
      for (int k = 0; k < U; ++k) sl[k] = s0 + k * nt < S.n_copy ? S.copy_off + s0 + k * nt : -1;
      bt_at_slots<U>(M, a.lam, sl, v);
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (sl[k] >= 0) {
          const int d = __ldg(M.slot_ldof + sl[k]);
          x[d] = a.in_mode == 0 ? T(v[k]) : x[d] - T(v[k]);
        }
    }
  }
  __syncthreads();
  if (tid < 6 && !a.no_fix)
    for (int r = 0; r < R; ++r) vec[r * npad + S0.fix[tid]] = T(0);
  __syncthreads();
}

// Sums over the warp of NR values per lane: lane / (32 / NR) gets the sum of v[lane / (32 / NR)].
template <typename T, int NR>
__device__ __forceinline__ T warp_sum_rows(T (&v)[NR], int lane) {
  T k;
  int o;
  if constexpr (NR == 4) {
    const bool h = lane & 16, g = lane & 8;
    T a = h ? v[2] : v[0], b = h ? v[3] : v[1];
    a += __shfl_xor_sync(0xffffffffu, h ? v[0] : v[2], 16);
    b += __shfl_xor_sync(0xffffffffu, h ? v[1] : v[3], 16);
    k = g ? b : a;
    k += __shfl_xor_sync(0xffffffffu, g ? a : b, 8);
    o = 4;
  } else if constexpr (NR == 2) {
    const bool h = lane & 16;
    k = h ? v[1] : v[0];
    k += __shfl_xor_sync(0xffffffffu, h ? v[0] : v[1], 16);
    o = 8;
  } else {
    k = v[0];
    o = 16;
  }
  for (; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  return k;
}

// Forward step in FP32, where the shared-memory reads bound it: a warp takes NR whole rows of the block,
// the lanes the columns, so that a column's x is read once for NR rows and no two lanes share a bank.
template <int R, int NR>
__device__ __forceinline__ void forward_rows32(const float* P, int bw, int jlo, int c0, int r0, int jb, float* vec,
                                               int npad) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* prow = P + warp * NR * bw;
  float acc[R][NR] = {};
#pragma unroll 4
  for (int j = jlo + lane; j < bw; j += 32) {
    float x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = vec[r * npad + c0 + j];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const float mv = prow[i * bw + j];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r][i] = fmaf(mv, x[r], acc[r][i]);
    }
  }
  const int t = warp * NR + lane / (32 / NR);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float v = warp_sum_rows<float, NR>(acc[r], lane);
    if (lane % (32 / NR) == 0 && t < jb) vec[r * npad + r0 + t] -= v;
  }
}

// The sweeps of one item with R right-hand sides, all threads of a CTA; the panels of the first NS steps
// (buffers of pstride entries at pan) are on their way.  Returns -1, or the step whose panel copy did not
// complete.
template <typename T, int R>
__device__ int sweep(const SubDev& S0, const T* __restrict__ fac, const T* __restrict__ dinv, const T* pan, int pstride,
                     int NS, T* vec, int npad, uint64_t* bar, int* s_fail, long long limit) {
  const int n = S0.n_dof, bw = S0.bw, nb = S0.nb, nblk = S0.nblk, rec = S0.rec;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nsteps = 2 * nblk;
  const uint32_t pbytes = (uint32_t)rec * (uint32_t)sizeof(T);
  auto step_block = [nblk, nsteps](int k) { return k < nblk ? k : nsteps - 1 - k; };
  // ---- x' = D^{-1} x, block-diagonal, 256 rows at a time through registers
  for (int base = 0; base < n; base += nt) {
    const int i = base + tid;
    T v[R] = {};
    if (i < n) {
      const int b = i / nb, t = i - b * nb, r0 = b * nb;
      const T* drow = dinv + (long long)b * nb * nb + t * nb;
      for (int q = 0; q <= t; ++q) {
        const T d = drow[q];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = fma(d, vec[r * npad + r0 + q], v[r]);
      }
    }
    __syncthreads();
    if (i < n)
#pragma unroll
      for (int r = 0; r < R; ++r) vec[r * npad + i] = v[r];
    __syncthreads();
  }

  // ---- block recurrences: forward y_b = x'_b - M_b y[r0-bw, r0), then backward
  //      z'[r0-bw, r0) -= M_b^T z'_b for b = nblk-1 .. 0
  // forward rows: 8 lanes each, or 16 where a block has at most 16 rows
  const int lpr = nb <= 16 ? 16 : 8, frow = tid / lpr, l = tid % lpr;
  int k_fail = -1, buf = 0;
  uint32_t phase = 0;
  for (int k = 0; k < nsteps; ++k) {
    const bool ok = limit != 0 && mbar_wait(&bar[buf], phase, limit);
    if (!ok) *s_fail = 1;
    const T* P = pan + buf * pstride;
    const int b = step_block(k);
    const int r0 = b * nb, jb = min(nb, n - r0);
    const int c0 = r0 - bw, jlo = max(0, -c0);
    if (ok) {
      bool done = false;
      if constexpr (sizeof(T) == 4) {
        if (k < nblk && nb == 32) forward_rows32<R, 32 * 32 / kThreads32>(P, bw, jlo, c0, r0, jb, vec, npad), done = true;
        else if (k < nblk && nb == 16) forward_rows32<R, 16 * 32 / kThreads32>(P, bw, jlo, c0, r0, jb, vec, npad), done = true;
      }
      if (done) {
      } else if (k < nblk) {
        const int t = frow;
        const bool act = t < jb;
        T acc[R] = {};
        if (act) {
          const T* prow = P + t * bw;
#pragma unroll 8
          for (int j = jlo + l; j < bw; j += lpr) {
            const T mv = prow[j];
            const int c = c0 + j;
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fma(mv, vec[r * npad + c], acc[r]);
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (lpr == 16) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], 8);
          acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], 4);
          acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], 2);
          acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], 1);
        }
        if (act && l == 0)
#pragma unroll
          for (int r = 0; r < R; ++r) vec[r * npad + r0 + t] -= acc[r];
      } else {
        // one (column, right-hand side) pair per thread: bw * R units spread evenly over the CTA
        const int units = (bw - jlo) * R;
        for (int u = tid; u < units; u += nt) {
          const int j = jlo + u / R, r = u - (u / R) * R;
          const int c = c0 + j;
          const T* zr = vec + r * npad + r0;
          T acc = T(0);
          int t = 0;
          if constexpr (sizeof(T) == 4) {   // z' four at a time (nb a multiple of 4 puts them on 16 bytes)
            if ((nb & 3) == 0)
#pragma unroll 4
              for (; t + 4 <= jb; t += 4) {
                const float4 z = *reinterpret_cast<const float4*>(zr + t);
                acc = fmaf(P[t * bw + j], z.x, acc);
                acc = fmaf(P[(t + 1) * bw + j], z.y, acc);
                acc = fmaf(P[(t + 2) * bw + j], z.z, acc);
                acc = fmaf(P[(t + 3) * bw + j], z.w, acc);
              }
          }
#pragma unroll 8
          for (; t < jb; ++t) acc = fma(P[t * bw + j], zr[t], acc);
          vec[r * npad + c] -= acc;
        }
      }
    }
    __syncthreads();
    if (*s_fail) {
      k_fail = k;
      break;
    }
    if (tid == 0 && k + NS < nsteps)
      bulk_copy(const_cast<T*>(P), fac + (long long)step_block(k + NS) * rec, pbytes, &bar[buf]);
    if (++buf == NS) {
      buf = 0;
      phase ^= 1;
    }
  }
  if (k_fail >= 0) return k_fail;

  // ---- z = D^{-T} z'
  for (int base = 0; base < n; base += nt) {
    const int i = base + tid;
    T v[R] = {};
    if (i < n) {
      const int b = i / nb, t = i - b * nb, r0 = b * nb;
      const int jb = min(nb, n - r0);
      const T* dblk = dinv + (long long)b * nb * nb;
      for (int s = t; s < jb; ++s) {
        const T d = dblk[s * nb + t];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = fma(d, vec[r * npad + r0 + s], v[r]);
      }
    }
    __syncthreads();
    if (i < n)
#pragma unroll
      for (int r = 0; r < R; ++r) vec[r * npad + i] = v[r];
    __syncthreads();
  }
  return -1;
}

template <typename T>
__global__ void __launch_bounds__(sizeof(T) == 4 ? kThreads32 : kThreads, 1) k_sub_solve(DevMesh M, SolveArgs a) {
  extern __shared__ __align__(128) unsigned char sm_raw[];
  T* sm = reinterpret_cast<T*>(sm_raw);
  __shared__ int s_fail;
  const SolveItem item = a.items[blockIdx.x];
  // unit right-hand sides (in_mode 2, 5) carry dof indices in item.sub[]: the geometry is rep_sub's
  const SubDev& S0 = M.subs[(a.in_mode == 2 || a.in_mode == 5) ? a.rep_sub : item.sub[0]];
  const int n = S0.n_dof, bw = S0.bw, nb = S0.nb, nblk = S0.nblk, rec = S0.rec;
  const int R = item.count;
  const int npad = a.npad;                       // vector stride (largest n of the launch, even)
  const int NS = a.stages;
  T* pan = sm;                                   // [NS][rec_max]
  T* vec = sm + NS * a.rec_max;                  // [rcap][npad]
  uint64_t* bar = reinterpret_cast<uint64_t*>(vec + ((a.rcap * npad + 1) & ~1));
  const bool own = (item.fac & kOwnFac) != 0;
  const T* fac = (sizeof(T) == 8 ? reinterpret_cast<const T*>(own ? a.fac_own : a.fac)
                                 : reinterpret_cast<const T*>(own ? a.fac32_own : a.fac32)) +
                 (item.fac & ~kOwnFac);
  const T* dinv = fac + (long long)nblk * rec;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int nsteps = 2 * nblk;
  const uint32_t pbytes = (uint32_t)rec * (uint32_t)sizeof(T);

  if (tid == 0) {
    s_fail = 0;
    for (int k = 0; k < NS; ++k) mbar_init(&bar[k]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // step k uses the panel of block k (forward, k < nblk) or 2 nblk - 1 - k (backward)
  auto step_block = [nblk, nsteps](int k) { return k < nblk ? k : nsteps - 1 - k; };
  if (tid == 0)
    for (int k = 0; k < NS && k < nsteps; ++k)
      bulk_copy(pan + k * a.rec_max, fac + (long long)step_block(k) * rec, pbytes, &bar[k]);

  const int n_bd = 3 * S0.n_bnd;
  load_rhs<T>(M, a, item, S0, vec, npad);
  // the sweeps are compiled for the item's number of right-hand sides: an FP64 instruction occupies
  // the pipe also where its predicate is off (a single right-hand side took 1200 us of the four's
  // 1600 us for a 2187-dof box when all four were predicated)
  int k_fail;
  if (R == 1) k_fail = sweep<T, 1>(S0, fac, dinv, pan, a.rec_max, NS, vec, npad, bar, &s_fail, a.wait_limit);
  else if (R == 2) k_fail = sweep<T, 2>(S0, fac, dinv, pan, a.rec_max, NS, vec, npad, bar, &s_fail, a.wait_limit);
  else if (R == 3) k_fail = sweep<T, 3>(S0, fac, dinv, pan, a.rec_max, NS, vec, npad, bar, &s_fail, a.wait_limit);
  else k_fail = sweep<T, 4>(S0, fac, dinv, pan, a.rec_max, NS, vec, npad, bar, &s_fail, a.wait_limit);
  if (k_fail >= 0) {
    // a panel copy never completed: report, give the copies still in flight (steps k_fail ..
    // k_fail + NS - 1) a bounded time to land, and leave
    if (tid == 0) {
      atomicOr(a.err, kErrPanel);
      for (int k = k_fail; k < k_fail + NS && k < nsteps; ++k) mbar_wait(&bar[k % NS], (uint32_t)((k / NS) & 1));
    }
    return;
  }
  if (tid < 6 && !a.no_fix)
    for (int r = 0; r < R; ++r) vec[r * npad + S0.fix[tid]] = T(0);
  __syncthreads();

  // ---- outputs
  if (a.out_mode == 4) {   // column item.sub[r] of the dense K^+ of the geometry rep_sub, FP64
    for (int r = 0; r < R; ++r) {
      const long long o = a.s_off + (long long)item.sub[r] * n;
      for (int i = tid; i < n; i += nt) a.S64[o + i] = (double)vec[r * npad + i];
    }
    return;
  }
  if (a.out_mode == 2) {
    for (int r = 0; r < R; ++r) {
      const long long o = a.s_off + (long long)item.sub[r] * n_bd;
      for (int i = tid; i < n_bd; i += nt) {
        const T v = vec[r * npad + 3 * M.shape_bln[S0.bnd_off + i / 3] + i % 3];
        a.S32[o + i] = (float)v;
        if (a.S64) a.S64[o + i] = (double)v;
      }
    }
    return;
  }
  for (int r = 0; r < R; ++r) {
    const int p = item.sub[r];
    const SubDev& S = M.subs[p];
    const T* x = vec + r * npad;
    if (a.out_mode == 0 || a.out_mode == 3) {
      for (int s = tid; s < S.n_copy; s += nt) {
        const long long slot = S.copy_off + s;
        a.cbuf[slot] = double(x[M.slot_ldof[slot]]);
      }
    }
    if (a.out_mode == 1 || a.out_mode == 3) {
      const double* Rb = M.R + S.r_off;
      for (int i = tid; i < n; i += nt) {
        double v = double(x[i]);
        if (a.alpha) {
          const double* al = a.alpha + 6 * (long long)p;
          for (int c = 0; c < 6; ++c) v += Rb[(long long)i * 6 + c] * al[c];
        }
        a.dst[S.dof_off + (a.in_mode == 4 ? box_dof(S, i) : i)] = v;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// The same solve by a cluster of C CTAs per item, for launches with fewer items than SMs.  One
// CTA per item leaves its two sweeps of 2 n / nb dependent block steps to one SM, whose FP64 pipe
// (two FMAs per clock) then sets the time.  Here CTA q owns rows [q nb / C, (q + 1) nb / C) of every
// block and streams only those rows of the panels:
//   forward:  y_t = x'_t - M_b[t][:] y[r0 - bw, r0) for its rows, sent to all CTAs' vectors;
//   backward: its rows' terms M_b[t][:] z'_t go into a running sum per column, kept by one thread
//             from the column's first step to its last; when a column's block is next, the sums
//             are sent to the rows' owners (before the other columns are worked on), which add them
//             in a fixed order and finish z'_t.
// The values travel as asynchronous remote stores that complete on an mbarrier of the receiver, so a
// step waits for one crossing and no CTA can run more than one step ahead; the panel slices arrive
// by bulk copies several steps ahead.
// ---------------------------------------------------------------------------
constexpr int kClThreads = 128;
constexpr int kClStages = 4;   // panel slices in flight
constexpr int kClRing = 4;     // exchange barriers and receive buffers in turn

__device__ __forceinline__ uint32_t cluster_addr(const void* p, unsigned rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(const double* p, unsigned rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(p, rank)), "d"(v) : "memory");
}
// Remote store of v to p in CTA rank, completing sizeof(v) bytes on bar there.
__device__ __forceinline__ void st_async(const double* p, const uint64_t* bar, unsigned rank, double v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(
                   cluster_addr(p, rank)),
               "l"(__double_as_longlong(v)), "r"(cluster_addr(bar, rank))
               : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() {
  cluster_arrive();
  cluster_wait();
}

// Shared memory of a cluster CTA in doubles: panel slices, the vectors, the own rows' x', the
// window of column sums (a power of two above bw + nb), the received sums.
struct ClLayout {
  int slice, npad, own, win, recv;
  __host__ __device__ ClLayout(int rec_max, int npad_, int max_bw, int C)
      : slice((rec_max / C + 3) & ~3), npad(npad_), own(npad_ / C + 2 * kMaxNB), recv(kClRing * kMaxNB) {
    win = 128;
    while (win < max_bw + kMaxNB) win *= 2;
  }
  __host__ __device__ size_t values(int R) const {
    return (size_t)kClStages * slice + (size_t)R * ((size_t)npad + own + win + recv);
  }
};

// R right-hand sides, NR own rows of a block per warp (nb / C = 4 NR).
template <int R, int NR>
__device__ void cl_solve(const DevMesh& M, const SolveArgs& a, const SolveItem& item, int C, unsigned q, double* sm,
                         uint64_t* bar, uint64_t* xbar) {
  using T = double;
  constexpr int rpc = 4 * NR;
  __shared__ T s_z[4][rpc][R];     // backward: z' of the own rows, one copy per warp
  const SubDev& S0 = M.subs[item.sub[0]];
  const int n = S0.n_dof, bw = S0.bw, nb = S0.nb, nblk = S0.nblk, rec = S0.rec;
  const ClLayout lay(a.rec_max, a.npad, a.max_bw, C);
  T* pan = sm;
  T* vec = pan + kClStages * lay.slice;      // [R][npad]
  T* xo = vec + R * lay.npad;                // [R][own]: x' of the own rows
  T* win = xo + R * lay.own;                 // [R][win]
  T* recv = win + R * lay.win;               // [kClRing][C][rpc][R]
  const int npad = lay.npad, wmask = lay.win - 1;
  const bool own = (item.fac & kOwnFac) != 0;
  const T* fac = (own ? a.fac_own : a.fac) + (item.fac & ~kOwnFac);
  const T* dinv = fac + (long long)nblk * rec;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nsteps = 2 * nblk;
  const uint32_t pbytes = (uint32_t)(rpc * bw) * (uint32_t)sizeof(T);   // rpc is a multiple of 4
  auto step_block = [nblk, nsteps](int k) { return k < nblk ? k : nsteps - 1 - k; };
  auto fetch = [&](int k) {
    bulk_copy(pan + (k % kClStages) * lay.slice, fac + (long long)step_block(k) * rec + (long long)q * rpc * bw, pbytes,
              &bar[k % kClStages]);
  };
  // after a wait that gave up, the remaining steps run through without waiting; thread 0 then neither fetches
  // panels nor opens exchange phases any more (a phase may be opened once the one before it has completed)
  bool ok = a.wait_limit != 0;
  auto wait_panel = [&](int k) {
    if (ok) ok = mbar_wait(&bar[k % kClStages], (uint32_t)((k / kClStages) & 1), a.wait_limit);
  };
  auto wait_exchange = [&](int e) {
    if (ok) ok = mbar_wait_cluster(&xbar[e % kClRing], (uint32_t)((e / kClRing) & 1), a.wait_limit);
  };
  int issued = 0;
  if (tid == 0)
    for (; issued < kClStages && issued < nsteps; ++issued) fetch(issued);
  load_rhs<T>(M, a, item, S0, vec, npad);

  // x' = D^-1 x on the own rows, one (block, row) per thread
  for (int i = tid; i < nblk * rpc; i += kClThreads) {
    const int b = i / rpc, t = (int)q * rpc + i % rpc, r0 = b * nb;
    T v[R] = {};
    if (r0 + t < n) {
      const T* drow = dinv + (long long)b * nb * nb + t * nb;
      for (int u = 0; u <= t; ++u) {
        const T d = drow[u];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = fma(d, vec[r * npad + r0 + u], v[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) xo[r * lay.own + i] = v[r];
  }
  for (int i = tid; i < R * lay.win; i += kClThreads) win[i] = T(0);
  cluster_barrier();   // every CTA has read its x (and set its barriers up) before the first y arrives

  // forward: a warp's NR rows, columns across the lanes
  for (int k = 0; k < nblk; ++k) {
    const int r0 = k * nb, c0 = r0 - bw, jlo = max(0, -c0);
    if (tid == 0 && ok) mbar_expect_tx(&xbar[k % kClRing], (uint32_t)(min(nb, n - r0) * R * (int)sizeof(T)));
    wait_panel(k);
    const T* P = pan + (k % kClStages) * lay.slice + warp * NR * bw;
    T acc[R][NR] = {};
#pragma unroll 4
    for (int j = jlo + lane; j < bw; j += 32) {
      T x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = vec[r * npad + c0 + j];
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        const T mv = P[i * bw + j];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r][i] = fma(mv, x[r], acc[r][i]);
      }
    }
    const int t = warp * NR + lane / (32 / NR), dst = lane % (32 / NR), gr = r0 + (int)q * rpc + t;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const T v = xo[r * lay.own + k * rpc + t] - warp_sum_rows<T, NR>(acc[r], lane);
      if (dst < C && gr < n) st_async(vec + r * npad + gr, &xbar[k % kClRing], (unsigned)dst, v);
    }
    wait_exchange(k);
    __syncthreads();
    if (tid == 0 && ok && issued < nsteps) fetch(issued++);
  }
  cluster_arrive();   // every y has arrived in this CTA's vectors
  // backward: column c belongs to lane c % 32 of warp (c / 32) % 4 from its first step to its last
  for (int k = nblk; k < nsteps; ++k) {
    const int b = nsteps - 1 - k, r0 = b * nb, lo = max(0, r0 - bw), nxt = r0 - nb;
    if (tid == 0 && ok && b > 0) mbar_expect_tx(&xbar[k % kClRing], (uint32_t)(nb * R * (int)sizeof(T)));
    // z' of the own rows: y less the CTAs' sums (lane = CTA x row), in every warp
    if (k > nblk) wait_exchange(k - 1);
    T zv[R];
    {
      const int t = lane % rpc, c = lane / rpc, gr = r0 + (int)q * rpc + t;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        T v = (k > nblk && c < C) ? recv[((((k - 1) % kClRing) * C + c) * rpc + t) * R + r] : T(0);
        for (int o = rpc; o < rpc * C; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane < rpc) {
          v = gr < n ? vec[r * npad + gr] - v : T(0);
          s_z[warp][t][r] = v;
        }
        zv[r] = v;
      }
    }
    __syncwarp();
    wait_panel(k);
    const T* P = pan + (k % kClStages) * lay.slice;
    const int top = (r0 - 1) >> 5;
    for (int u = top - ((top - warp) & 3); b > 0 && 32 * u + 31 >= min(lo, nxt) && u >= 0; u -= 4) {
      const int c = 32 * u + lane;
      if (c >= r0 || c < min(lo, nxt)) continue;
      T s[R];
#pragma unroll
      for (int r = 0; r < R; ++r) s[r] = win[r * lay.win + (c & wmask)];
      if (c >= lo) {
        const T* pc = P + (c - (r0 - bw));
#pragma unroll
        for (int t = 0; t < rpc; ++t) {
          const T mv = pc[t * bw];
#pragma unroll
          for (int r = 0; r < R; ++r) s[r] = fma(mv, s_z[warp][t][r], s[r]);
        }
      }
      const int t = c - nxt;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        // block b - 1 is next: its sums to the rows' owners; the window slot is free again
        if (t >= 0)
          st_async(recv + (((k % kClRing) * C + (int)q) * rpc + t % rpc) * R + r, &xbar[k % kClRing],
                   (unsigned)(t / rpc), s[r]);
        win[r * lay.win + (c & wmask)] = t >= 0 ? T(0) : s[r];
      }
    }
    __syncthreads();
    // z' to CTA b % C, which applies the block's D^-T below (only now: until here every warp of that CTA
    // may still read the y of its own rows from the same entries; and in the first step a y sent there must
    // not arrive after the z' that replaces it: the sums received before the later steps tell that it has)
    if (k == nblk) cluster_wait();
    if (warp == 0 && lane < rpc && r0 + (int)q * rpc + lane < n)
#pragma unroll
      for (int r = 0; r < R; ++r) st_cluster(vec + r * npad + r0 + (int)q * rpc + lane, (unsigned)(b % C), zv[r]);
    if (tid == 0 && ok && issued < nsteps) fetch(issued++);
  }
  if (!ok) atomicOr(a.err, kErrPanel);
  if (!ok && tid == 0)
    for (int k = max(0, issued - kClStages); k < issued; ++k)   // copies still in flight land first
      mbar_wait(&bar[k % kClStages], (uint32_t)((k / kClStages) & 1));
  cluster_barrier();   // the z' of the blocks below have arrived
  if (!ok) {           // the other CTAs' last asynchronous stores, which were not waited for, land before this CTA ends
    const long long t0 = clock64();
    while (clock64() - t0 < (1LL << 17)) {
    }
  }

  // z = D^-T z' on the blocks b % C == q
  __shared__ T s_col[kClThreads][R];
  const int rows_per = kClThreads / nb;   // blocks per round
  for (int i0 = (int)q; i0 < nblk; i0 += C * rows_per) {
    const int sub = tid / nb, t = tid % nb, b = i0 + sub * C, r0 = b * nb;
    const bool act = sub < rows_per && b < nblk && r0 + t < n;
    T v[R] = {};
    if (act) {
      const int jb = min(nb, n - r0);
      const T* dblk = dinv + (long long)b * nb * nb;
      for (int s = t; s < jb; ++s) {
        const T d = dblk[s * nb + t];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = fma(d, vec[r * npad + r0 + s], v[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) s_col[tid][r] = v[r];
    __syncthreads();
    if (act)
#pragma unroll
      for (int r = 0; r < R; ++r) vec[r * npad + r0 + t] = s_col[tid][r];
    __syncthreads();
  }
  if (tid < 6 && !a.no_fix)
    for (int r = 0; r < R; ++r) vec[r * npad + S0.fix[tid]] = T(0);   // (entries of other CTAs' blocks are not read)
  __syncthreads();
  for (int r = 0; r < item.count; ++r) {
    const SubDev& S = M.subs[item.sub[r]];
    const T* x = vec + r * npad;
    if (a.out_mode == 0 || a.out_mode == 3)
      for (int s = tid; s < S.n_copy; s += kClThreads) {
        const long long slot = S.copy_off + s;
        const int d = __ldg(M.slot_ldof + slot);
        if ((d / nb) % C == (int)q) a.cbuf[slot] = double(x[d]);
      }
    if (a.out_mode == 1 || a.out_mode == 3)
      for (int b = (int)q; b < nblk; b += C)
        for (int t = tid; t < nb && b * nb + t < n; t += kClThreads) {
          const int i = b * nb + t;
          a.dst[S.dof_off + (a.in_mode == 4 ? box_dof(S, i) : i)] = x[i];
        }
  }
}

template <int R>
__global__ void __launch_bounds__(kClThreads) k_solve_cl(DevMesh M, SolveArgs a) {
  extern __shared__ __align__(128) unsigned char sm_raw[];
  __shared__ uint64_t bar[kClStages], xbar[kClRing];
  const int C = (int)cluster_size();
  if (threadIdx.x == 0) {
    for (int k = 0; k < kClStages; ++k) mbar_init(&bar[k]);
    for (int k = 0; k < kClRing; ++k) mbar_init(&xbar[k]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const SolveItem item = a.items[blockIdx.x / C];
  double* sm = reinterpret_cast<double*>(sm_raw);
  const int rpc = M.subs[item.sub[0]].nb / C;   // 4, 8 or 16 (the same for the whole cluster)
  if (rpc == 4) cl_solve<R, 1>(M, a, item, C, cluster_rank(), sm, bar, xbar);
  else if (rpc == 8) cl_solve<R, 2>(M, a, item, C, cluster_rank(), sm, bar, xbar);
  else cl_solve<R, 4>(M, a, item, C, cluster_rank(), sm, bar, xbar);
}

// Launches the cluster form with C CTAs per item; false if it cannot run (nothing launched).
template <int R>
bool launch_cl(const DevMesh& M, const SolveArgs& a, int C, cudaStream_t st) {
  const ClLayout lay(a.rec_max, a.npad, a.max_bw, C);
  const size_t smem = sizeof(double) * lay.values(R);
  static const int lim = dyn_smem_limit((const void*)k_solve_cl<R>);
  if (smem > (size_t)lim) return false;
  cudaFuncSetAttribute(k_solve_cl<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(a.n_items * C));
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k_solve_cl<R>, M, a) == cudaSuccess) return true;
  cudaGetLastError();   // this launch's error, not one of an earlier call
  return false;
}

}  // namespace

// The device's opt-in shared-memory limit per block.  Kernels whose dynamic shared memory
// depends on the problem get the largest allowed size as their attribute (not the launch's
// own size), so that launches of different contexts from several host threads cannot
// undercut each other.
int smem_optin_max() {
  static const int v = [] {
    int dev = 0, m = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&m, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return m;
  }();
  return v;
}

// Largest dynamic shared memory a kernel may be given: the opt-in limit less its static
// shared memory (the two together must not exceed the limit).
int dyn_smem_limit(const void* fn) {
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) {
    cudaGetLastError();
    return 48 * 1024;
  }
  return smem_optin_max() - (int)fa.sharedSizeBytes;
}

static int sm_count() {
  int dev = 0, v = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  return v;
}

void launch_band_chol(const DevMesh& M, const int* sub_list, int n_list, const long long* band_off_list,
                      double* band, const long long* fac_off_list, double* fac, int* err, int max_bw,
                      int n_sm, cudaStream_t st) {
  if (n_list <= 0) return;
  const size_t smem = sizeof(double) * (2 * kMaxNB * kNB1 + (size_t)max_bw * kNB1);
  static const int lim = dyn_smem_limit((const void*)k_band_chol);
  cudaFuncSetAttribute(k_band_chol, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  const bool big = cudaFuncSetAttribute(k_band_chol, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                   cudaSuccess;
  if (!big) cudaGetLastError();
  // cluster size: the largest power of two with n_list * C <= 2 * n_sm (at most 16, or 8 if
  // non-portable cluster sizes are unavailable); 54 boxes of 8^3 elements take 17.4 ms with 4 CTAs each,
  // 19.8 ms with 8
  int C = 1;
  const int cmax = big ? 16 : 8;
  while (C < cmax && (long long)n_list * C * 2 <= 2LL * n_sm) C *= 2;
  for (;;) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(n_list * C));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int max_clusters = 0;
    if (C > 1 && (cudaOccupancyMaxActiveClusters(&max_clusters, k_band_chol, &cfg) != cudaSuccess ||
                  max_clusters < 1)) {
      cudaGetLastError();
      C /= 2;
      continue;
    }
    cudaLaunchKernelEx(&cfg, k_band_chol, M, sub_list, band_off_list, band, fac_off_list, fac, err);
    return;
  }
}

size_t sub_solve_smem(int rec_max, int npad, int rcap, int elem_bytes, int stages) {
  const size_t vec = ((size_t)rcap * npad + 1) & ~(size_t)1;
  return (size_t)elem_bytes * ((size_t)stages * rec_max + vec) + stages * sizeof(uint64_t);
}

void launch_sub_solve(const DevMesh& M, const SolveArgs& args, cudaStream_t st) {
  SolveArgs a = args;
  if (a.n_items <= 0) return;
  static const int n_sm = sm_count();
  // Cluster form for FP64 items of at most two right-hand sides: the most CTAs per item for which the
  // launch still has at most two per SM, counting the items by their work (n_eff = total work over
  // the largest item's; small boxes beside a large one end early).  Measured, pass of one CTA / 2 /
  // 4 / 8 CTAs per item: 54 boxes of 8^3 elements 559 / 432 / 354 / 499 us, 3 boxes of 6^3 (with
  // the other boxes' product) - / 167 / 123 / 102 us, 125 uneven boxes of 4..12 elements per edge
  // 1970 / 1401 / 1042 / - us.
  const bool plain = a.in_mode == 0 || a.in_mode == 1 || a.in_mode == 4;
  if (!a.fp32 && a.cl_max > 1 && a.max_count <= 2 && plain && !a.alpha) {
    int C = a.cl_max;
    while (C > 1 && a.n_eff * C > 2 * n_sm) C /= 2;
    if (C > 1) {
      if (a.max_count == 1 ? launch_cl<1>(M, a, C, st) : launch_cl<2>(M, a, C, st)) return;
    }
  }
  // One CTA per item.  A step's panel (35 KB in FP32 for an 8^3 box) takes about a microsecond from
  // L2 and a step a third of that, so as many panels are kept in flight as shared memory holds: of the
  // whole SM when the items fit one per SM, else of half of it.
  static const int lim64 = dyn_smem_limit((const void*)k_sub_solve<double>);
  static const int lim32 = dyn_smem_limit((const void*)k_sub_solve<float>);
  const int lim = a.fp32 ? lim32 : lim64, eb = a.fp32 ? 4 : 8;
  if (plain) a.rcap = std::max(1, std::min(a.rcap, a.max_count));
  const size_t room = a.n_items <= n_sm ? (size_t)lim : (size_t)lim / 2 - 1024;
  a.stages = 2;
  while (a.stages < kSolveStages && sub_solve_smem(a.rec_max, a.npad, a.rcap, eb, a.stages + 1) <= room) ++a.stages;
  const size_t smem = sub_solve_smem(a.rec_max, a.npad, a.rcap, eb, a.stages);
  if (a.fp32) {
    cudaFuncSetAttribute(k_sub_solve<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    k_sub_solve<float><<<a.n_items, kThreads32, smem, st>>>(M, a);
  } else {
    cudaFuncSetAttribute(k_sub_solve<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    k_sub_solve<double><<<a.n_items, kThreads, smem, st>>>(M, a);
  }
}

namespace {
__global__ void k_to_f32(const double* __restrict__ src, float* dst, const long long* __restrict__ off,
                         long long len) {
  const long long base = off[blockIdx.y];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < len; i += (long long)gridDim.x * blockDim.x)
    dst[base + i] = (float)src[base + i];
}
}  // namespace

void launch_fac_to_f32(const double* fac, float* fac32, const long long* off_list, int n_list, long long len,
                       cudaStream_t st) {
  if (n_list <= 0) return;
  dim3 grid(64, n_list);
  k_to_f32<<<grid, 256, 0, st>>>(fac, fac32, off_list, len);
}

namespace {
__global__ void k_to_f32_flat(const double* __restrict__ src, float* dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    dst[i] = (float)src[i];
}
}  // namespace

void launch_to_f32(const double* src, float* dst, long long n, cudaStream_t st) {
  if (n > 0) k_to_f32_flat<<<1024, 256, 0, st>>>(src, dst, n);
}

}  // namespace tfeti
