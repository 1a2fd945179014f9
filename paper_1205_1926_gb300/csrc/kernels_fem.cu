// FEM kernels: element tables, rigid-body modes, traction loads, the return
// mapping with its Clarke derivative (Sec. 2.4, Sec. 3.1), the element
// tangent corrections and the assembly of Algorithm 5 into banded subdomain
// matrices, the lumped-preconditioner blocks and the internal force.
#include <cfloat>

#include "dev.h"

namespace tfeti {

namespace {

constexpr double kSqrt32 = 1.2247448713915890491;   // sqrt(3/2), correctly rounded
constexpr double kSqrt23 = 0.81649658092772603273;  // sqrt(2/3), correctly rounded
constexpr double kTie = 1e-12;                       // exact-tie band of the elastic predictor test
constexpr double kThird = 1.0 / 3.0;

// element local node of offset (ox, oy, oz) -> index ox + 2 oy + 4 oz
__constant__ int c_off2local[8] = {0, 1, 3, 2, 4, 5, 7, 6};
__constant__ int c_local_off[8][3] = {{0, 0, 0}, {1, 0, 0}, {1, 1, 0}, {0, 1, 0},
                                      {0, 0, 1}, {1, 0, 1}, {1, 1, 1}, {0, 1, 1}};

__device__ __forceinline__ int tri_index(int i, int j) {  // packed lower triangle
  return i >= j ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i;
}

__device__ __forceinline__ int find_sub(const SubDev* subs, int n_sub, long long dof) {
  int lo = 0, hi = n_sub - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (subs[mid].dof_off <= dof) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// ---------------------------------------------------------------------------
// Element tables: physical shape-function gradients at the 8 Gauss points,
// the elastic brick stiffness and w detJ B_g^T E_eps B_g (eq. (K_def) pieces).
// ---------------------------------------------------------------------------
__global__ void k_tables(double h0, double h1, double h2, double lam, double mu, double* dN, double* Kel,
                         double* Qt) {
  __shared__ double B[8][6][24];
  __shared__ double dn[8][8][3];
  const double hh[3] = {h0, h1, h2};
  const double a = 1.0 / sqrt(3.0);
  const int t = threadIdx.x;
  if (t < 64 * 3) {
    const int g = t / 24, rem = t % 24, node = rem / 3, d = rem % 3;
    const double xi[3] = {(2 * (g & 1) - 1) * a, (2 * ((g >> 1) & 1) - 1) * a, (2 * ((g >> 2) & 1) - 1) * a};
    double v = (2 * c_local_off[node][d] - 1) / 8.0;
    for (int e = 0; e < 3; ++e)
      if (e != d) v *= 1.0 + (2 * c_local_off[node][e] - 1) * xi[e];
    dn[g][node][d] = v * (2.0 / hh[d]);
  }
  __syncthreads();
  for (int i = t; i < 8 * 8 * 3; i += blockDim.x) dN[i] = (&dn[0][0][0])[i];
  for (int i = t; i < 8 * 6 * 24; i += blockDim.x) (&B[0][0][0])[i] = 0.0;
  __syncthreads();
  if (t < 64) {
    const int g = t / 8, nd = t % 8;
    const double dx = dn[g][nd][0], dy = dn[g][nd][1], dz = dn[g][nd][2];
    const int c = 3 * nd;
    B[g][0][c] = dx;
    B[g][1][c + 1] = dy;
    B[g][2][c + 2] = dz;
    B[g][3][c] = dy;
    B[g][3][c + 1] = dx;
    B[g][4][c + 1] = dz;
    B[g][4][c + 2] = dy;
    B[g][5][c] = dz;
    B[g][5][c + 2] = dx;
  }
  __syncthreads();
  double C[6][6], E[6][6];
  for (int r = 0; r < 6; ++r)
    for (int s = 0; s < 6; ++s) {
      C[r][s] = 0.0;
      E[r][s] = 0.0;
    }
  for (int r = 0; r < 3; ++r) {
    for (int s = 0; s < 3; ++s) {
      C[r][s] = lam;
      E[r][s] = -1.0 / 3.0;
    }
    C[r][r] = lam + 2.0 * mu;
    C[3 + r][3 + r] = mu;
    E[r][r] = 2.0 / 3.0;
    E[3 + r][3 + r] = 0.5;
  }
  const double wdet = h0 * h1 * h2 / 8.0;
  for (int idx = t; idx < 9 * 576; idx += blockDim.x) {
    const int which = idx / 576, i = (idx % 576) / 24, j = idx % 24;
    double s = 0.0;
    if (which == 0) {
      for (int g = 0; g < 8; ++g)
        for (int r = 0; r < 6; ++r)
          for (int q = 0; q < 6; ++q) s += B[g][r][i] * C[r][q] * B[g][q][j];
      Kel[i * 24 + j] = wdet * s;
    } else {
      const int g = which - 1;
      for (int r = 0; r < 6; ++r)
        for (int q = 0; q < 6; ++q) s += B[g][r][i] * E[r][q] * B[g][q][j];
      if (j <= i) Qt[(size_t)g * kTri24 + tri_index(i, j)] = wdet * s;
    }
  }
}

// Assembled elastic stencils: for a node whose position along each axis of its box is low (an element on its
// high side only), inner or high (types 0, 1, 2 per axis, type tx + 3 ty + 9 tz) the 27 neighbour blocks
// Kst[type][neighbour (dx + 1) + 3 (dy + 1) + 9 (dz + 1)][3 a + c], the sum of Kel over the adjacent elements that
// hold both nodes.
__global__ void k_stencils(const double* __restrict__ Kel, double* Kst) {
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < 27 * 27 * 9; idx += gridDim.x * blockDim.x) {
    const int k = idx % 9, nbr = (idx / 9) % 27, type = idx / 243;
    const int t[3] = {type % 3, (type / 3) % 3, type / 9}, d[3] = {nbr % 3 - 1, (nbr / 3) % 3 - 1, nbr / 9 - 1};
    double s = 0.0;
    for (int o = 0; o < 8; ++o) {   // element on the low (bit set) or high side of the node along each axis
      int a = 0, b = 0;
      bool in = true;
      for (int x = 0; x < 3; ++x) {
        const int low = (o >> x) & 1, other = d[x] + low;   // local coordinates of the node (low) and the neighbour
        in = in && (low ? t[x] != 0 : t[x] != 2) && other >= 0 && other <= 1;
        a += low << x;
        b += other << x;
      }
      if (in) s += Kel[(3 * c_off2local[a] + k / 3) * 24 + 3 * c_off2local[b] + k % 3];
    }
    Kst[idx] = s;
  }
}

// ---------------------------------------------------------------------------
// Rigid-body modes of one subdomain shape: translations, rotations about the
// centroid, modified Gram-Schmidt (Sec. 4.2, orthonormal basis of Ker K_p).
// ---------------------------------------------------------------------------
__device__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    red[32] = s;
  }
  __syncthreads();
  return red[32];
}

__global__ void k_rigid(SubDev S, double h0, double h1, double h2, double* R) {
  __shared__ double red[33];
  const int n = S.n_dof;
  const double hh[3] = {h0, h1, h2};
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int node = i / 3, c = i % 3;
    const int li = node % S.nn[0], lj = (node / S.nn[0]) % S.nn[1], lk = node / (S.nn[0] * S.nn[1]);
    const double X[3] = {(li - 0.5 * S.dims[0]) * hh[0], (lj - 0.5 * S.dims[1]) * hh[1],
                         (lk - 0.5 * S.dims[2]) * hh[2]};
    double* row = R + (size_t)i * 6;
    row[0] = c == 0;
    row[1] = c == 1;
    row[2] = c == 2;
    // e_x x X = (0, -Xz, Xy); e_y x X = (Xz, 0, -Xx); e_z x X = (-Xy, Xx, 0)
    row[3] = c == 0 ? 0.0 : (c == 1 ? -X[2] : X[1]);
    row[4] = c == 0 ? X[2] : (c == 1 ? 0.0 : -X[0]);
    row[5] = c == 0 ? -X[1] : (c == 1 ? X[0] : 0.0);
  }
  __syncthreads();
  for (int j = 0; j < 6; ++j) {
    for (int q = 0; q < j; ++q) {
      double s = 0.0;
      for (int i = threadIdx.x; i < n; i += blockDim.x) s += R[(size_t)i * 6 + q] * R[(size_t)i * 6 + j];
      s = block_sum(s, red);
      for (int i = threadIdx.x; i < n; i += blockDim.x) R[(size_t)i * 6 + j] -= s * R[(size_t)i * 6 + q];
      __syncthreads();
    }
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += R[(size_t)i * 6 + j] * R[(size_t)i * 6 + j];
    s = block_sum(s, red);
    const double inv = 1.0 / sqrt(s);
    for (int i = threadIdx.x; i < n; i += blockDim.x) R[(size_t)i * 6 + j] *= inv;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Uniform traction on a face: t * area / 4 per element face and node.
// ---------------------------------------------------------------------------
__global__ void k_traction(DevMesh M, int face, int nel0, int nel1, int nel2, double t0, double t1, double t2,
                           double h0, double h1, double h2, double* f) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= M.n_dof) return;
  const int p = find_sub(M.subs, M.n_sub, i);
  const SubDev& S = M.subs[p];
  const int ld = (int)(i - S.dof_off);
  const int node = ld / 3, c = ld % 3;
  const int l[3] = {node % S.nn[0], (node / S.nn[0]) % S.nn[1], node / (S.nn[0] * S.nn[1])};
  const int axis = face / 2, side = face % 2;
  const int nel[3] = {nel0, nel1, nel2};
  const double hh[3] = {h0, h1, h2};
  double v = 0.0;
  const bool touches = side == 0 ? S.origin[axis] == 0 : S.origin[axis] + S.dims[axis] == nel[axis];
  const int lface = side == 0 ? 0 : S.dims[axis];
  if (touches && l[axis] == lface) {
    const int o1 = (axis + 1) % 3, o2 = (axis + 2) % 3;
    const int cnt = ((l[o1] > 0) + (l[o1] < S.dims[o1])) * ((l[o2] > 0) + (l[o2] < S.dims[o2]));
    const double tc = c == 0 ? t0 : (c == 1 ? t1 : t2);
    v = cnt * (tc * (hh[o1] * hh[o2]) / 4.0);
  }
  f[i] = v;
}

// ---------------------------------------------------------------------------
// Trilinear gradients by sum factorisation over the 8 lanes of an element (lane bits x + 2y + 4z
// give both the lane's Gauss point and the element node it loads).  An interpolation step takes the
// lane's own value with weight (1 + 1/sqrt 3)/2 and its partner's with (1 - 1/sqrt 3)/2 (the 2-point
// Gauss abscissae +-1/sqrt 3); as u + r u_partner with r = (1 - 1/sqrt 3)/(1 + 1/sqrt 3) it is one
// FMA, the factor ((1 + 1/sqrt 3)/2)^2 of two steps left to the caller (M.gs).
//
// The FP64 pipe (two lanes per SM and clock) bounds the Gauss-point kernels, so what is equal on two
// lanes is formed once: du/dx is the same at both x points of an element, so the lanes with x = 0
// carry component 0 through the x chain and the lanes with x = 1 component 1, and exchange the
// results; likewise y and z.  18 FP64 operations for the nine derivatives of a point where forming
// each on its own takes 39.
constexpr double kGr = 0.26794919243112270647;   // (1 - 1/sqrt 3) / (1 + 1/sqrt 3) = 2 - sqrt 3

// t[c][d] h_d-free derivative of component c along d at the lane's Gauss point: du_c/dx_d =
// M.gs[d] t[c][d].  u: the lane's node values.  All 32 lanes of the warp take part.
__device__ __forceinline__ void grad_lanes3(const double (&u)[3], int bx, int by, int bz, double (&t)[3][3]) {
  const unsigned all = 0xffffffffu;
  double up[3], I[3], Ip[3], J[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    up[c] = __shfl_xor_sync(all, u[c], 1);
    I[c] = fma(kGr, up[c], u[c]);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Ip[c] = __shfl_xor_sync(all, I[c], 2);
    J[c] = fma(kGr, Ip[c], I[c]);
  }
  // along x: differences on the x edges, interpolated in y and z
  double a = (bx ? u[1] : up[0]) - (bx ? up[1] : u[0]), b = (bx ? u[2] : up[2]) - (bx ? up[2] : u[2]);
  a = fma(kGr, __shfl_xor_sync(all, a, 2), a);
  b = fma(kGr, __shfl_xor_sync(all, b, 2), b);
  a = fma(kGr, __shfl_xor_sync(all, a, 4), a);
  t[2][0] = fma(kGr, __shfl_xor_sync(all, b, 4), b);
  double o = __shfl_xor_sync(all, a, 1);
  t[0][0] = bx ? o : a;
  t[1][0] = bx ? a : o;
  // along y: differences of the x interpolants, interpolated in z
  a = (by ? I[1] : Ip[0]) - (by ? Ip[1] : I[0]);
  b = (by ? I[2] : Ip[2]) - (by ? Ip[2] : I[2]);
  a = fma(kGr, __shfl_xor_sync(all, a, 4), a);
  t[2][1] = fma(kGr, __shfl_xor_sync(all, b, 4), b);
  o = __shfl_xor_sync(all, a, 2);
  t[0][1] = by ? o : a;
  t[1][1] = by ? a : o;
  // along z: differences of the x-y interpolants
  const double jo = __shfl_xor_sync(all, bz ? J[0] : J[1], 4), j2 = __shfl_xor_sync(all, J[2], 4);
  a = (bz ? J[1] : jo) - (bz ? jo : J[0]);
  t[2][2] = (bz ? J[2] : j2) - (bz ? j2 : J[2]);
  o = __shfl_xor_sync(all, a, 4);
  t[0][2] = bz ? o : a;
  t[1][2] = bz ? a : o;
}

// The transpose: given (fx, fy, fz) at the lane's Gauss point, returns at the lane's node
// h_x / ((1 + 1/sqrt 3) / 2)^2 times the sum over the element's points of grad N_node . (fx, fy, fz); ry = h_x / h_y,
// rz = h_x / h_z.  11 FP64 operations.
__device__ __forceinline__ double grad_lanes_t(double fx, double fy, double fz, int bx, int by, int bz, double ry,
                                               double rz) {
  const unsigned all = 0xffffffffu;
  const double xz = fma(kGr, __shfl_xor_sync(all, fx, 4), fx), yz = fma(kGr, __shfl_xor_sync(all, fy, 4), fy);
  const double zz = fz + __shfl_xor_sync(all, fz, 4);
  const double xy = fma(kGr, __shfl_xor_sync(all, xz, 2), xz);
  const double yy = yz + __shfl_xor_sync(all, yz, 2);
  const double zy = fma(kGr, __shfl_xor_sync(all, zz, 2), zz);
  // node signs of the differences: - at the low node, + at the high one
  const double i = fma(bz ? rz : -rz, zy, (by ? ry : -ry) * yy);
  const double xx = xy + __shfl_xor_sync(all, xy, 1);
  return fma(kGr, __shfl_xor_sync(all, i, 1), i) + (bx ? xx : -xx);
}

// ---------------------------------------------------------------------------
// Return mapping and Clarke derivative at one Gauss point.
// eta = B_g u_e; tau = sigma_k + C eta; Phi = sqrt(3/2)||dev tau|| - (sigma_y + H kappa_k).
// Phi <= 0: dsigma = C eta, dkappa = 0, D = C.
// Phi > 0 : dsigma = C eta - c sqrt(2/3) Phi n, dkappa = Phi/(3mu+H),
// A point returned to the yield surface has Phi = 0 in exact arithmetic (elastic by
// the rule above) but +-1 ulp after rounding: |Phi| <= kTie (sigma_y + H kappa_k)
// is read as that tie, i.e. elastic.
//           D = C - 2mu c (1 - rho) E_eps - 2mu c rho n n^T, rho = sqrt(2/3)(sigma_y+H kappa)/||dev tau||,
//           c = 3mu/(3mu+H)  (the Sec. 3.1 form of eq. (stress_op_deriv_plast)).
// ---------------------------------------------------------------------------
// Constants of the return mapping, formed once on the host: with s_d the factor of the derivatives
// along d (M.gs) the stress increment is ce = C eta, ce_dd = m2[d] t_dd + sum_k l[k] t_kk and
// ce_cd = m1[d] t_cd + m1[c] t_dc.
struct RmConst {
  double l[3], m2[3], m1[3];   // lam s_d, 2 mu s_d, mu s_d
  double cs, kd, a0;           // sqrt(2/3) c, 1 / (3 mu + H), 2 mu c, c = 3 mu / (3 mu + H)
};

// One thread per Gauss point, the 8 points of an element in 8 consecutive lanes (blockDim and n_gp
// multiples of 8); lanes past n_gp compute on the last element and store nothing.
// Bound by the FP64 pipe: about 52 operations per elastic point and, at a point past the test below, a square
// root, a division and 11 more (74 per elastic point, two further divisions and the derivatives formed one by one in
// the form before): at 96^3, half of the points yielding, 1028 us for 7.1 million points where that form took
// 1714.  The material constants come from the host.  kOut: 0 = increments only, 1 = also a, b, n, 2 = also T.
template <int kOut>
__global__ void __launch_bounds__(128) k_return_map(DevMesh M, RmConst K, const double* __restrict__ du,
                                                    const double* __restrict__ sig_k, const double* __restrict__ kap_k,
                                                    double* dsig, double* dkap, uint8_t* plastic, double* Dtan,
                                                    double* pa, double* pb, double* pn) {
  const long long gp_t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const bool live = gp_t < M.n_gp;
  const long long gp = live ? gp_t : M.n_gp - 8 + (gp_t & 7);
  const long long e = gp >> 3;
  const int g = (int)(gp & 7);
  const int bx = g & 1, by = (g >> 1) & 1, bz = (g >> 2) & 1;
  double tau[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) tau[c] = __ldg(sig_k + c * M.n_gp + gp);
  const double kap = __ldg(kap_k + gp);
  const int p = M.elem_sub[e];
  const SubDev& S = M.subs[p];
  const int le = (int)(e - S.elem_off);
  const int ex = le % S.dims[0], ey = (le / S.dims[0]) % S.dims[1], ez = le / (S.dims[0] * S.dims[1]);
  const int ln = (ex + bx) + S.nn[0] * ((ey + by) + S.nn[1] * (ez + bz));
  const double* un = du + S.dof_off + 3LL * ln;
  const double u[3] = {un[0], un[1], un[2]};
  double t[3][3];
  grad_lanes3(u, bx, by, bz, t);
  if (!live) return;
  const double lt = fma(K.l[2], t[2][2], fma(K.l[1], t[1][1], K.l[0] * t[0][0]));
  double ce[6];
  ce[0] = fma(K.m2[0], t[0][0], lt);
  ce[1] = fma(K.m2[1], t[1][1], lt);
  ce[2] = fma(K.m2[2], t[2][2], lt);
  ce[3] = fma(K.m1[1], t[0][1], K.m1[0] * t[1][0]);
  ce[4] = fma(K.m1[2], t[1][2], K.m1[1] * t[2][1]);
  ce[5] = fma(K.m1[2], t[0][2], K.m1[0] * t[2][0]);
#pragma unroll
  for (int c = 0; c < 6; ++c) tau[c] += ce[c];
  const double mean = (tau[0] + tau[1] + tau[2]) * kThird;
  const double dev[6] = {tau[0] - mean, tau[1] - mean, tau[2] - mean, tau[3], tau[4], tau[5]};
  const double nrm2 =
      dev[0] * dev[0] + dev[1] * dev[1] + dev[2] * dev[2] + 2.0 * (dev[3] * dev[3] + dev[4] * dev[4] + dev[5] * dev[5]);
  const double yield = fma(M.H, kap, M.sigma_y);
  // (3/2) |dev tau|^2 <= yield^2 puts Phi within rounding of <= 0, far inside the tie band: elastic
  // without the root (compared as integers: both are non-negative, and a NaN fails the test below)
  double phi = 0.0, inv = 0.0;
  bool pl = false;
  if (__double_as_longlong(1.5 * nrm2) > __double_as_longlong(yield * yield)) {
    const double nrm = sqrt(nrm2);
    inv = 1.0 / nrm;
    phi = fma(kSqrt32, nrm, -yield);
    pl = phi > kTie * yield;
  }
  const double f = pl ? K.cs * phi * inv : 0.0;   // dsigma = C eta - f dev tau
  if (pl) {
#pragma unroll
    for (int q = 0; q < 6; ++q) ce[q] = fma(-f, dev[q], ce[q]);
  }
#pragma unroll
  for (int q = 0; q < 6; ++q) dsig[q * M.n_gp + gp] = ce[q];
  if (dkap) dkap[gp] = pl ? K.kd * phi : 0.0;
  if (plastic) plastic[gp] = pl ? 1 : 0;
  if constexpr (kOut > 0) {
    double a = 0.0, b = 0.0, nb[6] = {0, 0, 0, 0, 0, 0};
    if (pl) {
      b = K.a0 * (kSqrt23 * yield * inv);   // 2 mu c rho
      a = K.a0 - b;
#pragma unroll
      for (int q = 0; q < 6; ++q) nb[q] = dev[q] * inv;
    }
    if (pa) {
      pa[gp] = a;
      pb[gp] = b;
#pragma unroll
      for (int q = 0; q < 6; ++q) pn[q * M.n_gp + gp] = nb[q];
    }
    if constexpr (kOut == 2) {
      const double c11 = M.lam + 2.0 * M.mu;   // uniform over the launch
      const double d11 = pl ? fma(-2.0 / 3.0, a, c11) : c11, d12 = pl ? fma(1.0 / 3.0, a, M.lam) : M.lam,
                   d44 = pl ? fma(-0.5, a, M.mu) : M.mu;
      int idx = 0;
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        const double br = pl ? -b * nb[r] : 0.0;
#pragma unroll
        for (int s = r; s < 6; ++s, ++idx) {
          const double base = (r < 3 && s < 3) ? (r == s ? d11 : d12) : (r == s ? d44 : 0.0);
          Dtan[idx * M.n_gp + gp] = pl ? fma(br, nb[s], base) : base;
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Element tangent correction dK_e = sum_{plastic g} (a_g Q_g + w detJ b_g v_g v_g^T),
// v_g = B_g^T n_g.  K_e = K_el - dK_e.  A warp looks through four elements (lane = 8 element + point)
// and works on the ones with plastic points together: two FMAs per point and entry of the packed lower
// triangle, bound by the FP64 pipe (4800 of them for an element that yields everywhere).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_elem_correction(DevMesh M, GPData gd, int* elem_np, int* sub_np, double* dKe) {
  __shared__ double v[8][8][24], bv[8][8][24];  // [warp][g][i]: v_g and w detJ b_g v_g
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long e0 = 4 * (blockIdx.x * (long long)(blockDim.x >> 5) + warp);
  if (e0 >= M.n_elem) return;
  const int flag = e0 + (lane >> 3) < M.n_elem ? gd.plastic[e0 * 8 + lane] : 0;
  const unsigned all = __ballot_sync(0xffffffffu, flag != 0);
  if ((lane & 7) == 0 && e0 + (lane >> 3) < M.n_elem) {
    const int cnt = __popc((all >> lane) & 0xffu);
    elem_np[e0 + (lane >> 3)] = cnt;
    if (cnt) atomicAdd(&sub_np[M.elem_sub[e0 + (lane >> 3)]], cnt);
  }
  for (int k = 0; k < 4; ++k) {
    const unsigned mask = (all >> (8 * k)) & 0xffu;
    if (!mask) continue;
    const long long gp0 = (e0 + k) * 8;
    __syncwarp();
    // lane = point + 8 x node pair: B_g^T n_g at nodes 2 (lane / 8), 2 (lane / 8) + 1
    if ((mask >> (lane & 7)) & 1u) {
      const int g = lane & 7;
      const long long gp = gp0 + g;
      const double wb = M.wdet * gd.pb[gp];
      double n[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) n[q] = gd.pn[q * M.n_gp + gp];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int a = 2 * (lane >> 3) + h;
        const double* dn = M.dN + g * 24 + 3 * a;
        const double dx = dn[0], dy = dn[1], dz = dn[2];
        const double w[3] = {dx * n[0] + dy * n[3] + dz * n[5], dy * n[1] + dx * n[3] + dz * n[4],
                             dz * n[2] + dy * n[4] + dx * n[5]};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          v[warp][g][3 * a + c] = w[c];
          bv[warp][g][3 * a + c] = wb * w[c];
        }
      }
    }
    __syncwarp();
    double ag[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) ag[g] = (mask >> g) & 1u ? gd.pa[gp0 + g] : 0.0;
    for (int idx = lane; idx < kTri24; idx += 32) {
      int i = (int)((sqrtf(8.0f * (float)idx + 1.0f) - 1.0f) * 0.5f);
      while (i * (i + 1) / 2 > idx) --i;
      while ((i + 1) * (i + 2) / 2 <= idx) ++i;
      const int j = idx - i * (i + 1) / 2;
      double s = 0.0;
#pragma unroll
      for (int g = 0; g < 8; ++g)
        if ((mask >> g) & 1u) s = fma(bv[warp][g][i], v[warp][g][j], fma(ag[g], __ldg(M.Qt + g * kTri24 + idx), s));
      dKe[(e0 + k) * kTri24 + idx] = s;
    }
  }
}

// Stencil type of the node at (i, j, k) of a box with nn nodes per axis (see k_stencils).
__device__ __forceinline__ int node_type(const SubDev& S, int i, int j, int k) {
  return (i == 0 ? 0 : (i == S.nn[0] - 1 ? 2 : 1)) + 3 * (j == 0 ? 0 : (j == S.nn[1] - 1 ? 2 : 1)) +
         9 * (k == 0 ? 0 : (k == S.nn[2] - 1 ? 2 : 1));
}

// K entry (true tangent) between component a of node r and component c of its neighbour r + d (inside the box):
// the elastic stencil less the corrections of the elements with plastic points that hold both nodes.
__device__ double stiffness_entry(const DevMesh& M, const SubDev& S, const int* elem_np, const double* dKe,
                                  const int (&r)[3], const int (&d)[3], int a, int c, bool elastic_only) {
  double sum = __ldg(M.Kst + (node_type(S, r[0], r[1], r[2]) * 27 + (d[0] + 1) + 3 * (d[1] + 1) + 9 * (d[2] + 1)) * 9 +
                     3 * a + c);
  if (elastic_only) return sum;
  int lo[3], hi[3];
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    lo[x] = max(max(r[x], r[x] + d[x]) - 1, 0);
    hi[x] = min(min(r[x], r[x] + d[x]), S.dims[x] - 1);
  }
  for (int ez = lo[2]; ez <= hi[2]; ++ez)
    for (int ey = lo[1]; ey <= hi[1]; ++ey)
      for (int ex = lo[0]; ex <= hi[0]; ++ex) {
        const long long ge = S.elem_off + ex + S.dims[0] * (ey + S.dims[1] * ez);
        if (!elem_np[ge]) continue;
        const int na = c_off2local[(r[0] - ex) + 2 * (r[1] - ey) + 4 * (r[2] - ez)];
        const int nc = c_off2local[(r[0] + d[0] - ex) + 2 * (r[1] + d[1] - ey) + 4 * (r[2] + d[2] - ez)];
        sum -= dKe[ge * kTri24 + tri_index(3 * na + a, 3 * nc + c)];
      }
  return sum;
}

// Band storage of subdomain K_p with the fixing dofs replaced by identity rows:
// band[r*(bw+1) + k] = K[r][r - bw + k] (lower band, row-major).
// interior = 0: the six fixing dofs of Remark 1 get identity rows and columns (K_rr of the generalised
// inverse); interior = 1: the descriptors' node boxes are the nodes without constraint rows and the band is
// K_ii of the Dirichlet preconditioner (Sec. 4.2), numbered within that box.  The band is cleared first;
// then one thread per (node, neighbour not after it, component pair) writes the stencil's entries: 126
// per node instead of an index decode for every of the 3 (bw + 1) band entries.
__global__ void k_band_clear(DevMesh M, const int* __restrict__ sub_list, double* band,
                             const long long* __restrict__ band_off_list) {
  const SubDev& S = M.subs[sub_list[blockIdx.y]];
  double* b = band + band_off_list[blockIdx.y];
  const long long total = (long long)S.n_dof * (S.bw + 1);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
    b[i] = 0.0;
}

__global__ void k_band_fill(DevMesh M, const int* __restrict__ sub_list, const int* elem_np, const double* dKe,
                            double* band, const long long* __restrict__ band_off_list, int elastic_only,
                            int interior) {
  const int item = blockIdx.y;
  const int p = sub_list[item];
  const SubDev& S = M.subs[p];
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int node = idx / 126, m = (idx / 9) % 14, k = idx % 9;   // neighbours 0..13: those not after the node
  if (node >= S.n_dof / 3) return;
  const int r[3] = {S.ilo[0] + node % S.inn[0], S.ilo[1] + (node / S.inn[0]) % S.inn[1],
                    S.ilo[2] + node / (S.inn[0] * S.inn[1])};
  const int d[3] = {m % 3 - 1, (m / 3) % 3 - 1, m / 9 - 1};
#pragma unroll
  for (int x = 0; x < 3; ++x)
    if (r[x] + d[x] < S.ilo[x] || r[x] + d[x] >= S.ilo[x] + S.inn[x]) return;
  const int row = 3 * node + k / 3, col = 3 * (node + d[0] + S.inn[0] * (d[1] + S.inn[1] * d[2])) + k % 3;
  if (col > row) return;
  bool fixed = false;
  if (!interior) {
#pragma unroll
    for (int t = 0; t < 6; ++t) fixed |= (S.fix[t] == row) | (S.fix[t] == col);
  }
  if (fixed && row != col) return;
  band[band_off_list[item] + (long long)row * (S.bw + 1) + S.bw - (row - col)] =
      fixed ? 1.0 : stiffness_entry(M, S, elem_np, dKe, r, d, k / 3, k % 3, elastic_only != 0);
}

// Lumped-preconditioner blocks of one subdomain (or its shape's elastic template):
// K[3 ln(b) + a][3 ln(nu) + c] for every box-boundary node b and its 27 stencil neighbours nu.
__global__ void k_kbb_fill(DevMesh M, const int* __restrict__ sub_list, const long long* __restrict__ dst_off,
                           const int* elem_np, const double* dKe, double* kbb, float* kbb32, int elastic_only) {
  const int p = sub_list[blockIdx.y];
  const SubDev& S = M.subs[p];
  const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (idx >= (long long)S.n_bnd * 243) return;
  // layout [t][cc][3 b + a]: for a fixed neighbour t and column cc the rows of all boundary
  // nodes are contiguous, so the lumped kernel's threads (consecutive rows) read coalesced
  const long long nr = 3LL * S.n_bnd;
  const int tc = (int)(idx / nr), ra = (int)(idx % nr);
  const int t = tc / 3, cc = tc % 3, b = ra / 3, a = ra % 3;
  const int nu = M.shape_tnbr[(S.bnd_off + b) * 27 + t];
  double v = 0.0;
  if (nu >= 0) {
    const int nr_ = M.shape_bln[S.bnd_off + b], nc = M.shape_bln[S.bnd_off + nu];
    const int r[3] = {nr_ % S.nn[0], (nr_ / S.nn[0]) % S.nn[1], nr_ / (S.nn[0] * S.nn[1])};
    const int d[3] = {nc % S.nn[0] - r[0], (nc / S.nn[0]) % S.nn[1] - r[1], nc / (S.nn[0] * S.nn[1]) - r[2]};
    v = stiffness_entry(M, S, elem_np, dKe, r, d, a, cc, elastic_only != 0);
  }
  kbb[dst_off[blockIdx.y] + idx] = v;
  if (kbb32) kbb32[dst_off[blockIdx.y] + idx] = (float)v;
}

// Internal force of eq. (F_def), element part: for every element node a (bit order x + 2y + 4z)
// and component c, fe = h_x / ((1 + 1/sqrt 3) / 2)^2 sum over the element's Gauss points of grad N_a . sigma_c (sigma_c
// the row c of the stress dsig), by the transposed sum factorisation over the element's 8 lanes (33
// FP64 operations per point; the factor is applied per dof by k_gather_force).
__global__ void k_elem_force(DevMesh M, const double* __restrict__ dsig, double* fe) {
  const long long gp_t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const bool live = gp_t < M.n_gp;
  const long long gp = live ? gp_t : M.n_gp - 8 + (gp_t & 7);
  const int g = (int)(gp & 7);
  const int bx = g & 1, by = (g >> 1) & 1, bz = (g >> 2) & 1;
  double sg[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) sg[q] = dsig[q * M.n_gp + gp];
  // Voigt order xx, yy, zz, xy, yz, xz
  const double f0 = grad_lanes_t(sg[0], sg[3], sg[5], bx, by, bz, M.gratio[1], M.gratio[2]);
  const double f1 = grad_lanes_t(sg[3], sg[1], sg[4], bx, by, bz, M.gratio[1], M.gratio[2]);
  const double f2 = grad_lanes_t(sg[5], sg[4], sg[2], bx, by, bz, M.gratio[1], M.gratio[2]);
  if (!live) return;
  double* o = fe + 3 * gp;   // element e = gp / 8, node g
  o[0] = f0;
  o[1] = f1;
  o[2] = f2;
}

// f = df - w detJ M.gs[0] (sum of the element parts at the dof), the adjacent elements in (z, y, x) order.
__global__ void k_gather_force(DevMesh M, const double* __restrict__ fe, const double* __restrict__ df, double* f) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= M.n_dof) return;
  const int p = find_sub(M.subs, M.n_sub, i);
  const SubDev& S = M.subs[p];
  const int ld = (int)(i - S.dof_off);
  const int node = ld / 3, c = ld % 3;
  const int li = node % S.nn[0], lj = (node / S.nn[0]) % S.nn[1], lk = node / (S.nn[0] * S.nn[1]);
  double s = 0.0;
  for (int ez = max(lk - 1, 0); ez <= min(lk, S.dims[2] - 1); ++ez)
    for (int ey = max(lj - 1, 0); ey <= min(lj, S.dims[1] - 1); ++ey)
      for (int ex = max(li - 1, 0); ex <= min(li, S.dims[0] - 1); ++ex) {
        const int a = (li - ex) + 2 * (lj - ey) + 4 * (lk - ez);
        const long long ge = S.elem_off + ex + S.dims[0] * (ey + S.dims[1] * ez);
        s += fe[(ge * 8 + a) * 3 + c];
      }
  f[i] = (df ? df[i] : 0.0) - M.wgs * s;
}

// y = K x per subdomain with the assembled tangent, one thread per dof: the elastic 27-node stencil of the
// node's type (81 FMAs, bound by the FP64 pipe and the loads' latency; the coefficients, mostly the same for
// a warp, come from L1), less the corrections of the adjacent elements with plastic points.
__global__ void __launch_bounds__(192) k_apply_K(DevMesh M, const int* __restrict__ elem_np,
                                                 const double* __restrict__ dKe, const double* __restrict__ x,
                                                 double* y) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= M.n_dof) return;
  const int p = find_sub(M.subs, M.n_sub, i);
  const SubDev& S = M.subs[p];
  const int n0 = S.nn[0], n1 = S.nn[1];
  const int dof = (int)(i - S.dof_off), node = dof / 3, r = dof % 3;
  const int li = node % n0, lj = (node / n0) % n1, lk = node / (n0 * n1);
  const double* xs = x + S.dof_off;
  const double* kt = M.Kst + node_type(S, li, lj, lk) * 243 + 3 * r;
  double s = 0.0;
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz) {
    double v[9][3], k[9][3];   // a plane of neighbours: loads issued together
    bool in[9];
#pragma unroll
    for (int m = 0; m < 9; ++m) {
      const int a = li + m % 3 - 1, b = lj + m / 3 - 1, c = lk + dz;
      in[m] = a >= 0 && a < n0 && b >= 0 && b < n1 && c >= 0 && c < S.nn[2];
      const double* xn = xs + 3 * (in[m] ? a + n0 * (b + n1 * c) : node);
      const double* kb = kt + (m + 9 * (dz + 1)) * 9;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        v[m][q] = __ldg(xn + q);
        k[m][q] = __ldg(kb + q);
      }
    }
#pragma unroll
    for (int m = 0; m < 9; ++m)
      if (in[m])
#pragma unroll
        for (int q = 0; q < 3; ++q) s = fma(k[m][q], v[m][q], s);
  }
  for (int ez = max(lk - 1, 0); ez <= min(lk, S.dims[2] - 1); ++ez)
    for (int ey = max(lj - 1, 0); ey <= min(lj, S.dims[1] - 1); ++ey)
      for (int ex = max(li - 1, 0); ex <= min(li, S.dims[0] - 1); ++ex) {
        const long long ge = S.elem_off + ex + S.dims[0] * (ey + S.dims[1] * ez);
        if (!elem_np[ge]) continue;
        const double* dk = dKe + ge * kTri24;
        const int row = 3 * c_off2local[(li - ex) + 2 * (lj - ey) + 4 * (lk - ez)] + r;
        double c = 0.0;
#pragma unroll
        for (int o = 0; o < 8; ++o) {
          const int nb = c_off2local[o];
          const double* xn = xs + 3 * (ex + (o & 1) + n0 * (ey + ((o >> 1) & 1) + n1 * (ez + (o >> 2))));
#pragma unroll
          for (int q = 0; q < 3; ++q) c = fma(__ldg(dk + tri_index(row, 3 * nb + q)), __ldg(xn + q), c);
        }
        s -= c;
      }
  y[i] = s;
}

__global__ void k_commit(long long n_dof, long long n_gp, const double* du, const double* dsig,
                         const double* dkap, double* u, double* sig, double* kap) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n_dof) u[i] += du[i];
  if (i < 6 * n_gp) sig[i] += dsig[i];
  if (i < n_gp) kap[i] += dkap[i];
}

__global__ void k_vm_partial(long long n_gp, const double* __restrict__ s, double* partial) {
  __shared__ double red[256];
  double m = 0.0;
  for (long long gp = blockIdx.x * (long long)blockDim.x + threadIdx.x; gp < n_gp;
       gp += (long long)gridDim.x * blockDim.x) {
    const double t0 = s[gp], t1 = s[n_gp + gp], t2 = s[2 * n_gp + gp];
    const double mean = (t0 + t1 + t2) / 3.0;
    const double d0 = t0 - mean, d1 = t1 - mean, d2 = t2 - mean;
    const double t3 = s[3 * n_gp + gp], t4 = s[4 * n_gp + gp], t5 = s[5 * n_gp + gp];
    const double q = kSqrt32 * sqrt(d0 * d0 + d1 * d1 + d2 * d2 + 2.0 * (t3 * t3 + t4 * t4 + t5 * t5));
    m = fmax(m, q);
  }
  red[threadIdx.x] = m;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + o]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void k_max_final(const double* partial, int n, double* out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double m = 0.0;
    for (int i = 0; i < n; ++i) m = fmax(m, partial[i]);
    *out = m;
  }
}

inline unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

void launch_tables(const double* h, double lam, double mu, double* dN, double* Kel, double* Qt, double* Kst,
                   cudaStream_t st) {
  k_tables<<<1, 256, 0, st>>>(h[0], h[1], h[2], lam, mu, dN, Kel, Qt);
  k_stencils<<<27, 256, 0, st>>>(Kel, Kst);
}

void launch_rigid_for_shape(const SubDev& S, const double* h, double* R_shape, cudaStream_t st) {
  k_rigid<<<1, 256, 0, st>>>(S, h[0], h[1], h[2], R_shape);
}

void launch_traction(const DevMesh& M, int face, const int* nel, const double* t, const double* h, double* f,
                     cudaStream_t st) {
  k_traction<<<blocks_for(M.n_dof, 256), 256, 0, st>>>(M, face, nel[0], nel[1], nel[2], t[0], t[1], t[2], h[0],
                                                          h[1], h[2], f);
}

void launch_return_map(const DevMesh& M, const double* du, const double* sig_k, const double* kap_k,
                       double* dsig, double* dkap, uint8_t* plastic, double* Dtan, double* pa, double* pb,
                       double* pn, cudaStream_t st) {
  RmConst K;
  for (int d = 0; d < 3; ++d) {
    K.l[d] = M.lam * M.gs[d];
    K.m2[d] = 2.0 * M.mu * M.gs[d];
    K.m1[d] = M.mu * M.gs[d];
  }
  const double c = 3.0 * M.mu / (3.0 * M.mu + M.H);
  K.cs = kSqrt23 * c;
  K.kd = 1.0 / (3.0 * M.mu + M.H);
  K.a0 = 2.0 * M.mu * c;
  const unsigned nblk = blocks_for(M.n_gp, 128);
  if (Dtan) k_return_map<2><<<nblk, 128, 0, st>>>(M, K, du, sig_k, kap_k, dsig, dkap, plastic, Dtan, pa, pb, pn);
  else if (pa) k_return_map<1><<<nblk, 128, 0, st>>>(M, K, du, sig_k, kap_k, dsig, dkap, plastic, Dtan, pa, pb, pn);
  else k_return_map<0><<<nblk, 128, 0, st>>>(M, K, du, sig_k, kap_k, dsig, dkap, plastic, Dtan, pa, pb, pn);
}

void launch_elem_correction(const DevMesh& M, GPData gp, int* elem_np, int* sub_np, double* dKe, cudaStream_t st) {
  k_elem_correction<<<blocks_for(M.n_elem, 32), 256, 0, st>>>(M, gp, elem_np, sub_np, dKe);
}

void launch_band_fill(const DevMesh& M, const int* sub_list, int n_list, const int* elem_np, const double* dKe,
                      double* band, const long long* band_off_list, int elastic_only, int max_rows, int max_bw,
                      cudaStream_t st, bool interior) {
  if (n_list <= 0) return;
  k_band_clear<<<dim3(blocks_for((long long)max_rows * (max_bw + 1), 256 * 16), n_list), 256, 0, st>>>(M, sub_list, band,
                                                                                                band_off_list);
  dim3 grid(blocks_for((long long)max_rows / 3 * 126, 256), n_list);
  k_band_fill<<<grid, 256, 0, st>>>(M, sub_list, elem_np, dKe, band, band_off_list, elastic_only,
                                       interior ? 1 : 0);
}

void launch_kbb_fill(const DevMesh& M, const int* sub_list, const long long* dst_off, int n_list, int max_bnd,
                     const int* elem_np, const double* dKe, double* kbb, float* kbb32, int elastic_only,
                     cudaStream_t st) {
  if (n_list <= 0) return;
  dim3 grid(blocks_for((long long)max_bnd * 243, 256), n_list);
  k_kbb_fill<<<grid, 256, 0, st>>>(M, sub_list, dst_off, elem_np, dKe, kbb, kbb32, elastic_only);
}

void launch_internal_force(const DevMesh& M, const double* dsig, const double* df, double* fe, double* f,
                           cudaStream_t st) {
  if (M.n_gp > 0) k_elem_force<<<blocks_for(M.n_gp, 128), 128, 0, st>>>(M, dsig, fe);
  k_gather_force<<<blocks_for(M.n_dof, 128), 128, 0, st>>>(M, fe, df, f);
}

void launch_apply_K(const DevMesh& M, const int* elem_np, const double* dKe, const double* x, double* y,
                    cudaStream_t st) {
  k_apply_K<<<blocks_for(M.n_dof, 192), 192, 0, st>>>(M, elem_np, dKe, x, y);
}

void launch_commit(const DevMesh& M, const double* du, const double* dsig, const double* dkap, double* u,
                   double* sig, double* kap, cudaStream_t st) {
  const long long n = 6 * M.n_gp > M.n_dof ? 6 * M.n_gp : M.n_dof;
  k_commit<<<blocks_for(n, 256), 256, 0, st>>>(M.n_dof, M.n_gp, du, dsig, dkap, u, sig, kap);
}

void launch_vm_max(const DevMesh& M, const double* dsig, double* partial, double* out, cudaStream_t st) {
  k_vm_partial<<<kRedBlocks, 256, 0, st>>>(M.n_gp, dsig, partial);
  k_max_final<<<1, 32, 0, st>>>(partial, kRedBlocks, out);
}

}  // namespace tfeti
