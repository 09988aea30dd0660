// Fermion, clover and gauge forces (App. C), accumulated in FP64 as algebra coefficients
// f[p][mu][a][cb] = dS/d omega_a for U_mu(x) -> exp(i omega_a T_a) U_mu(x).
//
// The fermion forces of App. C are sums of contractions Re[eta^dag (dK/dU) chi].  With
// K = M-hat^dag M-hat:
//   Re eta^dag dK chi = Re (M-hat chi)^dag dM-hat eta + Re (M-hat eta)^dag dM-hat chi,
// and with M-hat = A_ee - kappa^2 H_eo A_oo^{-1} H_oe,
//   a^dag dM-hat b = a^dag dA_ee b - kappa^2 [a^dag dH_eo y + w^dag dH_oe b - w^dag dA_oo y],
//   y = A_oo^{-1} H_oe b,  w = A_oo^{-1} H^dag_oe a.
// Hop terms: for a link U_mu(z) the forward term a(z)^dag (1 - g_mu) dU b(z+mu) and the
// backward term a(z+mu)^dag (1 + g_mu) dU^dag b(z) give, with dU = i w T U,
//   d/dw_a = i tr(T_a Z),  Z = sum_s (U R_f)_s ((1 - g_mu) L_f)_s^dag - sum_s R_b,s (U (1 + g_mu) L_b)_s^dag.
// Clover terms: a^dag (sigma (x) dF) b = tr_c(dF G), G = sum_{s s'} sigma_{s s'} b_s' a_s^dag;
// with F = traceless part of (Q - Q^dag)/(8i),
//   Re tr(dF G) = (1/8) Im tr(dQ H),  H = G~ + G~^dag (G~ traceless),
// so each site keeps one Hermitian traceless H per plane (8 reals) summed over every
// term, and one final kernel differentiates the clover leaves: for U_mu(z) in the plane
// (mu, nu) with corners z, z+mu, z+mu+nu, z+nu (above) and z-nu, z-nu+mu (below),
//   d/dw_a = (1/8) Re tr(T_a [U X_above - Y_below U^dag]),
//   X_above = H(z+mu) V1 V2 V3 + V1 H(z+mu+nu) V2 V3 + V1 V2 H(z+nu) V3 + V1 V2 V3 H(z),
//   Y_below = H(z) W1 W2 W3 + W1 H(z-nu) W2 W3 + W1 W2 H(z-nu+mu) W3 + W1 W2 W3 H(z+mu),
//   V1 = U_nu(z+mu), V2 = U_mu(z+nu)^dag, V3 = U_nu(z)^dag,
//   W1 = U_nu(z-nu)^dag, W2 = U_mu(z-nu), W3 = U_nu(z-nu+mu).
// Gauge force (Wilson action, beta/3 normalisation): d/dw_a = (beta/3) Im tr(T_a U S),
// S the sum of the six staples.
//
// The projectors satisfy P P = 2 P, so the spin sums above need only the two components of
// the half spinors: sum_s R_s (P L)_s^dag = sum_{k = 0, 1} (P R)_k (P L)_k^dag.  The four
// insertions of a clover leaf pair up along the links that connect them, with
//   D_nu(x) = H(x) U_nu(x) + U_nu(x) H(x+nu)   (H of the plane (mu, nu))
// computed once per site and (nu, mu) and used by four leaves:
//   X_above = D(z+mu) [U_nu(z) U_mu(z+nu)]^dag + U_nu(z+mu) [D(z) U_mu(z+nu)]^dag,
//   Y_below = D(z-nu)^dag [U_mu(z-nu) U_nu(z-nu+mu)] + U_nu(z-nu)^dag [U_mu(z-nu) D(z-nu+mu)],
// four matrix products per leaf where running prefixes took ten.
#include <algorithm>
#include <cmath>

#include "context.h"
#include "fields.cuh"
#include "hop_tile.cuh"
#include "mad.cuh"
#include "spin.cuh"

namespace pfmp {

constexpr double kInvSqrt3 = 0.57735026918962576451;

// c_a = tr(lambda_a M), a = 1..8 (complex)
template <typename T>
__device__ __forceinline__ void tr_lambda(const Mat3<T>& M, cplx<T> t[8]) {
  t[0] = M.m[1][0] + M.m[0][1];
  t[1] = times_i(M.m[0][1] - M.m[1][0]);
  t[2] = M.m[0][0] - M.m[1][1];
  t[3] = M.m[2][0] + M.m[0][2];
  t[4] = times_i(M.m[0][2] - M.m[2][0]);
  t[5] = M.m[2][1] + M.m[1][2];
  t[6] = times_i(M.m[1][2] - M.m[2][1]);
  t[7] = (T)kInvSqrt3 * (M.m[0][0] + M.m[1][1] - (T)2 * M.m[2][2]);
}

// H = sum_a h_a T_a (Hermitian traceless), in the arithmetic of T
template <typename T>
__device__ __forceinline__ Mat3<T> from_algebra(const T h[8]) {
  Mat3<T> H;
  const T s = (T)0.5, r3 = (T)kInvSqrt3;
  H.m[0][0] = mk<T>(s * (h[2] + r3 * h[7]), 0);
  H.m[1][1] = mk<T>(s * (-h[2] + r3 * h[7]), 0);
  H.m[2][2] = mk<T>(s * ((T)-2 * r3 * h[7]), 0);
  H.m[0][1] = mk<T>(s * h[0], -s * h[1]);
  H.m[1][0] = mk<T>(s * h[0], s * h[1]);
  H.m[0][2] = mk<T>(s * h[3], -s * h[4]);
  H.m[2][0] = mk<T>(s * h[3], s * h[4]);
  H.m[1][2] = mk<T>(s * h[5], -s * h[6]);
  H.m[2][1] = mk<T>(s * h[5], s * h[6]);
  return H;
}

// the link U_mu(x) at full coordinates: FP64 from the master field, FP32 from the
// 12-real compressed copy (third row rebuilt)
template <typename T>
__device__ __forceinline__ Mat3<T> glink(const void* gauge, const Geom& g, const int x[4], int mu);

__device__ __forceinline__ Mat3<double> mlink(const double2* U, const Geom& g, const int x[4], int mu) {
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  Mat3<double> M;
  load_link18(M, U + (size_t)((p * 4 + mu) * 9) * g.Vh, cb_index(g, x), g.Vh);
  return M;
}
template <>
__device__ __forceinline__ Mat3<double> glink<double>(const void* gauge, const Geom& g, const int x[4], int mu) {
  return mlink((const double2*)gauge, g, x, mu);
}
template <>
__device__ __forceinline__ Mat3<float> glink<float>(const void* gauge, const Geom& g, const int x[4], int mu) {
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  Mat3<float> M;
  load_link(M, link_plane<PFMP_F32>((const float4*)gauge, p * 4 + mu, g.Vh), cb_index(g, x), g.Vh);
  return M;
}
// y = x + d mu-hat (d = +-1), periodic, for a run-time mu (static indexing only)
__device__ __forceinline__ void shift_rt(const Geom& g, const int x[4], int mu, int d, int y[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int v = x[k] + (k == mu ? d : 0);
    y[k] = v == g.L[k] ? 0 : (v < 0 ? g.L[k] - 1 : v);
  }
}

__device__ __forceinline__ double* fptr(double* F, const Geom& g, int p, int mu, int a) {
  return F + (size_t)((p * 4 + mu) * 8 + a) * g.Vh;
}

// the link U_MU(z) of the force kernels: FP64 from the master field, FP32 from the
// 12-real compressed copy (third row rebuilt)
template <int PREC>
__device__ __forceinline__ Mat3<typename Prec<PREC>::real> force_link(const void* gauge, const Geom& g, int pz, int cb,
                                                                      const int z[4], int mu) {
  if constexpr (PREC == PFMP_F64) {
    return mlink((const double2*)gauge, g, z, mu);
  } else {
    Mat3<float> U;
    load_link(U, link_plane<PFMP_F32>((const float4*)gauge, pz * 4 + mu, g.Vh), cb, g.Vh);
    return U;
  }
}

// the spinor at site cb of a field that the kernels before this one wrote
__device__ __forceinline__ void load_spinor_live(Spinor<float>& s, const float4* f, int cb, int Vh) {
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float4 v = ld_live(f + (size_t)k * Vh + cb);
    s.s[(2 * k) / 3][(2 * k) % 3] = mk(v.x, v.y);
    s.s[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk(v.z, v.w);
  }
}
__device__ __forceinline__ void load_spinor_live(Spinor<double>& s, const double2* f, int cb, int Vh) {
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const double2 v = ld_live(f + (size_t)k * Vh + cb);
    s.s[k / 3][k % 3] = mk(v.x, v.y);
  }
}

// Spinor products in the arithmetic of PREC (FP64, or FP32 for the MD forces, whose
// value only has to be a deterministic function of the gauge field).  On the sites of
// parity pz the forward and backward fields of a contraction (a, b, y, w) are
// (L_f, R_f, L_b, R_b) = (a, y, w, b) for pz = 0 and (w, b, a, y) for pz = 1.  The link
// factors out of the batch's sum:
//   sum_k c_k Z_k = U X_f - X_b U^dag,  X_f = sum_k c_k (P- R_f)_k (P- L_f)_k^dag,
//                                       X_b = sum_k c_k (P+ R_b)_k (P+ L_b)_k^dag,
// with P-+ = 1 -+ g_mu, so each contraction costs two outer products of half spinors,
// accumulated in PREC, and the FP64 force is read and written once per batch.  A batch whose
// contractions share one coefficient (the filter and correction forces) has it applied to
// the sum.

// X += sum_k u_k v_k^dag
template <typename T>
__device__ __forceinline__ void outer_half(Mat3<T>& X, const Half<T>& u, const Half<T>& v) {
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) X.m[i][j] = cmad_nj(u.h[k][i], v.h[k][j], X.m[i][j]);
}

// F_mu(z) += c Im tr(lambda_a [U X_f - X_b U^dag]), from X_f and X_b of one link
template <typename T>
__device__ __forceinline__ void hop_force_store(double* F, const Geom& g, int pz, int mu, int cb, const Mat3<T>& U,
                                                const Mat3<T>& Xf, const Mat3<T>& Xb, double c) {
  Mat3<T> Z = mm(U, Xf), N;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) N.m[i][j] = -Xb.m[i][j];
  mac_nd(Z, N, U);
  cplx<T> t[8];
  tr_lambda(Z, t);
#pragma unroll
  for (int a = 0; a < 8; ++a) fptr(F, g, pz, mu, a)[cb] += c * (double)t[a].im;
}

// Re(i tr(T_a Z)) = -Im tr(T_a Z) = -(1/2) Im tr(lambda_a Z), with the boundary factor of the
// link and the coefficient shared by the batch
__device__ __forceinline__ double hop_force_factor(const Geom& g, const int z[4], int mu, const DerivBatch& B) {
  return ((mu == 3 && z[3] == g.L[3] - 1) ? -0.5 * g.bc_t : -0.5) * B.c_common;
}

template <int PREC, int MU>
__device__ __forceinline__ void hop_force_dir(double* F, const void* gauge, const Geom& g, int pz, int cb, const int z[4],
                                              const DerivBatch& B) {
  using T = typename Prec<PREC>::real;
  using V = typename Prec<PREC>::vec;
  const int n = nbr_cb(g, z, MU, +1);
  Mat3<T> Xf = mat_zero<T>(), Xb = mat_zero<T>();
#pragma unroll 1
  for (int k = 0; k < B.n; ++k) {
    const DerivSet& d = B.s[k];
    const T c = (T)(B.c_common == 1.0 ? d.c_hop : 1.0);
    {
      Spinor<T> lf, rf;
      load_spinor_live(lf, (const V*)(pz == 0 ? d.a : d.w), cb, g.Vh);
      load_spinor_live(rf, (const V*)(pz == 0 ? d.y : d.b), n, g.Vh);
      Half<T> l = project<MU, -1>(lf);
      scale_half(l, c);
      outer_half(Xf, project<MU, -1>(rf), l);
    }
    {
      Spinor<T> lb, rb;
      load_spinor_live(lb, (const V*)(pz == 0 ? d.w : d.a), n, g.Vh);
      load_spinor_live(rb, (const V*)(pz == 0 ? d.b : d.y), cb, g.Vh);
      Half<T> r = project<MU, +1>(rb);
      scale_half(r, c);
      outer_half(Xb, r, project<MU, +1>(lb));
    }
  }
  hop_force_store(F, g, pz, MU, cb, force_link<PREC>(gauge, g, pz, cb, z, MU), Xf, Xb, hop_force_factor(g, z, MU, B));
}

// FP32: a block takes 32 sites of both parities; warp (parity, mu) the links of direction mu.
// The warps of one parity read the same local spinors close together, and one parity's local
// fields are the other's neighbours, so L1 serves them after the first.
__global__ void __launch_bounds__(256, 2) k_force_hop(double* F, const void* gauge, Geom g, DerivBatch B) {
  chain_enter();
  const int cb = blockIdx.x * 32 + (threadIdx.x & 31);
  const int w = threadIdx.x >> 5, mu = w & 3, pz = w >> 2;
  if (cb >= g.Vh) return;
  int z[4];
  cb_coords(g, cb, pz, z);
  switch (mu) {
    case 0: hop_force_dir<PFMP_F32, 0>(F, gauge, g, pz, cb, z, B); break;
    case 1: hop_force_dir<PFMP_F32, 1>(F, gauge, g, pz, cb, z, B); break;
    case 2: hop_force_dir<PFMP_F32, 2>(F, gauge, g, pz, cb, z, B); break;
    default: hop_force_dir<PFMP_F32, 3>(F, gauge, g, pz, cb, z, B); break;
  }
}

// (1 + S g_mu) psi of the spinor at site cb for a run-time mu and sign: tile_term's phases
template <int PREC>
__device__ __forceinline__ void load_half_rt(Half<typename Prec<PREC>::real>& h, const typename Prec<PREC>::vec* f, int cb,
                                             int Vh, int mu, bool plus) {
  using T = typename Prec<PREC>::real;
  const bool low = mu < 2, isI = (mu & 1) == 0;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    cplx<T> u[3], v[3];
    load_spin<PREC>(u, f, k, cb, Vh);
    load_spin<PREC>(v, f, low ? 3 - k : 2 + k, cb, Vh);
    const bool neg = k == 0 ? (mu == 1) == plus : (mu == 2) == plus;
#pragma unroll
    for (int c = 0; c < 3; ++c) h.h[k][c] = u[c] + tile_unit(v[c], isI, neg);
  }
}

// FP64, and FP32 on lattices with too few sites for k_force_hop: a block takes 8 sites of one
// parity, a lane of each warp one link (site, mu) and the four warps every fourth contraction,
// their X_f and X_b added in shared memory.  FP64 is bound by its pipe (16 cycles a warp
// instruction): 192 instructions per link and contraction against ~500 with four-spin
// products and unfused sums, in pieces of 8 sites, so that every SM has its share
// (6x10x14x18, batch of 8: 531 us before; 4^4: 148).
constexpr int kForceSites = 8, kForceGroups = 4;
template <int PREC>
__global__ void __launch_bounds__(32 * kForceGroups) k_force_hop_split(double* F, const void* gauge, Geom g, DerivBatch B) {
  chain_enter();
  using T = typename Prec<PREC>::real;
  using V = typename Prec<PREC>::vec;
  __shared__ T sh[kForceGroups - 1][36][32];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int cb0 = blockIdx.x * kForceSites + (lane & (kForceSites - 1)), mu = lane / kForceSites;
  const int pz = blockIdx.y;
  const bool live = cb0 < g.Vh;
  const int cb = live ? cb0 : g.Vh - 1;
  int z[4];
  cb_coords(g, cb, pz, z);
  const int n = nbr_cb_rt(g, z, mu, +1);
  Mat3<T> Xf = mat_zero<T>(), Xb = mat_zero<T>();
#pragma unroll 1
  for (int k = grp; k < B.n; k += kForceGroups) {
    const DerivSet& d = B.s[k];
    const T c = (T)(B.c_common == 1.0 ? d.c_hop : 1.0);
    Half<T> l, r;
    load_half_rt<PREC>(l, (const V*)(pz == 0 ? d.a : d.w), cb, g.Vh, mu, false);
    load_half_rt<PREC>(r, (const V*)(pz == 0 ? d.y : d.b), n, g.Vh, mu, false);
    if (B.c_common == 1.0) scale_half(l, c);
    outer_half(Xf, r, l);
    load_half_rt<PREC>(r, (const V*)(pz == 0 ? d.b : d.y), cb, g.Vh, mu, true);
    load_half_rt<PREC>(l, (const V*)(pz == 0 ? d.w : d.a), n, g.Vh, mu, true);
    if (B.c_common == 1.0) scale_half(r, c);
    outer_half(Xb, r, l);
  }
  if (grp > 0)
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      sh[grp - 1][2 * e][lane] = Xf.m[e / 3][e % 3].re;
      sh[grp - 1][2 * e + 1][lane] = Xf.m[e / 3][e % 3].im;
      sh[grp - 1][18 + 2 * e][lane] = Xb.m[e / 3][e % 3].re;
      sh[grp - 1][18 + 2 * e + 1][lane] = Xb.m[e / 3][e % 3].im;
    }
  __syncthreads();
  if (grp > 0 || !live) return;
  const int ng = B.n < kForceGroups ? B.n : kForceGroups;
  for (int q = 0; q < ng - 1; ++q)
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      Xf.m[e / 3][e % 3] = Xf.m[e / 3][e % 3] + mk(sh[q][2 * e][lane], sh[q][2 * e + 1][lane]);
      Xb.m[e / 3][e % 3] = Xb.m[e / 3][e % 3] + mk(sh[q][18 + 2 * e][lane], sh[q][18 + 2 * e + 1][lane]);
    }
  hop_force_store(F, g, pz, mu, cb, glink<T>(gauge, g, z, mu), Xf, Xb, hop_force_factor(g, z, mu, B));
}

__device__ __forceinline__ double* hptr(double* Hc, const Geom& g, int p, int plane, int a) {
  return Hc + (size_t)((p * 6 + plane) * 8 + a) * g.Vh;
}

// P += P_K of chiral block B (spins 2B, 2B + 1) from O_ij = b_{2B+j} a_{2B+i}^dag:
// P_0 = O01 + O10, P_1 = -i (O01 - O10), P_2 = O00 - O11; P_1 is accumulated without its -i
template <int K, typename T>
__device__ __forceinline__ void pauli_acc(Mat3<T>& P, const Spinor<T>& a, const Spinor<T>& b, int B) {
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const cplx<T> b0 = b.s[2 * B][c], b1 = b.s[2 * B + 1][c], a0 = a.s[2 * B][d], a1 = a.s[2 * B + 1][d];
      if constexpr (K == 0)
        P.m[c][d] = cmad_nj(b0, a1, cmad_nj(b1, a0, P.m[c][d]));
      else if constexpr (K == 1)
        P.m[c][d] = cmad_nj(-b0, a1, cmad_nj(b1, a0, P.m[c][d]));
      else
        P.m[c][d] = cmad_nj(-b1, a1, cmad_nj(b0, a0, P.m[c][d]));
    }
}

// The two planes built from the Pauli component K, summed over the contractions of a
// batch: (planes, G) = K 2: (01, P+ + P-), (23, -P+ + P-); K 1: (02, P+ + P-),
// (13, P+ - P-); K 0: (03, -P+ + P-), (12, P+ + P-), with P+ / P- the blocks 0 / 1.
// P is linear in the contraction's fields: the batch's P+ and P- are accumulated in
// PREC and reduced to algebra components once.
template <int PREC, int K>
__device__ __forceinline__ void clover_insert_pair(double* Hc, const Geom& g, int p, int cb, const DerivBatch& B) {
  using T = typename Prec<PREC>::real;
  using V = typename Prec<PREC>::vec;
  Mat3<T> P[2] = {mat_zero<T>(), mat_zero<T>()};
#pragma unroll 1
  for (int s = 0; s < B.n; ++s) {
    const DerivSet& d = B.s[s];
    const T coef = (T)(2.0 * (p == 0 ? d.c_even : d.c_odd));
    Spinor<T> a, b;
    load_spinor_live(a, (const V*)(p == 0 ? d.a : d.w), cb, g.Vh);
    load_spinor_live(b, (const V*)(p == 0 ? d.b : d.y), cb, g.Vh);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int c = 0; c < 3; ++c) a.s[q][c] = coef * a.s[q][c];
#pragma unroll
    for (int q = 0; q < 2; ++q) pauli_acc<K>(P[q], a, b, q);
  }
  double r[2][8];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    cplx<T> t[8];
    tr_lambda(P[q], t);
    // P_1 = -i P: its traces' real parts are the imaginary parts of P's
#pragma unroll
    for (int k = 0; k < 8; ++k) r[q][k] = (double)(K == 1 ? t[k].im : t[k].re);
  }
  // plane index (0,1)=0 (0,2)=1 (0,3)=2 (1,2)=3 (1,3)=4 (2,3)=5
  constexpr int plA = K == 2 ? 0 : (K == 1 ? 1 : 2);
  constexpr int plB = K == 2 ? 5 : (K == 1 ? 4 : 3);
  constexpr double sA = K == 0 ? -1.0 : 1.0;  // sign of P+ in plane plA
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    hptr(Hc, g, p, plA, k)[cb] += sA * r[0][k] + r[1][k];
    if constexpr (K == 1)
      hptr(Hc, g, p, plB, k)[cb] += r[0][k] - r[1][k];
    else if constexpr (K == 2)
      hptr(Hc, g, p, plB, k)[cb] += -r[0][k] + r[1][k];
    else
      hptr(Hc, g, p, plB, k)[cb] += r[0][k] + r[1][k];
  }
}

// Hc[p] += coef (G~ + G~^dag) for G(a, b): h_a += 4 coef Re tr(T_a G) = 2 coef Re tr(lambda_a G),
// summed over the contractions of a batch: on the even sites G(a, b) with c_even, on the
// odd sites G(w, y) with c_odd.  A block takes 32 sites of parity blockIdx.y and warp K
// the Pauli component K (two of the six planes), so the three warps read the same
// spinors close together and each thread keeps 16 accumulators live instead of 48.
template <int PREC>
__global__ void __launch_bounds__(96) k_clover_insert(double* Hc, Geom g, DerivBatch B) {
  chain_enter();
  const int cb = blockIdx.x * 32 + (threadIdx.x & 31);
  const int K = threadIdx.x >> 5;
  const int p = blockIdx.y;
  if (cb >= g.Vh) return;
  switch (K) {
    case 0: clover_insert_pair<PREC, 0>(Hc, g, p, cb, B); break;
    case 1: clover_insert_pair<PREC, 1>(Hc, g, p, cb, B); break;
    default: clover_insert_pair<PREC, 2>(Hc, g, p, cb, B); break;
  }
}

// Hc[odd] += coef (G~ + G~^dag) with G = sum_{ij} sigma_{ji} Ainv_block(i, j) (det force)
__global__ void k_clover_insert_det(double* Hc, Geom g, const double2* Ainv, double coef) {
  const int cb = blockIdx.x * blockDim.x + threadIdx.x;
  if (cb >= g.Vh) return;
  HermBlock<double> B[2];
  load_clover(B, Ainv, cb, g.Vh);
  // full 6x6 blocks
  Mat3<double> P[2][3];
  for (int blk = 0; blk < 2; ++blk) {
    cplx<double> M[6][6];
    for (int i = 0; i < 6; ++i) M[i][i] = mk(B[blk].d[i], 0.0);
    for (int i = 1; i < 6; ++i)
      for (int j = 0; j < i; ++j) {
        M[i][j] = B[blk].o[tri_index(i, j)];
        M[j][i] = conj(M[i][j]);
      }
    // colour block (i, j) of spins (2 blk + i, 2 blk + j): M[3i + c][3j + d]
    // G = sum_{ij} sigma_{ji} X_ij; sigma_k blocks: s1 -> X01 + X10, s2 -> i X01 - i X10, s3 -> X00 - X11
    // (sigma_{ji}: s2_{10} = i multiplies X_01, s2_{01} = -i multiplies X_10)
    for (int c = 0; c < 3; ++c)
      for (int d = 0; d < 3; ++d) {
        cplx<double> x00 = M[c][d], x01 = M[c][3 + d], x10 = M[3 + c][d], x11 = M[3 + c][3 + d];
        P[blk][0].m[c][d] = x01 + x10;
        P[blk][1].m[c][d] = times_i(x01 - x10);
        P[blk][2].m[c][d] = x00 - x11;
      }
  }
  Mat3<double> G[6];
  for (int c = 0; c < 3; ++c)
    for (int d = 0; d < 3; ++d) {
      G[0].m[c][d] = P[0][2].m[c][d] + P[1][2].m[c][d];
      G[1].m[c][d] = P[0][1].m[c][d] + P[1][1].m[c][d];
      G[2].m[c][d] = P[1][0].m[c][d] - P[0][0].m[c][d];
      G[3].m[c][d] = P[0][0].m[c][d] + P[1][0].m[c][d];
      G[4].m[c][d] = P[0][1].m[c][d] - P[1][1].m[c][d];
      G[5].m[c][d] = P[1][2].m[c][d] - P[0][2].m[c][d];
    }
  for (int pl = 0; pl < 6; ++pl) {
    cplx<double> t[8];
    tr_lambda(G[pl], t);
    for (int k = 0; k < 8; ++k) hptr(Hc, g, 1, pl, k)[cb] += 2.0 * coef * t[k].re;
  }
}

// the insertion H of a plane at full coordinates x, times sgn, from a copy of Hc in T
template <typename T>
__device__ __forceinline__ Mat3<T> load_H(const T* Hc, const Geom& g, const int x[4], int plane, T sgn) {
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  const int cb = cb_index(g, x);
  T h[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) h[a] = sgn * ld_live(Hc + (size_t)((p * 6 + plane) * 8 + a) * g.Vh + cb);
  return from_algebra<T>(h);
}

__global__ void k_to_f32(const double* __restrict__ src, float* __restrict__ dst, long n) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    dst[i] = (float)src[i];
}

__device__ __forceinline__ int plane_index(int mu, int nu) {
  // (0,1)=0 (0,2)=1 (0,3)=2 (1,2)=3 (1,3)=4 (2,3)=5
  const int a = mu < nu ? mu : nu, b = mu < nu ? nu : mu;
  return a == 0 ? b - 1 : (a == 1 ? b + 1 : 5);
}

// index of D_nu of the plane (mu, nu) among a site's 12
__device__ __forceinline__ int d_index(int nu, int mu) { return nu * 3 + mu - (mu > nu); }

// D_nu(x) = H(x) U_nu(x) + U_nu(x) H(x+nu) of the 12 ordered planes (sign of H: + for
// mu < nu), [2 parity][12][9][Vh] complex
template <typename T>
__global__ void k_clover_d(cplx<T>* __restrict__ D, const void* gauge, const T* Hc, Geom g) {
  chain_enter();
  const int cb = blockIdx.x * blockDim.x + threadIdx.x;
  const int p = blockIdx.y, q = blockIdx.z, nu = q / 3;
  const int mu = q % 3 + (q % 3 >= nu);
  if (cb >= g.Vh) return;
  int x[4], xn[4];
  cb_coords(g, cb, p, x);
  shift_rt(g, x, nu, 1, xn);
  const int pl = plane_index(mu, nu);
  const T sg = mu < nu ? (T)1 : (T)-1;
  const Mat3<T> U = glink<T>(gauge, g, x, nu);
  Mat3<T> M = mm(load_H<T>(Hc, g, x, pl, sg), U);
  mac(M, U, load_H<T>(Hc, g, xn, pl, sg));
  cplx<T>* o = D + (size_t)((p * 12 + q) * 9) * g.Vh + cb;
#pragma unroll
  for (int e = 0; e < 9; ++e) o[(size_t)e * g.Vh] = M.m[e / 3][e % 3];
}

template <typename T>
__device__ __forceinline__ Mat3<T> load_d(const cplx<T>* D, const Geom& g, const int x[4], int nu, int mu) {
  const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
  const cplx<T>* o = D + (size_t)((p * 12 + d_index(nu, mu)) * 9) * g.Vh + cb_index(g, x);
  Mat3<T> M;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    if constexpr (sizeof(T) == 8) {
      const double2 v = ld_live(reinterpret_cast<const double2*>(o + (size_t)e * g.Vh));
      M.m[e / 3][e % 3] = mk(v.x, v.y);
    } else {
      const float2 v = ld_live(reinterpret_cast<const float2*>(o + (size_t)e * g.Vh));
      M.m[e / 3][e % 3] = mk(v.x, v.y);
    }
  }
  return M;
}

// what a leaf adds: the gauge staples (all to X), or X_above and Y_below of the clover term
enum { LEAF_GAUGE = 0, LEAF_CLOVER = 1 };

// M += the leaf of the link U_mu(z) on the upper or lower side of direction nu
template <typename T, int KIND>
__device__ __forceinline__ void add_leaf(Mat3<T>& M, const void* gauge, const cplx<T>* D, const Geom& g, const int z[4], int mu,
                                         int nu, bool up) {
  int zm[4], zn[4], znm[4];
  shift_rt(g, z, mu, 1, zm);
  if (up) {
    shift_rt(g, z, nu, 1, zn);
    const Mat3<T> Um = glink<T>(gauge, g, zn, mu);
    if constexpr (KIND == LEAF_GAUGE) {  // U_nu(z+mu) [U_nu(z) U_mu(z+nu)]^dag
      mac_nd(M, glink<T>(gauge, g, zm, nu), mm(glink<T>(gauge, g, z, nu), Um));
    } else {
      mac_nd(M, load_d<T>(D, g, zm, nu, mu), mm(glink<T>(gauge, g, z, nu), Um));
      mac_nd(M, glink<T>(gauge, g, zm, nu), mm(load_d<T>(D, g, z, nu, mu), Um));
    }
  } else {
    shift_rt(g, z, nu, -1, zn);
    shift_rt(g, zn, mu, 1, znm);
    const Mat3<T> Um = glink<T>(gauge, g, zn, mu), Un = glink<T>(gauge, g, zn, nu), Unm = glink<T>(gauge, g, znm, nu);
    if constexpr (KIND == LEAF_GAUGE) {  // [U_mu(z-nu) U_nu(z+mu-nu)]^dag U_nu(z-nu)
      mac_dn(M, mm(Um, Unm), Un);
    } else {
      mac_dn(M, load_d<T>(D, g, zn, nu, mu), mm(Um, Unm));
      mac_dn(M, Un, mm(Um, load_d<T>(D, g, znm, nu, mu)));
    }
  }
}

// tr(lambda_a Z) of one generator a (run-time), Z given by its entries
template <typename T, typename Get>
__device__ __forceinline__ cplx<T> tr_lambda_rt(int a, Get Z) {
  if (a == 2) return Z(0, 0) - Z(1, 1);
  if (a == 7) return (T)kInvSqrt3 * (Z(0, 0) + Z(1, 1) - (T)2 * Z(2, 2));
  const int i = a < 2 ? 0 : (a < 5 ? 0 : 1), j = a < 2 ? 1 : 2;
  const cplx<T> u = Z(i, j), l = Z(j, i);
  return (a == 0 || a == 3 || a == 5) ? l + u : times_i(u - l);
}

// The gauge force, F += (beta/6) Im tr(lambda_a U S), and the clover force,
// F += (1/16) Re tr(lambda_a [U X - Y U^dag]), one thread per link: FP32 on large lattices, and
// the FP64 gauge force on all but the smallest.
// A block takes 32 sites of parity blockIdx.y and warp mu the links U_mu of those sites,
// so the four warps share the fields they read through L1.
template <typename T, int KIND>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 4 : 2) k_leaf_force(double* F, const void* gauge, const cplx<T>* D, Geom g, double coef) {
  chain_enter();
  const int cb = blockIdx.x * 32 + (threadIdx.x & 31);
  const int mu = threadIdx.x >> 5;
  const int p = blockIdx.y;
  if (cb >= g.Vh) return;
  int z[4];
  cb_coords(g, cb, p, z);
  Mat3<T> X = mat_zero<T>(), Y = mat_zero<T>();
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    add_leaf<T, KIND>(X, gauge, D, g, z, mu, nu, true);
    add_leaf<T, KIND>(KIND == LEAF_GAUGE ? X : Y, gauge, D, g, z, mu, nu, false);
  }
  const Mat3<T> U = glink<T>(gauge, g, z, mu);
  Mat3<T> Z = mm(U, X);
  if (KIND == LEAF_CLOVER) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) Y.m[i][j] = -Y.m[i][j];
    mac_nd(Z, Y, U);
  }
  cplx<T> t[8];
  tr_lambda(Z, t);
#pragma unroll
  for (int a = 0; a < 8; ++a) fptr(F, g, p, mu, a)[cb] += coef * (double)(KIND == LEAF_GAUGE ? t[a].im : t[a].re);
}

// The same with 24 threads per site, one per leaf (mu, nu, side), in blocks of 4 sites: the FP64
// clover force (bound by its pipe: equal small pieces for every SM, no thread with a long
// chain) and both precisions on small lattices.  The leaves meet in shared memory; 12 threads per site take one row of
// Z = U X - Y U^dag each, then every thread one or two of the 32 components.
constexpr int kLeafSites = 4;
template <typename T, int KIND>
__global__ void __launch_bounds__(24 * kLeafSites) k_leaf_force_split(double* F, const void* gauge, const cplx<T>* D, Geom g,
                                                                      double coef) {
  constexpr int NS = kLeafSites;
  __shared__ cplx<T> L[24][9][NS], Zs[4][9][NS];
  const int site = threadIdx.x % NS, j = threadIdx.x / NS;
  const int p = blockIdx.y, cb0 = blockIdx.x * NS + site;
  const bool live = cb0 < g.Vh;
  const int cb = live ? cb0 : g.Vh - 1;
  int z[4];
  cb_coords(g, cb, p, z);
  {
    const int mu = j / 6, ni = (j % 6) >> 1;
    Mat3<T> M = mat_zero<T>();
    add_leaf<T, KIND>(M, gauge, D, g, z, mu, ni + (ni >= mu), (j & 1) == 0);
#pragma unroll
    for (int e = 0; e < 9; ++e) L[j][e][site] = M.m[e / 3][e % 3];
  }
  __syncthreads();
  if (j < 12) {
    const int mu = j / 3, i = j % 3;
    const Mat3<T> U = glink<T>(gauge, g, z, mu);
    cplx<T> zr[3] = {mk<T>(0, 0), mk<T>(0, 0), mk<T>(0, 0)};
    const cplx<T> u[3] = {i == 0 ? U.m[0][0] : (i == 1 ? U.m[1][0] : U.m[2][0]),
                          i == 0 ? U.m[0][1] : (i == 1 ? U.m[1][1] : U.m[2][1]),
                          i == 0 ? U.m[0][2] : (i == 1 ? U.m[1][2] : U.m[2][2])};
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        cplx<T> x = L[mu * 6][3 * k + c][site] + L[mu * 6 + 2][3 * k + c][site] + L[mu * 6 + 4][3 * k + c][site];
        if (KIND == LEAF_GAUGE)
          x = x + L[mu * 6 + 1][3 * k + c][site] + L[mu * 6 + 3][3 * k + c][site] + L[mu * 6 + 5][3 * k + c][site];
        zr[c] = cmad(u[k], x, zr[c]);
      }
    if (KIND == LEAF_CLOVER)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const cplx<T> y = L[mu * 6 + 1][3 * i + k][site] + L[mu * 6 + 3][3 * i + k][site] + L[mu * 6 + 5][3 * i + k][site];
#pragma unroll
        for (int c = 0; c < 3; ++c) zr[c] = cmad_nj(-y, U.m[c][k], zr[c]);
      }
#pragma unroll
    for (int c = 0; c < 3; ++c) Zs[mu][3 * i + c][site] = zr[c];
  }
  __syncthreads();
  if (!live) return;
  for (int q = j; q < 32; q += 24) {
    const int mu = q >> 3, a = q & 7;
    const cplx<T> t = tr_lambda_rt<T>(a, [&](int i, int k) { return Zs[mu][3 * i + k][site]; });
    fptr(F, g, p, mu, a)[cb] += coef * (double)(KIND == LEAF_GAUGE ? t.im : t.re);
  }
}

// ------------------------------------------------------------------ host side
// lattices whose links, 128 to a block, leave SMs idle or with one block in flight
static bool force_small(const Geom& g) { return g.Vh < 32 * 152 * 2; }

// FP64 gauge force: a thread per leaf (k_leaf_force_split) on the smallest lattices, a thread per
// link from this many sites per parity on.  The leaves' links come in pieces of 4 sites and
// cross shared memory again, which costs more than the pipe's share of a whole link once
// there is a block of links for most SMs (us per force, leaf / link: 37 / 62 at 256, 87 / 64 at
// 1296, 345 / 198 at 7560, 2840 / 1250 at 65536, where a thread per site took 2260).  Clover
// leaves have four products and 18 more numbers to load each, and stay with a thread per leaf.
constexpr int kGaugeWhole64 = 768;

template <typename T, int KIND>
static void leaf_force(pfmp_ctx* c, double* F, const void* gauge, const cplx<T>* D, double coef) {
  const dim3 split(nblocks(c->g.Vh, kLeafSites), 2);
  if constexpr (sizeof(T) == 8) {
    bool whole = false;
    if constexpr (KIND == LEAF_GAUGE) whole = c->g.Vh >= kGaugeWhole64;
    if (whole)
      k_leaf_force<T, LEAF_GAUGE><<<dim3(nblocks(c->g.Vh, 32), 2), 128, 0, c->stream>>>(F, gauge, D, c->g, coef);
    else
      k_leaf_force_split<T, KIND><<<split, 24 * kLeafSites, 0, c->stream>>>(F, gauge, D, c->g, coef);
  } else {
    if (force_small(c->g))
      k_leaf_force_split<T, KIND><<<split, 24 * kLeafSites, 0, c->stream>>>(F, gauge, D, c->g, coef);
    else
      launch_chained(k_leaf_force<T, KIND>, dim3(nblocks(c->g.Vh, 32), 2), 128, c->stream, F, gauge, D, c->g, coef);
  }
  PFMP_CHECK_LAUNCH();
}
void deriv_mhat_batch(pfmp_ctx* c, int prec, double* F, double* Hc, const DerivBatch& B) {
  if (B.n == 0) return;
  PFMP_REQUIRE(B.n <= kMaxDerivSets, PFMP_E_INVALID, "too many contractions in one force batch");
  bool clover = false;
  for (int k = 0; k < B.n; ++k) clover = clover || B.s[k].c_even != 0.0 || B.s[k].c_odd != 0.0;
  const dim3 grid(nblocks(c->g.Vh, 32), 2), split(nblocks(c->g.Vh, kForceSites), 2);
  DerivBatch C = B;
  // one coefficient for the whole batch: applied once to the sum
  C.c_common = B.s[0].c_hop;
  for (int k = 1; k < B.n; ++k)
    if (B.s[k].c_hop != B.s[0].c_hop) C.c_common = 1.0;
  if (prec == PFMP_F64)
    k_force_hop_split<PFMP_F64><<<split, 32 * kForceGroups, 0, c->stream>>>(F, c->U64, c->g, C);
  else if (force_small(c->g))
    launch_chained(k_force_hop_split<PFMP_F32>, split, 32 * kForceGroups, c->stream, F, c->U32, c->g, C);
  else
    launch_chained(k_force_hop, nblocks(c->g.Vh, 32), 256, c->stream, F, c->U32, c->g, C);
  PFMP_CHECK_LAUNCH();
  if (!clover) return;
  if (prec == PFMP_F64)
    k_clover_insert<PFMP_F64><<<grid, 96, 0, c->stream>>>(Hc, c->g, B);
  else
    launch_chained(k_clover_insert<PFMP_F32>, grid, 96, c->stream, Hc, c->g, B);
  PFMP_CHECK_LAUNCH();
}
void clover_insert_det(pfmp_op* op, double* Hc, double coef) {
  pfmp_ctx* c = op->ctx;
  k_clover_insert_det<<<nblocks(c->g.Vh, 128), 128, 0, c->stream>>>(Hc, c->g, op->clov64[1], coef);
  PFMP_CHECK_LAUNCH();
}
// prec = PFMP_F64: FP64 arithmetic on the master links; PFMP_F32: FP32 arithmetic on the
// compressed FP32 links (the forces of an MD with FP32 forces), FP64 accumulation
// prec = PFMP_F32 reads an FP32 copy of Hc (converted once here, not per leaf)
void clover_force(pfmp_ctx* c, int prec, double* F, const double* Hc) {
  const long n = 96L * c->g.Vh;
  const dim3 grid(nblocks(c->g.Vh, 64), 2, 12);
  const size_t words = (size_t)2 * 12 * 9 * c->g.Vh;
  if (prec == PFMP_F64) {
    if (!c->clov_d[0]) c->clov_d[0] = dev_alloc(words * sizeof(cplx<double>));
    cplx<double>* D = (cplx<double>*)c->clov_d[0];
    k_clover_d<double><<<grid, 64, 0, c->stream>>>(D, c->U64, Hc, c->g);
    PFMP_CHECK_LAUNCH();
    leaf_force<double, LEAF_CLOVER>(c, F, c->U64, D, 0.0625);
  } else {
    if (!c->hc32) c->hc32 = (float*)dev_alloc(n * sizeof(float));
    if (!c->clov_d[1]) c->clov_d[1] = dev_alloc(words * sizeof(cplx<float>));
    cplx<float>* D = (cplx<float>*)c->clov_d[1];
    k_to_f32<<<std::min(nblocks(n), 152 * 8), kBlock, 0, c->stream>>>(Hc, c->hc32, n);
    PFMP_CHECK_LAUNCH();
    launch_chained(k_clover_d<float>, grid, 64, c->stream, D, c->U32, c->hc32, c->g);
    PFMP_CHECK_LAUNCH();
    leaf_force<float, LEAF_CLOVER>(c, F, c->U32, D, 0.0625);
  }
}
void gauge_force(pfmp_ctx* c, int prec, double* F, double beta) {
  if (prec == PFMP_F64)
    leaf_force<double, LEAF_GAUGE>(c, F, c->U64, nullptr, beta / 6.0);
  else
    leaf_force<float, LEAF_GAUGE>(c, F, c->U32, nullptr, beta / 6.0);
}

}  // namespace pfmp
