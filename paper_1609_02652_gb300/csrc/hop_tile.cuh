// Stencil kernels that share one output site among several threads (FP64 and double-float
// at every size, FP32 on small lattices).  A block holds NS sites; the threads of one role
// are consecutive sites, so loads stay coalesced; the hop products meet in shared memory
// and each finishing thread sums and applies one clover row per component.
//
//   k_hop_tile  16 threads per site: thread (d, k) takes the hop term of direction d
//               (2 mu + {0 forward, 1 backward}) for component k of the half spinor
//   k_hop_pair  8 threads per site: thread (mu, k) takes both hops of mu and writes their
//               sum s = f + b and difference d = f - b, which is all the rebuild needs
//               (the upper spins add s, the lower spins a unit phase times d)
//
// What bounds them: GB300's FP64 pipe issues one warp instruction in 16 cycles per SM.
// With one thread per site and 128-site blocks (the earlier kernel) the lattice came in
// too few pieces (one SM busy at 4^4, 10 SMs with twice the others' share at 12^3x24), sums
// of products cost three FP64 instructions where a chain of fused multiply-adds costs two,
// and sign flips went through the FP64 pipe: 1464+ FP64 instructions per site and hop.
// Here a site costs 1156 (k_hop_tile) or 1108 (k_hop_pair, whose second product chain
// starts from the first one's result), signs are flipped by integer operations, and the
// pieces are 8 or 16 sites.  GB300, us per K (four launches), one thread per site before /
// now: FP64 4^4 220 / 25, 12^3x24 423 / 181, 16^3x32 828 / 506 (FP64 pipe 88% busy),
// 32^3x64 10920 / 7850.  On the FP32 pipe (double-float, and FP32 where a lattice has too
// few sites to hide one thread's chain of eight directions) the gain is latency: see the
// size rules at the end of this file.
#pragma once
#include "dfloat.cuh"
#include "hop.cuh"

namespace pfmp {

constexpr int kTileSites = 8;   // sites per 128-thread block of k_hop_tile
constexpr int kPairSites = 16;  // sites per 128-thread block of k_hop_pair

// x with its sign flipped where neg is set: an integer operation (the FP64 pipe is the one
// to spare here)
__device__ __forceinline__ float sign_if(float x, bool neg) {
  return __uint_as_float(__float_as_uint(x) ^ (neg ? 0x80000000u : 0u));
}
__device__ __forceinline__ double sign_if(double x, bool neg) {
  return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000u : 0), __double2loint(x));
}
__device__ __forceinline__ df sign_if(df x, bool neg) { return df(sign_if(x.hi, neg), sign_if(x.lo, neg)); }
// v times (isI ? i : 1) times (neg ? -1 : 1)
template <typename T>
__device__ __forceinline__ cplx<T> tile_unit(const cplx<T>& v, bool isI, bool neg) {
  return isI ? mk(sign_if(v.im, !neg), sign_if(v.re, neg)) : mk(sign_if(v.re, neg), sign_if(v.im, neg));
}

// complex components 3 s .. 3 s + 2 (spin s) of the spinor at site cb.  FP32: the kernels that
// take it are chained (reduce.cuh), so no load of a spinor goes through the read-only path.
template <int PREC>
__device__ __forceinline__ void load_spin(cplx<typename Prec<PREC>::real> v[3], const typename Prec<PREC>::vec* f, int s,
                                          int cb, int Vh) {
  if constexpr (PREC == PFMP_F32) {  // two components per word: spin s starts at word 3 s / 2
    const float4* q = f + (size_t)((3 * s) >> 1) * Vh + cb;
    const float4 a = ld_live(q), b = ld_live(q + Vh);
    const bool odd = s & 1;
    v[0] = odd ? mk(a.z, a.w) : mk(a.x, a.y);
    v[1] = odd ? mk(b.x, b.y) : mk(a.z, a.w);
    v[2] = odd ? mk(b.z, b.w) : mk(b.x, b.y);
  } else {
    const auto* q = f + (size_t)(3 * s) * Vh + cb;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const auto w = __ldg(q + (size_t)c * Vh);
      if constexpr (PREC == PREC_DF)
        v[c] = c_of(w);
      else
        v[c] = mk(w.x, w.y);
    }
  }
}

// one complex component (0..11) of the spinor at site cb
template <int PREC>
__device__ __forceinline__ cplx<typename Prec<PREC>::real> load_comp(const typename Prec<PREC>::vec* f, int comp, int cb,
                                                                     int Vh) {
  if constexpr (PREC == PFMP_F32) {
    const float2 w = ld_live(reinterpret_cast<const float2*>(f + (size_t)(comp >> 1) * Vh + cb) + (comp & 1));
    return mk(w.x, w.y);
  } else if constexpr (PREC == PREC_DF) {
    return c_of(__ldg(f + (size_t)comp * Vh + cb));
  } else {
    const double2 w = __ldg(f + (size_t)comp * Vh + cb);
    return mk(w.x, w.y);
  }
}
template <int PREC>
__device__ __forceinline__ void store_comp(typename Prec<PREC>::vec* f, cplx<typename Prec<PREC>::real> v, int comp, int cb,
                                           int Vh) {
  if constexpr (PREC == PFMP_F32)
    reinterpret_cast<float2*>(f + (size_t)(comp >> 1) * Vh + cb)[comp & 1] = make_float2(v.re, v.im);
  else if constexpr (PREC == PREC_DF)
    f[(size_t)comp * Vh + cb] = v_of(v);
  else
    f[(size_t)comp * Vh + cb] = make_double2(v.re, v.im);
}

// row i of chiral block blk: its diagonal entry and the off-diagonal entries B_ij, j != i in
// ascending order (the stored lower triangle, conjugated above the diagonal)
template <int PREC>
__device__ __forceinline__ void load_clover_row(typename Prec<PREC>::real& diag, cplx<typename Prec<PREC>::real> off[5],
                                                const typename Prec<PREC>::vec* clov, int blk, int i, int cb, int Vh) {
  if constexpr (PREC == PFMP_F32) {  // 36 reals in nine words: 6 diagonal, then 15 complex
    const float4* g = clov + (size_t)(9 * blk) * Vh + cb;
    diag = __ldg(reinterpret_cast<const float*>(g + (size_t)(i >> 2) * Vh) + (i & 3));
#pragma unroll
    for (int t = 0; t < 5; ++t) {
      const int j = t + (t >= i), o = j < i ? tri_index(i, j) : tri_index(j, i), q = 6 + 2 * o;
      const float2 w = __ldg(reinterpret_cast<const float2*>(g + (size_t)(q >> 2) * Vh) + ((q >> 1) & 1));
      off[t] = mk(w.x, sign_if(w.y, j > i));
    }
  } else {
    const auto* g = clov + (size_t)(18 * blk) * Vh + cb;
    if constexpr (PREC == PREC_DF) {
      const float2 w = __ldg(reinterpret_cast<const float2*>(g + (size_t)(i >> 1) * Vh) + (i & 1));
      diag = df(w.x, w.y);
    } else {
      diag = __ldg(reinterpret_cast<const double*>(g + (size_t)(i >> 1) * Vh) + (i & 1));
    }
#pragma unroll
    for (int t = 0; t < 5; ++t) {
      const int j = t + (t >= i), o = j < i ? tri_index(i, j) : tri_index(j, i);
      const auto w = __ldg(g + (size_t)(3 + o) * Vh);
      if constexpr (PREC == PREC_DF)
        off[t] = c_of(w);
      else
        off[t] = mk(w.x, w.y);
      off[t].im = sign_if(off[t].im, j > i);
    }
  }
}

// row i of the clover epilogue: v the six inputs of the chiral block (entry j at v[j * ld]),
// acc the hop's component of this row (EPI_CLOV: v holds the summed hop itself)
template <int EPI, typename T>
__device__ __forceinline__ cplx<T> clover_row(T diag, const cplx<T> off[5], const cplx<T>* v, int ld, int i, T cf,
                                              const cplx<T>& acc) {
  // the small off-diagonal terms first: the large diagonal term rounds the sum once
  cplx<T> y = off[0] * v[(i == 0) * ld];
#pragma unroll
  for (int t = 1; t < 5; ++t) y = cmad(off[t], v[(t + (t >= i)) * ld], y);
  if (EPI == EPI_XPAY) y = mk(mad(cf, acc.re, y.re), mad(cf, acc.im, y.im));
  const cplx<T> own = v[i * ld];
  y = mk(mad(diag, own.re, y.re), mad(diag, own.im, y.im));
  return y;
}

// the hop term of (d, k) at output site x (index cb): r[c] = [U h]_c with h the component k
// of the projected neighbour spinor.  Backward terms use U^dag h = conj(U^T conj(h)): the
// element (j, i) of the stored link takes the place of (i, j).
template <int PREC, bool DAG>
__device__ __forceinline__ void tile_term(cplx<typename Prec<PREC>::real> r[3], const HopParams<PREC>& a, const int x[4],
                                          int cb, int d, int k) {
  using T = typename Prec<PREC>::real;
  const Geom& g = a.g;
  const int mu = d >> 1;
  const bool fwd = (d & 1) == 0, sp = fwd ? DAG : !DAG;  // sp: the projector's sign is +
  const bool low = mu < 2, isI = (mu & 1) == 0;
  const int n = nbr_cb_rt(g, x, mu, fwd ? +1 : -1);
  const int lcb = fwd ? cb : n;
  const typename Prec<PREC>::vec* lf = link_plane<PREC>(a.gauge, (fwd ? a.p : 1 - a.p) * 4 + mu, g.Vh);
  cplx<T> u[3], v[3];
  load_spin<PREC>(u, a.in, k, n, g.Vh);
  load_spin<PREC>(v, a.in, low ? 3 - k : 2 + k, n, g.Vh);
  Mat3<T> U;
  if constexpr (PREC == PFMP_F32) {
    load_link(U, lf, lcb, g.Vh);
    dagger_if(U, !fwd);
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const auto w = __ldg(lf + (size_t)(fwd ? 3 * i + j : 3 * j + i) * g.Vh + lcb);
        if constexpr (PREC == PREC_DF)
          U.m[i][j] = c_of(w);
        else
          U.m[i][j] = mk(w.x, w.y);
      }
  }
  const bool neg = k == 0 ? (mu == 1) == sp : (mu == 2) == sp;
  const bool cj = PREC != PFMP_F32 && !fwd;
  cplx<T> h[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    h[c] = u[c] + tile_unit(v[c], isI, neg);
    h[c].im = sign_if(h[c].im, cj);
  }
  const bool flip = g.bc_t < 0 && mu == 3 && (fwd ? x[3] == g.L[3] - 1 : x[3] == 0);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cplx<T> t = U.m[i][0] * h[0];
    t = cmad(U.m[i][1], h[1], t);
    t = cmad(U.m[i][2], h[2], t);
    r[i] = mk(sign_if(t.re, flip), sign_if(t.im, flip != cj));
  }
}

// contribution of the hop term r (component kk of direction d, chosen by tile_source) to
// the spin s of the output
__device__ __forceinline__ int tile_source(int d, int s) { return s < 2 ? s : (d < 4 ? 3 - s : s - 2); }
template <bool DAG, typename T>
__device__ __forceinline__ cplx<T> tile_phase(const cplx<T>& r, int d, int s) {
  if (s < 2) return r;
  const int mu = d >> 1;
  const bool sp = (d & 1) == 0 ? DAG : !DAG, low = mu < 2, isI = (mu & 1) == 0;
  return tile_unit(r, isI, s == 2 ? isI == sp : low == sp);
}

// one block per 8 sites (small lattices only); EPI_CLOV has coef = 1, as in every caller
template <int PREC, bool DAG, int EPI, bool REDUCE>
__global__ void __launch_bounds__(16 * kTileSites, 5) k_hop_tile(HopParams<PREC> a) {
  using T = typename Prec<PREC>::real;
  constexpr int NS = kTileSites;
  if (a.scal && a.scal->done) return;
  __shared__ cplx<T> R[48][NS];  // [d][k][colour][site]
  __shared__ cplx<T> S[12][NS];  // the clover term's input
  const int Vh = a.g.Vh;
  const int site = threadIdx.x % NS, j = threadIdx.x / NS;
  const int cb0 = blockIdx.x * NS + site;
  const bool live = cb0 < Vh;
  const int cb = live ? cb0 : Vh - 1;
  const T cf = (T)a.coef;
  double nrm[1] = {0.0};
  {
    int x[4];
    cb_coords(a.g, cb, a.p, x);
    cplx<T> r[3];
    tile_term<PREC, DAG>(r, a, x, cb, j >> 1, j & 1);
#pragma unroll
    for (int c = 0; c < 3; ++c) R[j * 3 + c][site] = r[c];
  }
  const int s = j / 3, c = j % 3, blk = j / 6, i = j - 6 * blk;
  T diag;
  cplx<T> off[5], acc;
  if (EPI != EPI_PLAIN && j < 12) load_clover_row<PREC>(diag, off, a.clov, blk, i, cb, Vh);
  if (EPI == EPI_XPAY && j < 12) S[j][site] = load_comp<PREC>(a.x, j, cb, Vh);
  __syncthreads();
  if (j < 12) {
    acc = tile_phase<DAG>(R[tile_source(0, s) * 3 + c][site], 0, s);
#pragma unroll
    for (int d = 1; d < 8; ++d) acc = acc + tile_phase<DAG>(R[(2 * d + tile_source(d, s)) * 3 + c][site], d, s);
    if (EPI == EPI_CLOV) S[j][site] = acc;
  }
  if (EPI == EPI_CLOV) __syncthreads();
  if (j < 12 && live) {
    cplx<T> y;
    if (EPI == EPI_PLAIN)
      y = cf * acc;
    else
      y = clover_row<EPI>(diag, off, &S[6 * blk][site], NS, i, cf, acc);
    store_comp<PREC>(a.out, y, j, cb, Vh);
    if (REDUCE) nrm[0] = (double)norm2(y);
  }
  if (REDUCE) {
    double tot[1];
    if (grid_sum<1>(nrm, a.rb, tot)) {
      *a.norm_out = tot[0];
      if (a.scal) a.scal->alpha = a.scal->rr / tot[0];
    }
  }
}

// both hops of direction mu for component k at output site x (index cb): s = f + b and d =
// f - b, f = U_mu(x) h_+ and b = U_mu(x - mu)^dag h_-.  In FP64 b's product chain starts from
// f and d = 2 f - s: 6 instructions fewer of the pipe that bounds the kernel, for one more
// rounding of the size of s's own (K at 16^3x32 against 64-bit torch: 3.3e-16, 3.6e-16 before)
template <int PREC, bool DAG>
__device__ __forceinline__ void pair_term(cplx<typename Prec<PREC>::real> sm[3], cplx<typename Prec<PREC>::real> dm[3],
                                          const HopParams<PREC>& a, const int x[4], int cb, int mu, int k) {
  using T = typename Prec<PREC>::real;
  constexpr bool CHAIN = PREC == PFMP_F64;
  const Geom& g = a.g;
  const bool low = mu < 2, isI = (mu & 1) == 0;
  const int kp = low ? 3 - k : 2 + k;
  const bool neg = k == 0 ? (mu == 1) == DAG : (mu == 2) == DAG;  // forward projector; the backward one is opposite
  cplx<T> f[3];
  {
    const int n = nbr_cb_rt(g, x, mu, +1);
    const typename Prec<PREC>::vec* lf = link_plane<PREC>(a.gauge, a.p * 4 + mu, g.Vh);
    cplx<T> u[3], v[3];
    load_spin<PREC>(u, a.in, k, n, g.Vh);
    load_spin<PREC>(v, a.in, kp, n, g.Vh);
    Mat3<T> U;
    load_link(U, lf, cb, g.Vh);
    const bool flip = g.bc_t < 0 && mu == 3 && x[3] == g.L[3] - 1;
    cplx<T> h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const cplx<T> t = u[c] + tile_unit(v[c], isI, neg);
      h[c] = mk(sign_if(t.re, flip), sign_if(t.im, flip));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) f[i] = cmad(U.m[i][2], h[2], cmad(U.m[i][1], h[1], U.m[i][0] * h[0]));
  }
  {
    const int n = nbr_cb_rt(g, x, mu, -1);
    const typename Prec<PREC>::vec* lf = link_plane<PREC>(a.gauge, (1 - a.p) * 4 + mu, g.Vh);
    cplx<T> u[3], v[3];
    load_spin<PREC>(u, a.in, k, n, g.Vh);
    load_spin<PREC>(v, a.in, kp, n, g.Vh);
    Mat3<T> U;
    load_link(U, lf, n, g.Vh);
    const bool flip = g.bc_t < 0 && mu == 3 && x[3] == 0;
    cplx<T> h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const cplx<T> t = u[c] + tile_unit(v[c], isI, !neg);
      h[c] = mk(sign_if(t.re, flip), sign_if(t.im, flip));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      cplx<T> t = CHAIN ? f[i] : cj_mul(U.m[0][i], h[0]);
#pragma unroll
      for (int j = CHAIN ? 0 : 1; j < 3; ++j) {  // + conj(U_ji) h_j
        const cplx<T> e = U.m[j][i];
        t = mk(mad(e.im, h[j].im, mad(e.re, h[j].re, t.re)), mad(-e.im, h[j].re, mad(e.re, h[j].im, t.im)));
      }
      sm[i] = CHAIN ? t : f[i] + t;
      dm[i] = CHAIN ? mk(mad((T)2, f[i].re, -t.re), mad((T)2, f[i].im, -t.im)) : f[i] - t;
    }
  }
}

template <int PREC, bool DAG, int EPI, bool REDUCE>
__global__ void __launch_bounds__(8 * kPairSites, 5) k_hop_pair(HopParams<PREC> a) {
  if constexpr (PREC == PFMP_F32) chain_enter();
  using T = typename Prec<PREC>::real;
  constexpr int NS = kPairSites;
  if (a.scal && a.scal->done) return;
  __shared__ cplx<T> R[48][NS];  // [mu][k][s | d][colour][site]
  __shared__ cplx<T> S[12][NS];  // the clover term's input
  const int Vh = a.g.Vh;
  const int site = threadIdx.x % NS, j = threadIdx.x / NS;
  const T cf = (T)a.coef;
  double nrm[1] = {0.0};
  for (int tile = blockIdx.x; tile * NS < Vh; tile += gridDim.x) {
    const int cb0 = tile * NS + site;
    const bool live = cb0 < Vh;
    const int cb = live ? cb0 : Vh - 1;
    {
      int x[4];
      cb_coords(a.g, cb, a.p, x);
      cplx<T> sm[3], d[3];
      pair_term<PREC, DAG>(sm, d, a, x, cb, j >> 1, j & 1);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        R[j * 6 + c][site] = sm[c];
        R[j * 6 + 3 + c][site] = d[c];
      }
    }
    if (EPI == EPI_XPAY && j < 6) {
      S[j][site] = load_comp<PREC>(a.x, j, cb, Vh);
      S[j + 6][site] = load_comp<PREC>(a.x, j + 6, cb, Vh);
    }
    __syncthreads();
    const int k = j / 3, c = j % 3;
    cplx<T> acc[2];
    if (j < 6) {
      acc[0] = R[k * 6 + c][site];
#pragma unroll
      for (int mu = 1; mu < 4; ++mu) acc[0] = acc[0] + R[(2 * mu + k) * 6 + c][site];
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {  // out_{2+k} += phase d_{kk}, kk = 1 - k for mu < 2
        const bool low = mu < 2, isI = (mu & 1) == 0;
        const int kk = low ? 1 - k : k;
        const cplx<T> v = tile_unit(R[(2 * mu + kk) * 6 + 3 + c][site], isI, k == 0 ? isI == DAG : low == DAG);
        acc[1] = mu == 0 ? v : acc[1] + v;
      }
      if (EPI == EPI_CLOV) {
        S[j][site] = acc[0];
        S[j + 6][site] = acc[1];
      }
    }
    if (EPI == EPI_CLOV) __syncthreads();
    if (j < 6) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        cplx<T> y;
        if (EPI == EPI_PLAIN) {
          y = cf * acc[b];
        } else {
          T diag;
          cplx<T> off[5];
          load_clover_row<PREC>(diag, off, a.clov, b, j, cb, Vh);
          y = clover_row<EPI>(diag, off, &S[6 * b][site], NS, j, cf, acc[b]);
        }
        if (live) {
          store_comp<PREC>(a.out, y, 6 * b + j, cb, Vh);
          if (REDUCE) nrm[0] += (double)norm2(y);
        }
      }
    }
    __syncthreads();  // R and S are rewritten by the next tile
  }
  if (REDUCE) {
    double tot[1];
    if (grid_sum<1>(nrm, a.rb, tot)) {
      *a.norm_out = tot[0];
      if (a.scal) a.scal->alpha = a.scal->rr / tot[0];
    }
  }
}

// ---------------------------------------------------------------- host
// Several threads per site below, one thread per site from these sizes on (sites per
// parity; us per K of four launches, GB300):
//  * FP32: a lattice with few sites leaves k_hop's 128-site blocks on a few SMs, each waiting
//    for one thread's chain of eight neighbours.  k_hop_pair against k_hop (196 registers):
//    16.5 / 24.7 at 256 to 2048, 17.2 / 24.7 at 4096, 24.7 / 24.6 at 6144, 32.9 / 24.6 at 20736,
//    41.0 / 28.8 at 27648.
//  * FP64 and double-float, always several threads: k_hop_tile (8-site blocks, 16 threads
//    per site) while the 16-site blocks of k_hop_pair would leave SMs idle, k_hop_pair from
//    there on.  FP64 tile / pair: 25 / 34 at 128, 33 / 41 at 2048, 56 / 49 at 4096, 531 /
//    506 at 65536; double-float (true residual) 72 / 75 at 128, 302 / 297 at 65536.
constexpr int kPairMaxF32 = 32 * 152;
constexpr int kTileMax = kPairSites * 152;
inline bool hop_shared_f32(int Vh) { return Vh <= kPairMaxF32; }

template <int PREC, bool DAG, int EPI, bool RED>
void launch_shared(const HopParams<PREC>& a, cudaStream_t st) {
  const int Vh = a.g.Vh;
  if constexpr (PREC != PFMP_F32) {
    if (Vh <= kTileMax) {
      launch_plain(k_hop_tile<PREC, DAG, EPI, RED>, nblocks(Vh, kTileSites), 16 * kTileSites, st, a);
      return;
    }
  }
  // the kernel loops over its site blocks, so the grid stays within the reduction buffer
  const int n = nblocks(Vh, kPairSites);
  const int blocks = n < kMaxReduceBlocks ? n : kMaxReduceBlocks;
  if constexpr (PREC == PFMP_F32)
    launch_chained(k_hop_pair<PREC, DAG, EPI, RED>, blocks, 8 * kPairSites, st, a);
  else
    launch_plain(k_hop_pair<PREC, DAG, EPI, RED>, blocks, 8 * kPairSites, st, a);
}

}  // namespace pfmp
