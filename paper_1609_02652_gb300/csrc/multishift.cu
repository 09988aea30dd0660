// Multi-shift CG with complex shifts and the Chebyshev polynomial filter.
//
// Multi-shift CG (the solver the paper pairs with the filter correction term, Sec. 3.1
// and App. C eq. force_polycorr): x_s = (K + sigma_s)^{-1} b for every shift from the
// Krylov space of the seed system K.  The shifted residuals stay collinear with the
// seed residual, r_s = zeta_s r, with the recurrences (Jegerlehner, hep-lat/9612014)
//   zeta_s' = zeta_s zeta_s^- a^- / [a^- zeta_s^- (1 + a sigma_s) + a b^- (zeta_s^- - zeta_s)]
//   alpha_s = a zeta_s' / zeta_s,  beta_s = b (zeta_s' / zeta_s)^2,
//   x_s += alpha_s p_s,  p_s = zeta_s' r + beta_s p_s,
// where a, b are the seed CG's alpha, beta and ^- marks the previous iteration.  All
// scalars live on the device (FP64); one iteration is K (the reduction finisher writes
// a), the seed residual (whose last block writes b and, one thread per shift, the shifts'
// coefficients and which of them have converged) and the seed direction.  The shifts'
// vectors wait: the residuals of up to kMsBlock iterations are kept, and ONE pass then
// carries every shift still running through all of them, so that its x_s and p_s cross
// memory once per block instead of once per iteration.  A shift whose residual
// |zeta_s| |r| is below tol |b| takes this iteration's x update and then stops: the
// large shifts of a Chebyshev filter converge in a fraction of the seed's iterations,
// and their vectors leave the memory traffic.  The loop ends when every shift has
// converged (the seed system itself need not be one of them).
//
// Vectors (solutions, directions, seed residual) are FP64, or FP32 for the solves inside
// the MD forces (K on the FP32 stencil, FP64 global sums and scalars): a deterministic
// force needs no FP64 solve, and the trajectory's end actions stay FP64.
//
// Polynomial (App. A): P_n(K) v = a_n prod_{k=1}^{n} (K - z_k) v, roots
// z_k = mu (1 - cos t_k) - i sqrt(mu^2 - nu^2) sin t_k, t_k = 2 pi k/(n+1),
// a_n = 1/(mu prod_k (mu - z_k)); each factor is one K application and a complex axpby.
// R(K) = sqrt(a_n) prod_{Im z_k < 0} (K - z_k) (P = R^dag R for even n), R^dag with the
// conjugate roots.  The factors commute; they are applied in bit-reversed index order
// (stable_order), which keeps every partial product within a few orders of magnitude of
// the final one (in index order the partial products of P_64 reach 1e11 times it, and
// the rounding of each factor is amplified accordingly).
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "context.h"
#include "fields.cuh"

namespace pfmp {

constexpr int kMsBlock = 8;  // iterations per pass over the shifts' vectors
constexpr int kMsUpdX = 1, kMsUpdP = 2;
struct MSShift {
  double2 sigma;
  double2 zeta, zeta_next;  // of the previous iteration and of this one
  int keep;                 // still running after this iteration
  // the block's iterations: x_s += alpha p_s (kMsUpdX), p_s = zeta r + beta p_s (kMsUpdP)
  double2 alpha[kMsBlock], zn[kMsBlock], beta[kMsBlock];
  int upd[kMsBlock];
};
struct MSSeed {
  double alpha_prev, beta_prev;
  int nact;        // shifts active in the block's first iteration, listed in act[]
  int count;       // iterations of the block that ran
  int ns;          // shifts of this solve
};

__device__ __forceinline__ double2 cm(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  const double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 cs(double s, double2 a) { return make_double2(s * a.x, s * a.y); }

// complex words of a vector field: double2 = one complex number, float4 = two
__device__ __forceinline__ double2 axpy_c(double2 a, double2 x, double2 y) {
  return make_double2(fma(-a.y, x.y, fma(a.x, x.x, y.x)), fma(a.y, x.x, fma(a.x, x.y, y.y)));
}
// a x + b y
__device__ __forceinline__ double2 axpby_c(double2 a, double2 x, double2 b, double2 y) { return axpy_c(a, x, cm(b, y)); }
__device__ __forceinline__ float4 axpby_c(double2 a, float4 x, double2 b, float4 y) {
  const float ar = (float)a.x, ai = (float)a.y, br = (float)b.x, bi = (float)b.y;
  return make_float4(ar * x.x - ai * x.y + br * y.x - bi * y.y, ar * x.y + ai * x.x + br * y.y + bi * y.x,
                     ar * x.z - ai * x.w + br * y.z - bi * y.w, ar * x.w + ai * x.z + br * y.w + bi * y.z);
}
__device__ __forceinline__ double2 sub_real(double2 r, double a, double2 q) { return make_double2(r.x - a * q.x, r.y - a * q.y); }
__device__ __forceinline__ float4 sub_real(float4 r, double ad, float4 q) {
  const float a = (float)ad;
  return make_float4(r.x - a * q.x, r.y - a * q.y, r.z - a * q.z, r.w - a * q.w);
}
__device__ __forceinline__ double nrm(double2 v) { return v.x * v.x + v.y * v.y; }
__device__ __forceinline__ double nrm(float4 v) { return (double)(v.x * v.x + v.y * v.y) + (double)(v.z * v.z + v.w * v.w); }
// |v|^2 added to a thread's running sum
struct NormSum64 {
  double t = 0.0;
  __device__ __forceinline__ void add(double2 v) { t += nrm(v); }
  __device__ __forceinline__ bool ok() const { return true; }
  __device__ __forceinline__ double value() const { return t; }
};
struct NormSum32 {
  TripleSum t;
  __device__ __forceinline__ void add(float4 v) {
    t.add(v.x * v.x + v.y * v.y);
    t.add(v.z * v.z + v.w * v.w);
  }
  __device__ __forceinline__ bool ok() const { return t.ok(); }
  __device__ __forceinline__ double value() const { return t.value(); }
};
template <typename V>
struct NormOf {
  using type = NormSum64;
};
template <>
struct NormOf<float4> {
  using type = NormSum32;
};
__device__ __forceinline__ double2 xpby_real(double2 r, double b, double2 p) { return make_double2(r.x + b * p.x, r.y + b * p.y); }
__device__ __forceinline__ float4 xpby_real(float4 r, double bd, float4 p) {
  const float b = (float)bd;
  return make_float4(r.x + b * p.x, r.y + b * p.y, r.z + b * p.z, r.w + b * p.w);
}

// seed residual r = r_prev - alpha Ap, |r|^2 (r, r_prev: neighbouring slots of the block's
// residuals; this is iteration `slot` of the block).  The last block then takes one thread
// per shift: the zetas move on, zeta_next and alpha_s from the seed's alpha and the previous
// alpha, beta, the direction coefficients, and whether the shift keeps running
// (|zeta_s'|^2 |r|^2 >= stop); the solve is done when none does.  (One thread doing this for
// every shift in turn cost 10-25 us an iteration, FP64 divisions in a serial chain: the
// kernel at 24^3x48 with 13 shifts 41 -> 27 us.)
template <typename V>
__global__ void k_ms_r(V* __restrict__ r, const V* r_prev, const V* Ap, long n, ReduceBuf rb,
                       CGScalars* s, MSSeed* sd, MSShift* sh, int* act, int slot, bool chained) {
  chain_enter(chained);
  if (s->done) {  // a block that starts after the end has no iterations
    if (slot == 0 && blockIdx.x == 0 && threadIdx.x == 0) sd->count = 0;
    return;
  }
  const double al = s->alpha;
  typename NormOf<V>::type acc;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const V rr = sub_real(ld_live(r_prev + i), al, ld_live(Ap + i));
    r[i] = rr;
    acc.add(rr);
  }
  double v[1] = {acc.value()};
  if (!acc.ok()) {
    v[0] = 0.0;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) v[0] += nrm(r[i]);
  }
  double t[1];
  if (!grid_sum_last<1>(v, rb, t)) return;
  __shared__ int wcount[kBlock / 32];
  const double rr0 = s->rr, stop = s->stop_rr, beta = t[0] / rr0;
  const double ap = sd->alpha_prev, bp = sd->beta_prev;
  const int ns = sd->ns;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int any = 0, listed = 0;
  for (int k0 = 0; k0 < ns; k0 += blockDim.x) {
    const int k = k0 + threadIdx.x;
    int on = 0, keep = 0;
    if (k < ns) {
      MSShift& S = sh[k];
      on = S.keep;
      if (on) {
        const double2 zp = S.zeta, z = S.zeta_next;  // this iteration's zeta_prev and zeta
        const double2 one_as = make_double2(1.0 + al * S.sigma.x, al * S.sigma.y);
        const double2 den = cadd(cs(ap, cm(zp, one_as)), cs(al * bp, csub(zp, z)));
        const double2 zn = cdiv(cs(ap, cm(z, zp)), den);
        const double2 q = cdiv(zn, z);
        keep = nrm(zn) * t[0] >= stop;
        S.zeta = z;
        S.zeta_next = zn;
        S.keep = keep;
        S.alpha[slot] = cs(al, q);
        S.zn[slot] = zn;
        S.beta[slot] = cs(beta, cm(q, q));
      }
      S.upd[slot] = on ? (keep ? kMsUpdX | kMsUpdP : kMsUpdX) : 0;
    }
    if (slot == 0) {  // list the block's shifts in ascending order
      const unsigned m = __ballot_sync(0xffffffffu, on);
      if (lane == 0) wcount[warp] = __popc(m);
      __syncthreads();
      int at = listed + __popc(m & ((1u << lane) - 1));
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        if (w < warp) at += wcount[w];
        listed += wcount[w];
      }
      if (on) act[at] = k;
    }
    any |= __syncthreads_or(keep);
  }
  if (threadIdx.x == 0) {
    sd->alpha_prev = al;
    sd->beta_prev = beta;
    if (slot == 0) sd->nact = listed;
    sd->count = slot + 1;
    s->beta = beta;
    s->rr = t[0];
    s->iter += 1;
    if (!any || !(t[0] == t[0])) s->done = 1;
  }
}

// seed direction p = r + beta p
template <typename V>
__global__ void k_ms_p(V* p, const V* r, long n, const CGScalars* s, bool chained) {
  chain_enter(chained);
  if (s->done) return;
  const double be = s->beta;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    p[i] = xpby_real(ld_live(r + i), be, ld_live(p + i));
}

// coefficients and fields of one shift in the arithmetic of its vectors
template <typename V>
struct MSCoef;
template <>
struct MSCoef<double2> {
  using C = double2;
  static __device__ __forceinline__ C make(double2 a) { return a; }
};
template <>
struct MSCoef<float4> {
  using C = float2;
  static __device__ __forceinline__ C make(double2 a) { return make_float2((float)a.x, (float)a.y); }
};
__device__ __forceinline__ float4 axpy_c(float2 a, float4 x, float4 y) {
  return make_float4(y.x + a.x * x.x - a.y * x.y, y.y + a.x * x.y + a.y * x.x, y.z + a.x * x.z - a.y * x.w,
                     y.w + a.x * x.w + a.y * x.z);
}
__device__ __forceinline__ float4 axpby_c(float2 a, float4 x, float2 b, float4 y) {
  return make_float4(a.x * x.x - a.y * x.y + b.x * y.x - b.y * y.y, a.x * x.y + a.y * x.x + b.x * y.y + b.y * y.x,
                     a.x * x.z - a.y * x.w + b.x * y.z - b.y * y.w, a.x * x.w + a.y * x.z + b.x * y.w + b.y * y.z);
}

// The shifts' pass: for every shift listed, the block's iterations in order,
// x_s += alpha_s p_s and p_s = zeta_s' r + beta_s p_s (the direction only while the shift
// keeps running), with r[slot] the residual of iteration `slot`.  Bound by the copy
// bandwidth: two vectors read and two written per shift and kMsBlock iterations (24^3x48,
// 13 FP32 shifts: 265 us an iteration at 0.97 of the bandwidth when the pass ran every
// iteration, 391 us for eight now).  Block row blockIdx.y takes every gridDim.y-th shift of the list
// (small lattices: the shifts are the parallelism).  The coefficients are converted once
// per block and held in shared memory.
constexpr int kMsTile = 16;
template <typename V>
struct MSRing {
  V* r[kMsBlock];
};
template <typename V>
__global__ void __launch_bounds__(kBlock) k_ms_xp(V* const* x, V* const* p, MSRing<V> ring, const MSShift* sh,
                                                  const int* act, const MSSeed* sd, long n, bool chained) {
  chain_enter(chained);
  using C = typename MSCoef<V>::C;
  const int cnt = sd->count;
  if (cnt == 0) return;
  __shared__ V* sx[kMsTile];
  __shared__ V* sp[kMsTile];
  __shared__ C ca[kMsTile][kMsBlock], cz[kMsTile][kMsBlock], cb[kMsTile][kMsBlock];
  __shared__ int up[kMsTile][kMsBlock];
  const int na = sd->nact, G = gridDim.y;
  const int mine = na > (int)blockIdx.y ? (na - 1 - (int)blockIdx.y) / G + 1 : 0;  // shifts of this row
  const long step = (long)gridDim.x * blockDim.x, i0 = blockIdx.x * (long)blockDim.x + threadIdx.x;
  for (int j0 = 0; j0 < mine; j0 += kMsTile) {
    const int m = mine - j0 < kMsTile ? mine - j0 : kMsTile;
    __syncthreads();
    for (int q = threadIdx.x; q < m * kMsBlock; q += blockDim.x) {
      const int j = q / kMsBlock, b = q % kMsBlock, k = act[(j0 + j) * G + blockIdx.y];
      if (b == 0) {
        sx[j] = x[k];
        sp[j] = p[k];
      }
      up[j][b] = b < cnt ? sh[k].upd[b] : 0;
      ca[j][b] = MSCoef<V>::make(sh[k].alpha[b]);
      cz[j][b] = MSCoef<V>::make(sh[k].zn[b]);
      cb[j][b] = MSCoef<V>::make(sh[k].beta[b]);
    }
    __syncthreads();
    for (long i = i0; i < n; i += step) {
      V rr[kMsBlock];
#pragma unroll
      for (int b = 0; b < kMsBlock; ++b)
        if (b < cnt) rr[b] = ld_live(ring.r[b] + i);
#pragma unroll 2
      for (int j = 0; j < m; ++j) {
        V pk = ld_live(sp[j] + i), xk = ld_live(sx[j] + i);
        int last = 0;
#pragma unroll
        for (int b = 0; b < kMsBlock; ++b) {
          const int u = up[j][b];
          if (u) {
            xk = axpy_c(ca[j][b], pk, xk);
            if (u & kMsUpdP) pk = axpby_c(cz[j][b], rr[b], cb[j][b], pk);
            last = u;
          }
        }
        sx[j][i] = xk;
        if (last & kMsUpdP) sp[j][i] = pk;
      }
    }
  }
}

// y = a x + b y (complex a, b) on FP64 or FP32 even fields; with b = 0, y = a x without
// reading y (its previous contents may be anything, NaN included)
template <typename V>
__global__ void k_caxpby(double2 a, const V* x, double2 b, V* y, long n) {
  chain_enter();
  const bool read_y = b.x != 0.0 || b.y != 0.0;
  const double2 zero = make_double2(0.0, 0.0);
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const V xi = ld_live(x + i);
    y[i] = read_y ? axpby_c(a, xi, b, ld_live(y + i)) : axpby_c(a, xi, zero, xi);
  }
}

static int ms_grid(long n) {
  long b = (n + kBlock - 1) / kBlock;
  return (int)(b < 152 * 8 ? b : 152 * 8);
}
static long words(const Geom& g, int prec) { return (prec == PFMP_F64 ? 12L : 6L) * g.Vh; }

void caxpby(pfmp_ctx* c, int prec, std::complex<double> a, const void* x, std::complex<double> b, void* y) {
  const long n = words(c->g, prec);
  const double2 da = make_double2(a.real(), a.imag()), db = make_double2(b.real(), b.imag());
  if (prec == PFMP_F64)
    k_caxpby<double2><<<ms_grid(n), kBlock, 0, c->stream>>>(da, (const double2*)x, db, (double2*)y, n);
  else
    launch_chained(k_caxpby<float4>, ms_grid(n), kBlock, c->stream, da, (const float4*)x, db, (float4*)y, n);
  PFMP_CHECK_LAUNCH();
}
void caxpby(pfmp_ctx* c, std::complex<double> a, const void* x, std::complex<double> b, void* y) {
  caxpby(c, PFMP_F64, a, x, b, y);
}

// per-operator workspace for the shifted search directions and device scalar arrays
struct MSWork {
  std::vector<double2*> p;
  void** d_x = nullptr;
  void** d_p = nullptr;
  MSShift* d_sh = nullptr;
  MSSeed* d_seed = nullptr;
  int* d_act = nullptr;
  int cap = 0;
  std::vector<void*> ring[2];  // the block's residuals, FP64 and FP32
  ~MSWork() {
    for (auto q : p) dev_free(q);
    for (auto& v : ring)
      for (auto q : v) dev_free(q);
    dev_free(d_x);
    dev_free(d_p);
    dev_free(d_sh);
    dev_free(d_seed);
    dev_free(d_act);
  }
};

static MSWork& ms_work(pfmp_op* op, int ns, int prec) {
  if (!op->ms) op->ms = new MSWork();
  MSWork& w = *op->ms;
  if (w.cap < ns) {
    // a chunk's graph holds the arrays that are replaced here
    for (int g : {kGraphMs64, kGraphMs32})
      if (op->graph[g].exec) {
        cudaGraphExecDestroy(op->graph[g].exec);
        op->graph[g].exec = nullptr;
      }
    while ((int)w.p.size() < ns) w.p.push_back((double2*)dev_alloc(spinor_bytes(op->ctx->g, PFMP_F64)));
    dev_free(w.d_x);
    dev_free(w.d_p);
    dev_free(w.d_sh);
    dev_free(w.d_act);
    w.d_x = (void**)dev_alloc(ns * sizeof(void*));
    w.d_p = (void**)dev_alloc(ns * sizeof(void*));
    w.d_sh = (MSShift*)dev_alloc(ns * sizeof(MSShift));
    w.d_act = (int*)dev_alloc(ns * sizeof(int));
    if (!w.d_seed) w.d_seed = (MSSeed*)dev_alloc(sizeof(MSSeed));
    w.cap = ns;
  }
  auto& ring = w.ring[prec == PFMP_F64 ? 0 : 1];
  while ((int)ring.size() < kMsBlock) ring.push_back(dev_alloc(spinor_bytes(op->ctx->g, prec)));
  return w;
}

void ms_work_free(pfmp_op* op) {
  delete op->ms;
  op->ms = nullptr;
}

template <typename V>
static void ms_chunk(pfmp_op* op, int prec, MSWork& w, void* pseed, void* Ap, long n, int chunk) {
  pfmp_ctx* c = op->ctx;
  const bool chained = chain_launches(c->stream);
  MSRing<V> ring;
  for (int b = 0; b < kMsBlock; ++b) ring.r[b] = (V*)w.ring[prec == PFMP_F64 ? 0 : 1][b];
  // rows of shifts until the pass has about four blocks per SM; for as many shifts as the
  // workspace holds, so that a chunk serves solves with any number of them (the rows beyond
  // this solve's shifts end at once)
  const int nb = ms_grid(n), rows = std::max(1, std::min(w.cap, 152 * 4 / nb));
  for (int k = 0; k < chunk; ++k) {
    const int slot = k % kMsBlock;
    kop(op, prec, Ap, pseed, &op->scal->pAp, op->scal);
    // the residual before a chunk is in the last slot (every chunk but the last is whole blocks)
    const V* prev = ring.r[slot == 0 ? kMsBlock - 1 : slot - 1];
    launch_chained(k_ms_r<V>, nb, kBlock, c->stream, ring.r[slot], prev, (const V*)Ap, n, c->rb, op->scal, w.d_seed, w.d_sh,
                                            w.d_act, slot, chained);
    PFMP_CHECK_LAUNCH();
    launch_chained(k_ms_p<V>, nb, kBlock, c->stream, (V*)pseed, ring.r[slot], n, op->scal, chained);
    PFMP_CHECK_LAUNCH();
    if (slot == kMsBlock - 1 || k == chunk - 1) {
      launch_chained(k_ms_xp<V>, dim3(nb, rows), kBlock, c->stream, (V* const*)w.d_x, (V* const*)w.d_p, ring, w.d_sh, w.d_act,
                                                           w.d_seed, n, chained);
      PFMP_CHECK_LAUNCH();
    }
  }
}

// Up to this many sites per parity the kernels of an iteration are shorter than the
// host takes to launch them, and a chunk is replayed as a CUDA graph (recorded, not captured from
// a stream: other threads may synchronise the device meanwhile).  The graph depends on the
// workspace only, not on the solve's shifts: solves that alternate between numbers of shifts
// share it (with a graph made at each change of their number a solve of 0.21 ms took 0.35).
// A chunk cut short by the iteration cap is launched directly.
constexpr int kMsGraphMax = 32768;

// x[k] = (K + sigma_k)^{-1} b in FP64 or FP32 (x, b of precision prec).  Returns the
// status; iterations, K applications and (FP64, on request) the largest true residual.
int solve_multishift(pfmp_op* op, int prec, int ns, const std::complex<double>* sigma, void* const* x, const void* b,
                     double tol, int max_iter, int check, int* iters, double* max_true_res, long* kapply,
                     bool want_true_res) {
  pfmp_ctx* c = op->ctx;
  PFMP_REQUIRE(prec == PFMP_F64 || prec == PFMP_F32, PFMP_E_INVALID, "multi-shift CG: precision must be F64 or F32");
  PFMP_REQUIRE(ns >= 1 && ns <= 1024, PFMP_E_INVALID, "number of shifts must be in [1, 1024]");
  PFMP_REQUIRE(tol > 0 && max_iter > 0, PFMP_E_INVALID, "tol and max_iter must be positive");
  // K is Hermitian positive definite, so K + sigma is singular only for real sigma < 0
  // (at sigma = -lambda for an eigenvalue lambda of K); such shifts are refused
  for (int k = 0; k < ns; ++k) {
    PFMP_REQUIRE(std::isfinite(sigma[k].real()) && std::isfinite(sigma[k].imag()), PFMP_E_INVALID,
                 "multi-shift CG: a shift is not finite");
    PFMP_REQUIRE(!(sigma[k].imag() == 0.0 && sigma[k].real() < 0.0), PFMP_E_INVALID,
                 "multi-shift CG: a real negative shift can make K + sigma singular");
  }
  if (check <= 0) check = 8;
  check = (check + kMsBlock - 1) / kMsBlock * kMsBlock;  // whole blocks between host checks
  MSWork& w = ms_work(op, ns, prec);
  const size_t bytes = spinor_bytes(c->g, prec);
  const long n = words(c->g, prec);
  blas_norm2(c, prec, b, c->d_sums);
  PFMP_CUDA(cudaMemcpyAsync(c->h_sums, c->d_sums, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  PFMP_CUDA(cudaStreamSynchronize(c->stream));
  const double bb = c->h_sums[0];
  *iters = 0;
  *kapply = 0;
  *max_true_res = 0;
  for (int k = 0; k < ns; ++k) blas_zero(c, prec, x[k]);
  if (bb == 0.0) return PFMP_OK;
  PFMP_REQUIRE(std::isfinite(bb), PFMP_E_NAN, "right-hand side is not finite");
  void* r = w.ring[prec == PFMP_F64 ? 0 : 1][kMsBlock - 1];
  void* pseed = prec == PFMP_F64 ? (void*)op->cg64[1] : (void*)op->cg32[1];
  void* Ap = prec == PFMP_F64 ? (void*)op->cg64[2] : (void*)op->cg32[2];
  PFMP_CUDA(cudaMemcpyAsync(r, b, bytes, cudaMemcpyDeviceToDevice, c->stream));
  PFMP_CUDA(cudaMemcpyAsync(pseed, b, bytes, cudaMemcpyDeviceToDevice, c->stream));
  std::vector<void*> hx(ns), hp(ns);
  std::vector<MSShift> hs(ns);
  std::vector<int> act(ns);
  for (int k = 0; k < ns; ++k) {
    hx[k] = x[k];
    hp[k] = w.p[k];
    act[k] = k;
    PFMP_CUDA(cudaMemcpyAsync(w.p[k], b, bytes, cudaMemcpyDeviceToDevice, c->stream));
    MSShift s{};
    s.sigma = make_double2(sigma[k].real(), sigma[k].imag());
    s.zeta = s.zeta_next = make_double2(1.0, 0.0);
    s.keep = 1;
    hs[k] = s;
  }
  PFMP_CUDA(cudaMemcpyAsync(w.d_x, hx.data(), ns * sizeof(void*), cudaMemcpyHostToDevice, c->stream));
  PFMP_CUDA(cudaMemcpyAsync(w.d_p, hp.data(), ns * sizeof(void*), cudaMemcpyHostToDevice, c->stream));
  PFMP_CUDA(cudaMemcpyAsync(w.d_sh, hs.data(), ns * sizeof(MSShift), cudaMemcpyHostToDevice, c->stream));
  PFMP_CUDA(cudaMemcpyAsync(w.d_act, act.data(), ns * sizeof(int), cudaMemcpyHostToDevice, c->stream));
  MSSeed sd{1.0, 0.0, ns, 0, ns};
  PFMP_CUDA(cudaMemcpyAsync(w.d_seed, &sd, sizeof(MSSeed), cudaMemcpyHostToDevice, c->stream));
  CGScalars* h = op->h_scal;
  *h = CGScalars{};
  h->rr = bb;
  h->stop_rr = tol * tol * bb;
  PFMP_CUDA(cudaMemcpyAsync(op->scal, h, sizeof(CGScalars), cudaMemcpyHostToDevice, c->stream));
  int done = 0;
  const long long kapply0 = op->kapply;  // queued iterations after convergence do no work
  while (done < max_iter) {
    const int chunk = check < max_iter - done ? check : max_iter - done;
    auto launch = [&]() {
      if (prec == PFMP_F64)
        ms_chunk<double2>(op, prec, w, pseed, Ap, n, chunk);
      else
        ms_chunk<float4>(op, prec, w, pseed, Ap, n, chunk);
    };
    if (c->g.Vh <= kMsGraphMax && !c->prof.on && chunk == check) {
      const void* key[4] = {w.d_sh, w.d_x, w.d_p, w.d_act};
      run_recorded(op, op->graph[prec == PFMP_F64 ? kGraphMs64 : kGraphMs32], key, chunk, launch);
    } else {
      launch();
    }
    PFMP_CUDA(cudaMemcpyAsync(h, op->scal, sizeof(CGScalars), cudaMemcpyDeviceToHost, c->stream));
    PFMP_CUDA(cudaStreamSynchronize(c->stream));
    done = h->iter;
    PFMP_REQUIRE(std::isfinite(h->rr), PFMP_E_NAN, "multi-shift CG residual became NaN/Inf");
    if (h->done) break;
  }
  *iters = done;
  *kapply = done;
  op->kapply = kapply0 + done;
  if (want_true_res && prec == PFMP_F64) {
    // || b - (K + sigma) x || / ||b|| for every shift, FP64
    for (int k = 0; k < ns; ++k) {
      kop(op, PFMP_F64, Ap, x[k], nullptr, nullptr);
      caxpby(c, sigma[k], x[k], 1.0, Ap);      // Ap = (K + sigma) x
      blas_xmy_norm(c, b, Ap, r, c->d_sums);
      PFMP_CUDA(cudaMemcpyAsync(c->h_sums, c->d_sums, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
      PFMP_CUDA(cudaStreamSynchronize(c->stream));
      const double res = std::sqrt(c->h_sums[0] / bb);
      if (res > *max_true_res) *max_true_res = res;
      *kapply += 1;
    }
  }
  return h->done ? PFMP_OK : PFMP_E_NOT_CONVERGED;
}

// bit-reversed order of 0..n-1 (indices >= n skipped): a permutation that interleaves
// roots from all around the ellipse, so that no partial product is dominated by one
// side of it
std::vector<int> stable_order(int n) {
  int b = 0;
  while ((1 << b) < n) ++b;
  std::vector<int> o;
  for (int i = 0; i < (1 << b); ++i) {
    int r = 0;
    for (int k = 0; k < b; ++k)
      if (i & (1 << k)) r |= 1 << (b - 1 - k);
    if (r < n) o.push_back(r);
  }
  return o;
}

std::vector<std::complex<double>> stable_ordered(const std::vector<std::complex<double>>& z) {
  std::vector<std::complex<double>> o;
  for (int k : stable_order((int)z.size())) o.push_back(z[k]);
  return o;
}

// ------------------------------------------------------------------ polynomial
std::vector<std::complex<double>> cheb_roots(int n, double mu, double nu) {
  std::vector<std::complex<double>> z(n);
  const double b = std::sqrt(mu * mu - nu * nu);
  for (int k = 1; k <= n; ++k) {
    const double t = 2.0 * M_PI * k / (n + 1);
    z[k - 1] = std::complex<double>(mu * (1.0 - std::cos(t)), -b * std::sin(t));
  }
  return z;
}
double cheb_norm(int n, double mu, double nu) {
  auto z = cheb_roots(n, mu, nu);
  std::complex<double> p = mu;
  for (auto zk : z) p *= (mu - zk);
  return (1.0 / p).real();
}

// out = scale * prod_k (K - z_k) in, factors applied in the given order (callers pass
// stable_ordered lists); FP64
void poly_product(pfmp_op* op, const std::vector<std::complex<double>>& z, double scale, void* out, const void* in) {
  pfmp_ctx* c = op->ctx;
  const size_t bytes = spinor_bytes(c->g, PFMP_F64);
  void* w = op->cg64[2];
  PFMP_CUDA(cudaMemcpyAsync(out, in, bytes, cudaMemcpyDeviceToDevice, c->stream));
  for (auto zk : z) {
    kop(op, PFMP_F64, w, out, nullptr, nullptr);   // w = K out
    caxpby(c, 1.0, w, -zk, out);                    // out = K out - z out
  }
  if (scale != 1.0) caxpby(c, 0.0, out, scale, out);
}

}  // namespace pfmp
