// Tensor-core inference of the gauge-covariant network 1 -> 8 -> ... -> 8 -> 1.
//
// A layer is a dense contraction per site and colour:
//   y[o][a](x, c) = sum_d sum_i sum_b W_d[o][i][a][b] t_d[i][b](x, c),
// t_d = the input channel parallel-transported from the neighbour in direction d (the
// site itself, four forward and four backward hops, fermion boundary factor included).
// As a real GEMM per colour: rows = 128 sites of one parity (M = 128, one TMEM lane each),
// K = directions x C_in channels x 4 spins x (re, im), N = C_out x 4 spins x (re, im)
// (padded to 16), with B = [[Re W, -Im W], [Im W, Re W]] so that the complex product
// comes out in (re, im) column pairs.  Operands are FP16, the accumulator FP32 in
// tensor memory; the transport itself is FP32 (links and products).
//
// The network input lives on even sites and its output is read there, so two of the layers
// are half empty:
//   first (1 -> 8)   even sites see only their own input, odd sites only their eight
//                    neighbours: one stage per tile, straight from the FP32 input field
//                    (k_nn_single<true>; nine direction slots of 8 columns, K = 16 or 80)
//   hidden (8 -> 8)  nine stages of K = 64, one direction each (k_nn_hidden)
//   last (8 -> 1)    the channels are mixed at every site first (the colour transport commutes
//                    with the weights): z_0 = W_0 a on even sites, z_d = W_d a for the eight
//                    hops on odd sites (k_nn_single<false>, K = 64), then out(x) = z_0(x) +
//                    sum_d U_d(x) z_d(x + d) on even sites in FP32 (k_nn_last)
// Activations between the layers are FP16, scaled by sigma = 1/rms of the network input so
// that FP16 keeps its precision (the network is linear; the last layer divides by sigma).
// Layout [parity][block of 32 sites][channel][12][32 sites], a complex number per word: the
// 96 words of a site lie at constant offsets (one address per neighbour) and a warp's 32
// neighbours touch one or two blocks.
//
// What bounds k_nn_hidden: instruction issue and the L2 gather (3.5 KB per site), not the
// tensor pipe.  The earlier kernel ran load -> transport -> barrier in lockstep (issue slots
// half idle, 196 us at 16^3x32).  Now eight warps gather (two threads per site, four channels
// each) and a ninth issues the MMAs: they meet only on mbarriers, a channel pair's registers
// are refilled for the next stage as soon as it is transported, two channels share one packed
// FP32 instruction (fma.rn.f32x2), the site's own stage is copied bit for bit, and a tile's
// accumulators are read two stages into the next tile (two sets in tensor memory).
// The rounding points and the order of the transport's products are fixed (transport_pair):
// an FP16 activation turns a change in the last bit of its FP32 value into one of 2^-11.
// One application of [1, 8, 8, 8, 1] at 16^3x32: 568 -> 319 us; per kernel (before): scale 9 (9),
// first layer 28 (61 with the embedding), hidden 115 (196), mixing 16 (39), last 12 (40).
// Tried and slower: sixteen gathering warps of 128 registers (150 us per hidden layer: the
// links' work doubles), eight warps with 255 registers that issue the MMAs themselves (155).
//
// Every mbarrier wait is bounded; on a timeout the kernel raises a device error flag,
// waits (bounded) for the work it has in flight, frees its tensor memory and returns.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "context.h"
#include "fields.cuh"
#include "mad.cuh"

namespace pfmp {
namespace tc {

constexpr int kM = 128;        // sites per tile = TMEM lanes
constexpr int kGather = 256;   // gathering threads: two per site
constexpr int kWords = 96;     // complex words of a site's activations (8 channels)
constexpr int kSiteBlock = 32; // sites per activation block
constexpr int kCh = 8;         // hidden channels
constexpr int kK = 8 * kCh;    // reals of one stage
constexpr int kATile = kM * kK * 2;  // A tile of one colour
constexpr int kABuf = 3 * kATile;

struct Hidden {
  static constexpr int NST = 9;
  static constexpr int N = 64;
  static constexpr int B_ST = N * kK * 2;
  static constexpr int B_ALL = NST * B_ST;
  static constexpr int SMEM = B_ALL + 2 * kABuf;
  static constexpr int SET = 3 * N;  // TMEM columns of one accumulator set
  static constexpr int TMEM_COLS = 512;  // two sets
  static_assert(2 * SET <= TMEM_COLS && SMEM <= 227 * 1024, "tile shape");
};
// the one-stage layers: A of 8 SLOTS columns (first: the site, eight hops, padding; last: the
// channels), B for the even and the odd sites
template <bool FIRST>
struct Single {
  static constexpr int KD = FIRST ? 80 : kK;        // columns of the A tile
  static constexpr int K_EVEN = FIRST ? 16 : kK;    // of them used on even sites
  static constexpr int N_EVEN = FIRST ? 64 : 16, N_ODD = 64;
  static constexpr int B_EVEN = N_EVEN * K_EVEN * 2, B_ODD = N_ODD * KD * 2;
  static constexpr int B_ALL = B_EVEN + B_ODD;
  static constexpr int A_TILE = kM * KD * 2;
  static constexpr int SMEM = B_ALL + 3 * A_TILE;
  static constexpr int TMEM_COLS = 256;  // two blocks per SM share the 512 columns
};

// stage order of the nine directions (0 = site, 1 + mu = forward, 5 + mu = backward)
__host__ __device__ __forceinline__ int dir_of(int i) {
  return i == 0 ? 0 : (i & 1 ? 1 + (i >> 1) : 5 + ((i - 1) >> 1));
}

__host__ __device__ __forceinline__ size_t act_blocks(int Vh) { return (size_t)(Vh + kSiteBlock - 1) / kSiteBlock; }

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of element (row r, column k) in a K-major no-swizzle tile with kdim columns
__host__ __device__ __forceinline__ uint32_t kmajor(int r, int k, int kdim) {
  return (uint32_t)((r >> 3) * (kdim / 8) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// shared-memory matrix descriptor: start >> 4, leading (K) byte offset >> 4, stride
// (8-row group) byte offset >> 4, version 1, no swizzle
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// instruction descriptor of kind::f16: D FP32, A and B FP16, both K-major, N >> 3, M >> 4
__host__ __device__ constexpr uint32_t idesc(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// bounded wait: polls that suspend for at most a microsecond each, given up after half a second
// (a lost completion cannot hang the GPU)
__device__ __forceinline__ unsigned long long timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(1000u)
      : "memory");
  return ok;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_poll(bar, parity)) return true;
  const unsigned long long t0 = timer_ns();
  while (timer_ns() - t0 < 500000000ull)
    if (mbar_poll(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("{\n .reg .b64 t;\n mbarrier.arrive.shared::cta.b64 t, [%0];\n}\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "r"(cols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          d_tmem),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
  __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// ---------------------------------------------------------------- packed weights
// [[Re w, -Im w], [Im w, Re w]] at (row n = output reals, column k = input reals)
__device__ __forceinline__ float b_entry(const float2 w, int n, int k) {
  const int ro = n & 1, ri = k & 1;
  return ro == ri ? w.x : (ro == 0 ? -w.y : w.y);
}
// hidden: nine stages [64 x 64], each a K-major canonical tile
__global__ void k_pack_hidden(const float2* __restrict__ W, __half* __restrict__ B) {
  using S = Hidden;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= S::NST * S::N * kK) return;
  const int st = i / (S::N * kK), n = i % (S::N * kK) / kK, k = i % kK;
  const int o = n >> 3, a = (n >> 1) & 3, ic = k >> 3, b = (k >> 1) & 3;
  const float v = b_entry(W[(((size_t)dir_of(st) * kCh + o) * kCh + ic) * 16 + a * 4 + b], n, k);
  B[(size_t)st * (S::B_ST / 2) + kmajor(n, k, kK) / 2] = __float2half_rn(v);
}
// first: column slot j holds direction dir_of(j) (slot 9 is padding, as is slot 1 on even
// sites); last: the rows of even sites are the direction 0 (rows 8.. padding), those of odd
// sites the hops 1..8
template <bool FIRST>
__global__ void k_pack_single(const float2* __restrict__ W, __half* __restrict__ B) {
  using S = Single<FIRST>;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= S::B_ALL / 2) return;
  const bool even = i < S::B_EVEN / 2;
  const int K = even ? S::K_EVEN : S::KD, e = even ? i : i - S::B_EVEN / 2;
  const int n = e / K, k = e % K;
  const int o = n >> 3, a = (n >> 1) & 3, j = k >> 3, b = (k >> 1) & 3;
  float v = 0.f;
  if (FIRST) {
    if (even ? j == 0 : j < 9) v = b_entry(W[((size_t)dir_of(j) * kCh + o) * 16 + a * 4 + b], n, k);
  } else {
    if (!even || o == 0) v = b_entry(W[((size_t)(even ? 0 : 1 + o) * kCh + j) * 16 + a * 4 + b], n, k);
  }
  B[(even ? 0 : S::B_EVEN / 2) + kmajor(n, k, K) / 2] = __float2half_rn(v);
}

// sigma = sqrt(n) / |in| (1 for a zero input) of an even FP32 field
__device__ __forceinline__ float sigma_of(double rr, int Vh) { return rr > 0 ? (float)sqrt(24.0 * Vh / rr) : 1.0f; }
__global__ void k_rms_scale(const float4* __restrict__ in, int Vh, ReduceBuf rb, float* sigma,
                            const int* __restrict__ skip) {
  if (skip && *skip) return;
  float st = 0.f;  // per-thread sum in FP32, across threads in FP64
  const long n = 6L * Vh;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const float4 v = in[i];
    st += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  double s[1] = {(double)st};
  double t[1];
  if (grid_sum<1>(s, rb, t)) *sigma = sigma_of(t[0], Vh);
}

// ---------------------------------------------------------------- transport
// a site of the tile: coordinates and lexicographic index
struct Site {
  int x[4], lex;
};
__device__ __forceinline__ Site site_at(const Geom& g, int cb, int p) {
  Site s;
  cb_coords(g, cb, p, s.x);
  s.lex = lex_index(g, s.x);
  return s;
}
// checkerboard index of the neighbour of stage i (1..8: +x, -x, +y, ...) and whether the hop
// crosses the time boundary
__device__ __forceinline__ int hop_site(const Geom& g, const Site& s, int i, bool& edge) {
  const int mu = (i - 1) >> 1;
  const bool fwd = i & 1;
  int xm = s.x[0], Lm = g.L[0], stride = 1;
  if (mu >= 1) xm = s.x[1], stride = g.L[0], Lm = g.L[1];
  if (mu >= 2) xm = s.x[2], stride *= g.L[1], Lm = g.L[2];
  if (mu == 3) xm = s.x[3], stride *= g.L[2], Lm = g.L[3];
  const bool wrap = xm == (fwd ? Lm - 1 : 0);
  edge = wrap && mu == 3;
  const int step = wrap ? -(Lm - 1) * stride : stride;
  return (s.lex + (fwd ? step : -step)) >> 1;
}
// rows 0 and 1 of the link of stage i seen from the site cb (index n: its neighbour)
__device__ __forceinline__ void load_link_raw(float4 l[3], const float4* __restrict__ U32, int Vh, int p, int i, int cb,
                                              int n) {
  const int mu = (i - 1) >> 1;
  const bool fwd = i & 1;
  const float4* f = U32 + (size_t)(((fwd ? p : 1 - p) * 4 + mu) * 3) * Vh + (fwd ? cb : n);
#pragma unroll
  for (int k = 0; k < 3; ++k) l[k] = __ldg(f + (size_t)k * Vh);
}
// the transport matrix f U or f U^dag, f = bc on hops across the time boundary, else 1
template <bool FWD>
__device__ __forceinline__ Mat3<float> transport_matrix(const float4 l[3], bool edge, float bc) {
  Mat3<float> L, M;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    L.m[(2 * k) / 3][(2 * k) % 3] = mk(l[k].x, l[k].y);
    L.m[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk(l[k].z, l[k].w);
  }
  reconstruct_row2(L);
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      M.m[r][c] = FWD ? L.m[r][c] : conj(L.m[c][r]);
    }
  if (edge) {
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) M.m[r][c] = bc * M.m[r][c];
  }
  return M;
}

// two FP32 numbers in one register pair: the same operation on both in one instruction
typedef unsigned long long f2x;
__device__ __forceinline__ f2x f2x_mk(float a, float b) {
  f2x r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f2x_get(f2x v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2x f2x_mul(f2x a, f2x b) {
  f2x r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2x f2x_fma(f2x a, f2x b, f2x c) {
  f2x r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2x f2x_add(f2x a, f2x b) {
  f2x r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
struct Mat3x2 {  // a transport matrix for two channels at once
  f2x re[3][3], im[3][3], ni[3][3];
};
__device__ __forceinline__ Mat3x2 pair_matrix(const Mat3<float>& M) {
  Mat3x2 P;
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      P.re[r][c] = f2x_mk(M.m[r][c].re, M.m[r][c].re);
      P.im[r][c] = f2x_mk(M.m[r][c].im, M.m[r][c].im);
      P.ni[r][c] = f2x_mk(-M.m[r][c].im, -M.m[r][c].im);
    }
  return P;
}
// M v for two spinor colour vectors at once (v0, v1: three FP16 colours each), back to FP16.
// Each complex product is rounded by itself (real part fma(re, re, -(im im)), imaginary part
// fma(im, re, re im)) and the three are added in order.
__device__ __forceinline__ void transport_pair(const Mat3x2& P, const uint32_t v0[3], const uint32_t v1[3], uint32_t o0[3],
                                               uint32_t o1[3]) {
  f2x re[3], im[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float2 a = h2_to_f2(v0[c]), b = h2_to_f2(v1[c]);
    re[c] = f2x_mk(a.x, b.x);
    im[c] = f2x_mk(a.y, b.y);
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    f2x x, y;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const f2x px = f2x_fma(P.re[r][c], re[c], f2x_mul(P.ni[r][c], im[c]));
      const f2x py = f2x_fma(P.im[r][c], re[c], f2x_mul(P.re[r][c], im[c]));
      x = c == 0 ? px : f2x_add(x, px);
      y = c == 0 ? py : f2x_add(y, py);
    }
    const float2 xr = f2x_get(x), yi = f2x_get(y);
    o0[r] = pack_h2(xr.x, yi.x);
    o1[r] = pack_h2(xr.y, yi.y);
  }
}
// the 12 words (spin, colour) of a spinor as 16-byte rows of the three colour tiles
__device__ __forceinline__ void store_row(unsigned char* A, int a_tile, uint32_t at, const uint32_t w[12]) {
#pragma unroll
  for (int r = 0; r < 3; ++r) *reinterpret_cast<uint4*>(A + r * a_tile + at) = make_uint4(w[r], w[3 + r], w[6 + r], w[9 + r]);
}

// first word of site c of parity q
__device__ __forceinline__ size_t act_at(int q, int c, size_t nb32) {
  return ((size_t)q * nb32 + c / kSiteBlock) * (kWords * kSiteBlock) + c % kSiteBlock;
}

// accumulators -> FP16 activations: TMEM lanes 32 (warp % 4) .., output channels 4 grp .. 4 grp
// + 3 of site cb (parity p); columns [colour][channel][spin][re, im]
__device__ __forceinline__ void store_act(uint32_t acc, int warp, __half2* __restrict__ out, int p, int cb, int Vh) {
  const int grp = warp >> 2, lane0 = (warp & 3) * 32;
  __half2* q = out + act_at(p, cb, act_blocks(Vh));
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float v[3][16];
#pragma unroll
    for (int r = 0; r < 3; ++r) tmem_ld16(acc + ((uint32_t)lane0 << 16) + r * 64 + grp * 32 + h * 16, v[r]);
    if (cb < Vh) {
#pragma unroll
      for (int o = 0; o < 2; ++o)
#pragma unroll
        for (int k = 0; k < 12; ++k)
          q[((4 * grp + 2 * h + o) * 12 + k) * kSiteBlock] =
              __floats2half2_rn(v[k % 3][o * 8 + (k / 3) * 2], v[k % 3][o * 8 + (k / 3) * 2 + 1]);
    }
  }
}

// ---------------------------------------------------------------- one-stage layers
// Per tile: gather, MMA, epilogue; two resident blocks per SM overlap each other's phases.
// Thread (row, half).  First layer: even sites, half 0 takes the site's spinor and half 1 the
// padding slot; odd sites, half h takes the hops of mu = 2 h and 2 h + 1.  The input is rounded
// to FP16 before the transport.  Last layer: half h copies the channels 4 h .. 4 h + 3; the
// output z has the layout of the activations, with the hop 1 + o in place of channel o on odd
// sites and z_0 in place of channel 0 on even ones.
// rr (first layer, optional): |in|^2 known to the caller (FGCR); sigma then comes from it and
// is stored for the last layer.
template <bool FIRST>
__global__ void __launch_bounds__(kGather, 2)
    k_nn_single(Geom g, const float4* __restrict__ U32, const __half* __restrict__ Bg, const void* __restrict__ in,
                __half2* __restrict__ out, float* __restrict__ sigma_p, const double* __restrict__ rr, int* __restrict__ err,
                const int* __restrict__ skip) {
  using S = Single<FIRST>;
  if (skip && *skip) return;  // block-uniform: nothing allocated yet
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) uint64_t bar_w, bar_m;
  unsigned char* sB = sm;
  unsigned char* A = sm + S::B_ALL;
  const int tid = threadIdx.x, row = tid & (kM - 1), half = tid >> 7, warp = tid >> 5;
  const int Vh = g.Vh;
  const float bcf = (float)g.bc_t;
  float sigma = 1.f;
  if (FIRST) {
    if (rr) {
      sigma = sigma_of(*rr, Vh);
      if (blockIdx.x == 0 && tid == 0) *sigma_p = sigma;
    } else {
      sigma = *sigma_p;
    }
  }
  if (tid == 0) {
    mbar_init(&bar_w, 1);
    mbar_init(&bar_m, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 32) tmem_alloc(&tmem_slot, S::TMEM_COLS);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot, barw = smem_addr(&bar_w), barm = smem_addr(&bar_m);
  if (tid == 0) {
    expect_tx(barw, S::B_ALL);
    bulk_load(sB, Bg, S::B_ALL, barw);
  }
  bool fail = !mbar_wait(barw, 0);
  if (fail) atomicExch(err, 1);
  // the abort decisions are block-uniform (__syncthreads_or of the threads' wait results)
  bool aborted = __syncthreads_or(fail);
  const int nt = (Vh + kM - 1) / kM;
  uint32_t n = 0;        // tiles done: parity of bar_m
  bool pending = false;  // MMAs committed and not waited for (thread 0)
  for (int t = blockIdx.x; t < 2 * nt && !aborted; t += gridDim.x, ++n) {
    const int p = t & 1, cb = (t >> 1) * kM + row;
    const int cs = cb < Vh ? cb : Vh - 1;  // rows past the end gather a valid site and are not stored
    if constexpr (!FIRST) {
      const uint32_t* w = (const uint32_t*)in + act_at(p, cs, act_blocks(Vh)) + half * (48 * kSiteBlock);
      uint32_t raw[4][12];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 12; ++k) raw[c][k] = __ldg(w + (c * 12 + k) * kSiteBlock);
#pragma unroll
      for (int c = 0; c < 4; ++c) store_row(A, S::A_TILE, kmajor(row, (4 * half + c) * 8, S::KD), raw[c]);
    } else {
      auto spinor16 = [&](int site, uint32_t w[12]) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const float4 v = __ldg((const float4*)in + (size_t)k * Vh + site);
          w[2 * k] = pack_h2(sigma * v.x, sigma * v.y);
          w[2 * k + 1] = pack_h2(sigma * v.z, sigma * v.w);
        }
      };
      uint32_t w[12];
      if (p == 0 && half == 0) {
        spinor16(cs, w);
      } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) w[k] = 0;
      }
      // even: slot 0 the site, slot 1 zero; odd: slots 0 and 9 zero
      store_row(A, S::A_TILE, kmajor(row, (half == 0 ? 0 : (p == 0 ? 1 : 9)) * 8, S::KD), w);
      if (p == 1) {
        const Site s = site_at(g, cs, 1);
        auto hop = [&](auto fwd, int i) {
          bool edge;
          const int nb = hop_site(g, s, i, edge);
          float4 l[3];
          load_link_raw(l, U32, Vh, 1, i, cs, nb);
          spinor16(nb, w);
          const Mat3x2 P = pair_matrix(transport_matrix<decltype(fwd)::value>(l, edge, bcf));
          transport_pair(P, w, w + 3, w, w + 3);
          transport_pair(P, w + 6, w + 9, w + 6, w + 9);
          store_row(A, S::A_TILE, kmajor(row, i * 8, S::KD), w);
        };
#pragma unroll 1
        for (int i = 4 * half + 1; i < 4 * half + 5; i += 2) {
          hop(std::true_type(), i);
          hop(std::false_type(), i + 1);
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    fence_before();
    __syncthreads();
    if (tid == 0) {
      fence_after();
      const uint32_t b0 = smem_addr(sB + (p ? S::B_EVEN : 0));
      const int K = p ? S::KD : S::K_EVEN;
      const uint32_t id = idesc(kM, p ? S::N_ODD : S::N_EVEN);
      for (int r = 0; r < 3; ++r) {
        const uint32_t a0 = smem_addr(A + r * S::A_TILE);
        for (int kk = 0; kk < K / 16; ++kk)
          mma_f16(tmem + r * 64, sdesc(a0 + kk * 256, 128, 16 * S::KD), sdesc(b0 + kk * 256, 128, 16 * K), id, kk > 0);
      }
      mma_commit(barm);
      pending = true;
    }
    fail = !mbar_wait(barm, n & 1);
    if (fail) atomicExch(err, 2);
    aborted = __syncthreads_or(fail);
    if (aborted) break;
    pending = false;
    fence_after();
    const int c = (t >> 1) * kM + (warp & 3) * 32 + (tid & 31);
    if (FIRST || p == 1) {
      store_act(tmem, warp, out, p, c, Vh);
    } else if (warp < 4) {
      float v[3][16];
#pragma unroll
      for (int r = 0; r < 3; ++r) tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + r * 64, v[r]);
      if (c < Vh) {
        __half2* q = out + act_at(0, c, act_blocks(Vh));
#pragma unroll
        for (int k = 0; k < 12; ++k) q[k * kSiteBlock] = __floats2half2_rn(v[k % 3][(k / 3) * 2], v[k % 3][(k / 3) * 2 + 1]);
      }
    }
    fence_before();
    __syncthreads();
  }
  if (tid == 0 && pending) mbar_wait(barm, n & 1);
  fence_before();
  __syncthreads();
  fence_after();
  if (tid < 32) tmem_free(tmem, S::TMEM_COLS);
}

// The network's output on even sites, out(x) = (z_0(x) + sum_d U_d(x) z_d(x + d)) / sigma: a
// block takes 32 sites, warp mu both hops of direction mu (48 words in flight per thread where
// one thread per site looped over the hops: 40 us at 16^3x32), the sums meet in shared memory.
__global__ void __launch_bounds__(128) k_nn_last(Geom g, const float4* __restrict__ U32, const uint32_t* __restrict__ z,
                                                 float4* __restrict__ out, const float* __restrict__ sigma_p,
                                                 const int* __restrict__ skip) {
  if (skip && *skip) return;
  __shared__ float2 sh[4][12][32];
  const int lane = threadIdx.x & 31, mu = threadIdx.x >> 5;
  const int cb = blockIdx.x * 32 + lane, Vh = g.Vh, cs = cb < Vh ? cb : Vh - 1;
  const size_t nb32 = act_blocks(Vh);
  const Site s = site_at(g, cs, 0);
  const float bcf = (float)g.bc_t;
  uint32_t w[2][12];
  float4 l[2][3];
  bool edge[2];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const int i = 2 * mu + 1 + b;  // stage: +mu, -mu
    const int nb = hop_site(g, s, i, edge[b]);
    const uint32_t* q = z + act_at(1, nb, nb32) + (dir_of(i) - 1) * (12 * kSiteBlock);
#pragma unroll
    for (int k = 0; k < 12; ++k) w[b][k] = __ldg(q + k * kSiteBlock);
    load_link_raw(l[b], U32, Vh, 0, i, cs, nb);
  }
  cplx<float> acc[12];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const Mat3<float> M = b == 0 ? transport_matrix<true>(l[b], edge[b], bcf) : transport_matrix<false>(l[b], edge[b], bcf);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const int sp = k / 3, r = k % 3;
      cplx<float> y = b ? acc[k] : mk(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float2 v = h2_to_f2(w[b][3 * sp + c]);
        y = cmad(M.m[r][c], mk(v.x, v.y), y);
      }
      acc[k] = y;
    }
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) sh[mu][k][lane] = make_float2(acc[k].re, acc[k].im);
  __syncthreads();
  const float inv = 1.0f / *sigma_p;
  for (int j = mu; j < 6; j += 4) {  // components 2 j, 2 j + 1
    float2 o[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int k = 2 * j + e;
      o[e] = h2_to_f2(__ldg(z + act_at(0, cs, nb32) + k * kSiteBlock));
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        o[e].x += sh[m][k][lane].x;
        o[e].y += sh[m][k][lane].y;
      }
    }
    if (cb < Vh) out[(size_t)j * Vh + cb] = make_float4(inv * o[0].x, inv * o[0].y, inv * o[1].x, inv * o[1].y);
  }
}

// ---------------------------------------------------------------- hidden layer
// Warps 0-7 gather and transport (thread (row, half): channels 4 half .. 4 half + 3), warp 8
// issues the MMAs.  Per stage: wait until the A buffer is free (MMAs of two stages before),
// transport the prefetched words into it and refill their registers for the next stage (the
// next tile's first stage after the ninth), arrive on full.  Rows past the end of the lattice
// gather the last site and are not stored.
__global__ void __launch_bounds__(kGather + 32, 1)
    k_nn_hidden(Geom g, const float4* __restrict__ U32, const __half* __restrict__ Bg, const uint32_t* __restrict__ in,
                __half2* __restrict__ out, int* __restrict__ err, const int* __restrict__ skip) {
  using S = Hidden;
  if (skip && *skip) return;  // block-uniform: nothing allocated yet
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(8) uint64_t bar_w, bar_full[2], bar_free[2], bar_acc[2], bar_read[2];
  unsigned char* sB = sm;
  unsigned char* sA = sm + S::B_ALL;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int Vh = g.Vh;
  if (tid == 0) {
    mbar_init(&bar_w, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bar_full[b], kGather / 32);
      mbar_init(&bar_free[b], 1);
      mbar_init(&bar_acc[b], 1);
      mbar_init(&bar_read[b], kGather / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 32) tmem_alloc(&tmem_slot, S::TMEM_COLS);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;
  const int ntiles = 2 * ((Vh + kM - 1) / kM);  // parity t & 1

  if (warp == kGather / 32) {
    // ---- MMA issue: one thread
    if ((tid & 31) == 0) {
      const uint32_t barw = smem_addr(&bar_w);
      expect_tx(barw, S::B_ALL);
      for (int st = 0; st < S::NST; ++st)
        bulk_load(sB + st * S::B_ST, Bg + (size_t)st * (S::B_ST / 2), S::B_ST, barw);
      bool ok = mbar_wait(barw, 0);
      const uint32_t id = idesc(kM, S::N);
      uint32_t use = 0, i = 0;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
        const uint32_t set = i & 1;
        if (i >= 2) ok = mbar_wait(smem_addr(&bar_read[set]), ((i >> 1) - 1) & 1);
        for (int st = 0; st < S::NST && ok; ++st) {
          const uint32_t buf = use & 1;
          ok = mbar_wait(smem_addr(&bar_full[buf]), (use >> 1) & 1);
          if (!ok) break;
          fence_after();
          const uint32_t b0 = smem_addr(sB + st * S::B_ST);
#pragma unroll 1
          for (int r = 0; r < 3; ++r) {
            const uint32_t a0 = smem_addr(sA + buf * kABuf + r * kATile);
#pragma unroll
            for (int kk = 0; kk < kK / 16; ++kk)
              mma_f16(tmem + set * S::SET + r * S::N, sdesc(a0 + kk * 256, 128, 16 * kK), sdesc(b0 + kk * 256, 128, 16 * kK),
                      id, (st > 0 || kk > 0) ? 1u : 0u);
          }
          mma_commit(smem_addr(&bar_free[buf]));
          ++use;
        }
        if (ok) mma_commit(smem_addr(&bar_acc[set]));
      }
      if (!ok) atomicExch(err, 2);
      // nothing may still be running on the tensor core when its memory is freed
      for (uint32_t b = 0; b < 2; ++b)
        if (use > b) mbar_wait(smem_addr(&bar_free[(use - 1 - b) & 1]), ((use - 1 - b) >> 1) & 1);
    }
  } else {
    // ---- gather and transport
    const int row = tid & (kM - 1), half = tid >> 7;
    const size_t nb32 = act_blocks(Vh);
    const float bcf = (float)g.bc_t;
    uint32_t raw[4][12];
    float4 link[3];
    bool edge = false, ok = true;
    int tile = blockIdx.x;
    Site s{};
    int p = 0, cb = 0;
    auto place = [&](int t) {  // the row's site in tile t
      p = t & 1;
      const int c = (t >> 1) * kM + row;
      cb = c < Vh ? c : Vh - 1;
      s = site_at(g, cb, p);
    };
    auto words = [&](int q, int c) {  // activations of this half's channels at site c of parity q
      return in + act_at(q, c, nb32) + half * (48 * kSiteBlock);
    };
    // accumulators of this block's tile number i (tile index t) -> output
    auto epilogue = [&](uint32_t i, int t) {
      const uint32_t set = i & 1;
      ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&bar_acc[set]), (i >> 1) & 1));
      if (!ok) return;
      fence_after();
      store_act(tmem + set * S::SET, warp, out, t & 1, (t >> 1) * kM + (warp & 3) * 32 + (tid & 31), Vh);
      fence_before();
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(smem_addr(&bar_read[set]));
    };
    if (tile < ntiles) {
      place(tile);
      const uint32_t* w = words(p, cb);
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 12; ++k) raw[c][k] = __ldg(w + (c * 12 + k) * kSiteBlock);
    }
    uint32_t use = 0, i = 0;
    // stage st of the tile; KIND: 0 the site itself, 1 a forward hop, 2 a backward hop
    auto stage = [&](auto kind, int st) {
      constexpr int KIND = decltype(kind)::value;
      const uint32_t buf = use & 1;
      if (use >= 2) ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&bar_free[buf]), ((use >> 1) - 1) & 1));
      if (!ok) return;
      Mat3x2 P;
      if constexpr (KIND != 0) P = pair_matrix(transport_matrix<KIND == 1>(link, edge, bcf));
      // where the next stage reads: the next hop of this site, or the next tile's own site
      int nx = cb, np = p;
      if (KIND != 2 || st + 1 < S::NST) {
        nx = hop_site(g, s, st + 1, edge);
        np = 1 - p;
        load_link_raw(link, U32, Vh, p, st + 1, cb, nx);
      } else if (tile + (int)gridDim.x < ntiles) {
        place(tile + gridDim.x);
        nx = cb;
        np = p;
      }
      const uint32_t* w = words(np, nx);
      unsigned char* A = sA + buf * kABuf;
#pragma unroll
      for (int c = 0; c < 4; c += 2) {
        if constexpr (KIND != 0) {
#pragma unroll
          for (int sp = 0; sp < 4; ++sp) transport_pair(P, &raw[c][3 * sp], &raw[c + 1][3 * sp], &raw[c][3 * sp], &raw[c + 1][3 * sp]);
        }
#pragma unroll
        for (int q = c; q < c + 2; ++q) store_row(A, kATile, kmajor(row, (4 * half + q) * 8, kK), raw[q]);
#pragma unroll
        for (int q = c; q < c + 2; ++q)
#pragma unroll
          for (int k = 0; k < 12; ++k) raw[q][k] = __ldg(w + (q * 12 + k) * kSiteBlock);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if ((tid & 31) == 0) mbar_arrive(smem_addr(&bar_full[buf]));
      ++use;
    };
    for (; tile < ntiles && ok; tile += gridDim.x, ++i) {
      stage(std::integral_constant<int, 0>(), 0);
#pragma unroll 1
      for (int st = 1; st < S::NST && ok; st += 2) {
        stage(std::integral_constant<int, 1>(), st);
        if (st == 1 && ok && i > 0) epilogue(i - 1, tile - gridDim.x);
        if (ok) stage(std::integral_constant<int, 2>(), st + 1);
      }
    }
    if (ok && i > 0) epilogue(i - 1, tile - gridDim.x);
    if (!ok && (tid & 31) == 0) atomicExch(err, 3);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (tid < 32) tmem_free(tmem, S::TMEM_COLS);
}

}  // namespace tc

// ---------------------------------------------------------------- host side
// networks 1 -> 8 -> ... -> 8 -> 1: layers (1, 8), (8, 8), (8, 1)
bool nn_tc_supported(int cin, int cout) {
  return (cin == 1 && cout == 8) || (cin == 8 && cout == 8) || (cin == 8 && cout == 1);
}

size_t nn_tc_packed_bytes(int cin, int cout) {
  if (cin == 1) return tc::Single<true>::B_ALL;
  return cout == 1 ? tc::Single<false>::B_ALL : tc::Hidden::B_ALL;
}

// activations of 8 channels between two layers
size_t nn_tc_act_bytes(const Geom& g) { return 2 * tc::act_blocks(g.Vh) * tc::kWords * tc::kSiteBlock * 4; }

void nn_tc_pack(pfmp_ctx* c, int cin, int cout, const void* W, void* Bp) {
  const float2* w = (const float2*)W;
  __half* B = (__half*)Bp;
  if (cin == 1)
    tc::k_pack_single<true><<<nblocks(tc::Single<true>::B_ALL / 2), kBlock, 0, c->stream>>>(w, B);
  else if (cout == 1)
    tc::k_pack_single<false><<<nblocks(tc::Single<false>::B_ALL / 2), kBlock, 0, c->stream>>>(w, B);
  else
    tc::k_pack_hidden<<<nblocks(tc::Hidden::B_ALL / 2), kBlock, 0, c->stream>>>(w, B);
  PFMP_CHECK_LAUNCH();
}

void nn_tc_scale(pfmp_ctx* c, const void* in_even_f32, float* sigma_dev, const int* skip) {
  const long n = 6L * c->g.Vh;
  long b = (n + kBlock - 1) / kBlock;
  const int grid = (int)(b < 152 * 4 ? b : 152 * 4);
  tc::k_rms_scale<<<grid, kBlock, 0, c->stream>>>((const float4*)in_even_f32, c->g.Vh, c->rb, sigma_dev, skip);
  PFMP_CHECK_LAUNCH();
}

// kernel attributes set outside any stream capture; returns the number of SMs
int nn_tc_init() {
  static const int sms = [] {
    auto smem = [](auto* k, int bytes) {
      PFMP_CUDA(cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    };
    smem(tc::k_nn_single<true>, tc::Single<true>::SMEM);
    smem(tc::k_nn_single<false>, tc::Single<false>::SMEM);
    smem(tc::k_nn_hidden, tc::Hidden::SMEM);
    int dev = 0, n = 0;
    PFMP_CUDA(cudaGetDevice(&dev));
    PFMP_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    return n;
  }();
  return sms;
}

static int parity_tiles(const pfmp_ctx* c) { return 2 * nblocks(c->g.Vh, tc::kM); }

// in (even FP32) -> FP16 activations; sigma is read, or with rr (|in|^2) set
void nn_tc_first(pfmp_ctx* c, const void* Bp, const void* in, void* act, float* sigma, const double* rr, int* err,
                 const int* skip) {
  const int grid = std::min(parity_tiles(c), 2 * nn_tc_init());
  tc::k_nn_single<true><<<grid, tc::kGather, tc::Single<true>::SMEM, c->stream>>>(
      c->g, c->U32, (const __half*)Bp, in, (__half2*)act, sigma, rr, err, skip);
  PFMP_CHECK_LAUNCH();
}
void nn_tc_hidden(pfmp_ctx* c, const void* Bp, const void* in, void* out, int* err, const int* skip) {
  const int grid = std::min(parity_tiles(c), nn_tc_init());
  tc::k_nn_hidden<<<grid, tc::kGather + 32, tc::Hidden::SMEM, c->stream>>>(c->g, c->U32, (const __half*)Bp,
                                                                           (const uint32_t*)in, (__half2*)out, err, skip);
  PFMP_CHECK_LAUNCH();
}
// FP16 activations -> out (even FP32), divided by sigma; z: room for one set of activations
void nn_tc_last(pfmp_ctx* c, const void* Bp, const void* in, void* z, void* out, float* sigma, int* err, const int* skip) {
  const int grid = std::min(parity_tiles(c), 2 * nn_tc_init());
  tc::k_nn_single<false><<<grid, tc::kGather, tc::Single<false>::SMEM, c->stream>>>(
      c->g, c->U32, (const __half*)Bp, in, (__half2*)z, sigma, nullptr, err, skip);
  PFMP_CHECK_LAUNCH();
  tc::k_nn_last<<<nblocks(c->g.Vh, 32), 128, 0, c->stream>>>(c->g, c->U32, (const uint32_t*)z, (float4*)out, sigma, skip);
  PFMP_CHECK_LAUNCH();
}

}  // namespace pfmp
