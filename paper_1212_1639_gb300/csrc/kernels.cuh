// Kernels of the particle-learning cycle (sm_103a).
//
// One cycle for observation y = y_{t+1} (paper Section 2, Algorithm
// "Particle Learning"):
//   k_weights       l_i = log p(y | x_i, sigma_i^2, tau_i^2) + log(2 pi)/2, max_i l_i
//   k_sums, k_slots W_i = quantised exp(l_i - max), Q = inclusive scan of W
//                   (eq. resample.cdf as exact 64-bit integers), ancestors of
//                   systematic and stratified resampling, the cut-point table
//                   (slots.cuh; binary64: k_exp forms the exponentials first)
//   k_spacing_sums, k_multi_split, k_multi   multinomial ancestors
//                   a_j = #{i : Q_i * S_n <= S_j * T} (multi.cuh)
//   k_cutpoint_*    the paper's Section 3.2 algorithms (same ancestors)
//   k_propagate     gather ancestor, draw x, update b_sigma/b_tau, draw theta
//                   (binary32: k_propagate2)
//   k_estimate      posterior summaries on demand
// k_scan is the CDF alone, for given weights (one pass, decoupled look-back).
// A small filter's cycles are one cluster launch (small.cuh).
//
// Data layout in HBM (structure of arrays, one entry per particle):
//   x, sigma2, tau2 : R (binary32 or binary64), two ping-pong copies
//   b_sigma, b_tau  : uint64 2^-32 fixed point (FP32) / binary64 (FP64)
//   l               : R,    Q : uint64,   anc : uint32
#pragma once
#include <cstddef>
#include <cstdint>

#include "device.cuh"

namespace pfk {

constexpr int BLOCK = 256;
constexpr int WARPS = BLOCK / 32;
constexpr int CHUNK = 128;                 // elements per warp per chunk (4 per lane)
constexpr int CHUNKS = 4;                  // chunks per warp
constexpr int TILE = WARPS * CHUNKS * CHUNK;  // 4096 elements per scan tile

constexpr uint64_t FLAG_A = 1ull << 62;    // tile aggregate published
constexpr uint64_t FLAG_P = 2ull << 62;    // tile inclusive prefix published
constexpr uint64_t VAL_MASK = (1ull << 62) - 1;
constexpr uint32_t SPIN_LIMIT = 1u << 22;  // bounded look-back wait

enum ErrBits : uint32_t {
  ERR_TIMEOUT = 1u,   // look-back gave up
  ERR_NUMERIC = 2u,   // non-finite max, gamma sampler failure, b overflow
  ERR_WEIGHTS = 4u,   // negative / non-finite / all-zero input weights
};

// Per-filter control block in device memory.
struct Ctl {
  uint32_t t;             // cycles completed
  uint32_t err;           // ErrBits
  unsigned long long maxenc;  // order-encoded max of l (or of the input weights)
  uint32_t ticket_w;      // scan tile ticket
  uint32_t done_prop;     // last-block counter of k_propagate
  uint32_t done_est;      // last-block counter of k_estimate
  double logml;           // accumulated log marginal likelihood
  double est[8];          // t, x mean/var, sigma2 mean/var, tau2 mean/var, log_marglik
  // per-cycle constants written by k_weights (block 0) for k_propagate:
  double y;               // this cycle's observation y_{t+1}
  double mtd[6];          // Marsaglia-Tsang d, c for sigma^2 and tau^2 ([0..3]) and the
                          // squeeze coefficients K_sigma, K_tau ([4], [5]), binary64
  float yf;               // y rounded to binary32
  float mtf[6];           // the same constants rounded to binary32
  // resampling constants written by k_sums: T = Q_{n-1} and the systematic offset r
  uint64_t keyT, keyR;
  // the next cycle's maximum of l, gathered by a propagation that also
  // computes the next cycle's predictive weights (order-encoded, as maxenc)
  unsigned long long maxenc_nx;
  // adaptive resampling: this cycle's decision (written by k_sums) and
  // sum_i exp(lambda_i) of the carried log-weights (n after a resampling)
  uint32_t resamp;
  double slam;
  // binary32 propagation: the next unit of 64 slots to hand out
  unsigned long long prop_ticket;
  // weights kernel: the next round of WARPS chunks to hand out
  uint32_t w_ticket;
  // k_sums: last-block counter, and the slot map's constants (SlotMap)
  uint32_t done_sums;
  int32_t slot_z;
  uint64_t slot_rho, slot_r32;
  uint32_t heavy_count, heavy_chunks;
  // multinomial: last-block counter of k_spacing_sums, S_n, and the constants of
  // the slots' positions (k_multi_split)
  uint32_t done_spc;
  int32_t multi_z;
  uint64_t keyS, multi_rho, bucket_rho;
};

// Tile status words carry their value and flag in one aligned 64-bit word and
// nothing else is read through them, so relaxed (single-copy atomic) accesses
// suffice; unlike acquire loads, several can be in flight at once.
__device__ __forceinline__ void st_status(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t ld_status(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

template <class T>
__device__ __forceinline__ T shfl_up(T v, int d) {
  return __shfl_up_sync(0xffffffffu, v, d);
}
__device__ __forceinline__ uint64_t warp_incl_scan(uint64_t v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

// ---------------------------------------------------------------------------
// State views.
// ---------------------------------------------------------------------------
template <class R> struct SuffT;
template <> struct SuffT<float> { typedef uint64_t B; };
template <> struct SuffT<double> { typedef double B; };

template <class R>
struct StateV {
  R* x;
  R* s2;
  R* t2;
  typename SuffT<R>::B* bs;
  typename SuffT<R>::B* bt;
};

// Host-mapped words of a synchronous cycle with summaries (pf_step_estimate):
// the observation, and the host's sequence number, which the summary kernel
// copies to seq_out once the summaries are in the host mirror.
struct EstIO {
  double y;
  unsigned long long seq_in;
  unsigned long long seq_out;
  unsigned long long pad;
};

template <class R>
struct FilterArgs {
  StateV<R> st[2];          // ping-pong by cycle parity
  R* ell;
  uint64_t* Q;
  uint32_t* anc;
  uint32_t* I;              // cut-point table
  void* part;               // per-tile log-ML partial (U128 for FP32, double for FP64)
  double* part_est;         // per-block estimate partials
  Ctl* ctl;
  // device address of the handle's pinned host mirror of the control block
  // (mapped), or NULL: the summary kernels write the control block's summary
  // prefix there directly, so no copy follows them
  Ctl* ctl_mirror;
  EstIO* io;                // mapped words of pf_step_estimate, or NULL
  // this cycle's observation: *y_src when y_src is set (device-resident
  // observations), else y_val (set per launch in the graph's weights node)
  const double* y_src;
  double y_val;
  // the next cycle's observation y_{t+2}, for a propagation that computes
  // the next cycle's predictive weights (*y_nx_src when set, else y_nx_val)
  const double* y_nx_src;
  double y_nx_val;
  R* lam;                   // adaptive resampling: carried log-weights (NULL: resample every cycle)
  uint64_t n;
  uint32_t ntiles;
  uint32_t nparts;          // log-ML partials written this cycle (binary64: one per 4096 particles)
  int k;                    // CDF shift: W <= 2^k
  uint64_t seed;
  uint32_t filter;
  uint32_t rk[20];          // Philox round keys of seed (philox_rk)
  double x0_mean, x0_var, a_sigma, b_sigma, a_tau, b_tau, sigma2, tau2;
};

// ---------------------------------------------------------------------------
// Initialisation (Algorithm "Particle Learning", Step 0).
// ---------------------------------------------------------------------------
template <class R> struct SuffOps;
template <> struct SuffOps<float> {
  static __device__ __forceinline__ uint64_t from_prior(double b) {
    return __double2ull_rz(b * 0x1p32);
  }
  // b + r^2 / 2 in 2^-32 fixed point: trunc(r^2 2^31), which is
  // (r^2 / 2) 2^32 exactly; below 2^32 by one u32 truncation
  static __device__ __forceinline__ uint64_t incr(float v) {
    return v < 0x1p32f ? (uint64_t)__float2uint_rz(v) : f2u64_rz(v);
  }
  static __device__ __forceinline__ uint64_t add_half_square(uint64_t b, float r, bool* fail) {
    const float r2 = r * r;
    const float v = r2 * 0x1p31f;
    if (!(v < 0x1p63f)) {
      *fail = true;
      return b;
    }
    return b + incr(v);
  }
  // b 2^-32 in binary32 from the two 32-bit halves, each converted to
  // nearest, joined by one fused multiply-add
  static __device__ __forceinline__ float bscale(uint64_t b) {
    const float hi = __uint2float_rn((uint32_t)(b >> 32));
    const float lo = __uint2float_rn((uint32_t)b);
    return __fmaf_rn(lo, 0x1p-32f, hi);
  }
  static __device__ __forceinline__ float ig(uint64_t b, float G) { return bscale(b) / G; }
};
template <> struct SuffOps<double> {
  static __device__ __forceinline__ double from_prior(double b) { return b; }
  // b + r^2 / 2: the halving is exact, so it shares the addition's rounding
  static __device__ __forceinline__ double add_half_square(double b, double r, bool*) {
    const double r2 = r * r;
    return __fma_rn(r2, 0.5, b);
  }
  static __device__ __forceinline__ double ig(double b, double G) { return div_rn(b, G); }
};

// Constants of Marsaglia-Tsang for shape a, in binary64: d = a - 1/3,
// c = 1/sqrt(9 d) and the squeeze coefficient K = 0.0331 (2/3) / d, with
// 0.0331 (2/3) = 331/15000 rounded to nearest.
__device__ __forceinline__ void mt_constants(double a, double* d, double* c, double* K) {
  const double ONE_THIRD = 0x1.5555555555555p-2;
  const double SQZ = 0x1.698a4eea9073cp-6;
  const double dd = a - ONE_THIRD;
  const double nine_d = 9.0 * dd;
  const double s = sqrt_rn(nine_d);
  *d = dd;
  *c = div_rn(1.0, s);
  *K = div_rn(SQZ, dd);
}
// This cycle's constants for the propagation (observation and the
// Marsaglia-Tsang constants of the shapes a0 + (t+1)/2), in both precisions.
__device__ __forceinline__ void write_cycle_constants(Ctl* c, double y, double a_sigma,
                                                      double a_tau, uint32_t t1) {
  double ds, cs, ks, dt, ct, kt;
  mt_constants(a_sigma + 0.5 * (double)t1, &ds, &cs, &ks);
  mt_constants(a_tau + 0.5 * (double)t1, &dt, &ct, &kt);
  c->y = y;
  c->yf = (float)y;
  const double v[6] = {ds, cs, dt, ct, ks, kt};
  for (int i = 0; i < 6; ++i) {
    c->mtd[i] = v[i];
    c->mtf[i] = (float)v[i];
  }
}

template <class R, bool LEARN>
__global__ void __launch_bounds__(BLOCK) k_init(FilterArgs<R> a) {
  __shared__ double s_c[7];
  if (threadIdx.x == 0) {
    double ds, cs, ks, dt, ct, kt;
    mt_constants(a.a_sigma, &ds, &cs, &ks);
    mt_constants(a.a_tau, &dt, &ct, &kt);
    s_c[0] = ds; s_c[1] = cs; s_c[2] = dt; s_c[3] = ct;
    s_c[4] = sqrt(a.x0_var);
    s_c[5] = ks; s_c[6] = kt;
  }
  __syncthreads();
  const uint64_t j = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (j >= a.n) return;
  const StateV<R> st = a.st[0];
  const R x0m = (R)a.x0_mean;
  const R sdx = (R)s_c[4];
  const R Z = bm_normal(draw(a.seed, a.filter, 0, (uint32_t)j, P_INIT_X, 0), (R)0);
  const R p = sdx * Z;
  st.x[j] = x0m + p;
  const auto bs0 = SuffOps<R>::from_prior(a.b_sigma);
  const auto bt0 = SuffOps<R>::from_prior(a.b_tau);
  st.bs[j] = bs0;
  st.bt[j] = bt0;
  if (!LEARN) {
    st.s2[j] = (R)a.sigma2;
    st.t2[j] = (R)a.tau2;
    return;
  }
  bool fail = false;
  const R Gs = gamma_mt<R>((R)s_c[0], (R)s_c[1], (R)s_c[5], a.seed, a.filter, 0, (uint32_t)j,
                          P_INIT_SIGMA, &fail);
  const R Gt = gamma_mt<R>((R)s_c[2], (R)s_c[3], (R)s_c[6], a.seed, a.filter, 0, (uint32_t)j,
                          P_INIT_TAU, &fail);
  st.s2[j] = SuffOps<R>::ig(bs0, Gs);
  st.t2[j] = SuffOps<R>::ig(bt0, Gt);
  if (fail) atomicOr(&a.ctl->err, ERR_NUMERIC);
}

// ---------------------------------------------------------------------------
// Step 1a: predictive log-likelihood and its maximum.
// ---------------------------------------------------------------------------
template <class R>
__device__ __forceinline__ R log_pred(R x, R s2, R t2, R y) {
  const R s = s2 + t2;
  const R dx = y - x;
  const R q = dx * dx;
  const R lg = det_log(s);
  const R r = div_rn(q, s);
  const R sum = lg + r;
  return (R)-0.5 * sum;
}

// a / b of a pair: paired where both lanes' operands are safe for it
__device__ __forceinline__ float2 quot2(float2 a, float2 b) {
  return pair_safe(b, a) ? div_rn2(a, b) : make_float2(a.x / b.x, a.y / b.y);
}
// log_pred on two particles with paired operations; per lane the same IEEE
// operations in the same order, so the same bits.
__device__ __forceinline__ float2 log_pred2(float2 x, float2 s2, float2 t2, float yn) {
  const float2 s = add2(s2, t2);
  const float2 dx = sub2(splat2(yn), x);
  const float2 q = mul2(dx, dx);
  const float2 lg = det_log2(s);
  const float2 r = quot2(q, s);
  const float2 sum = add2(lg, r);
  return mul2(splat2(-0.5f), sum);
}

// Running maximum of log-likelihoods and whether one was NaN or +inf (such a
// value is left out of the maximum; the cycle fails).  Binary64 keeps the
// order-preserving signed integer of the value, so that neither the comparison
// nor the check goes to the binary64 pipe.
template <class R>
struct MaxL {
  float mx = -INFINITY;
  bool bad = false;
  __device__ __forceinline__ void take(float l) {
    bad |= !(l < INFINITY);
    mx = fmaxf(mx, l);
  }
  __device__ __forceinline__ float value() const { return mx; }
};
template <>
struct MaxL<double> {
  static constexpr long long NEG_INF = (long long)0x800FFFFFFFFFFFFFull;  // key of -inf
  long long mx = NEG_INF;
  bool bad = false;
  static __device__ __forceinline__ long long key(long long b) { return b ^ (long long)((unsigned long long)(b >> 63) >> 1); }
  __device__ __forceinline__ void take(double l) {
    const long long b = __double_as_longlong(l);
    // exponent field all ones: infinite or NaN; -inf is a weight of zero
    const bool odd = (__double2hiint(l) & 0x7FF00000) == 0x7FF00000;
    const long long v = key(b);
    const bool wrong = odd && v != NEG_INF;
    bad |= wrong;
    if (!wrong && v > mx) mx = v;
  }
  __device__ __forceinline__ double value() const { return __longlong_as_double(key(mx)); }
};

__device__ __forceinline__ unsigned long long enc_max(float x) { return enc_f(x); }
__device__ __forceinline__ unsigned long long enc_max(double x) { return enc_d(x); }

template <class R>
__device__ __forceinline__ R block_max(R v, R* s_red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane == 0) s_red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < WARPS ? s_red[lane] : (R)-INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}

// Binary64 kernels over single particles: warp w of CTA b takes 32 consecutive
// ones at (w gridDim + b) 32, then steps by the grid's threads.  A sub-partition
// takes 64 cycles per binary64 warp instruction, so a small filter finishes
// sooner with one warp on each of many SMs than with the eight warps of a CTA
// on one: N = 1024 weights 15.7 -> 11.2 us by events (all on one SM before).
__device__ __forceinline__ uint64_t spread_slot() {
  return ((uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
}

// Persistent over the particles: per pass a warp takes a chunk of 64 16-byte
// vectors of each array (2 x 32 x W_VEC particles), each load and store
// instruction 512 contiguous bytes, two of each in flight per thread and array;
// the rest of the last chunk element by element.  One block maximum and one
// atomic per CTA.
template <class R> struct WVec;
template <> struct WVec<float> {
  static constexpr int N = 4;
  typedef float4 V;
  static __device__ __forceinline__ void get(const V& v, float* o) { o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w; }
  static __device__ __forceinline__ V make(const float* o) { return make_float4(o[0], o[1], o[2], o[3]); }
};
template <> struct WVec<double> {
  static constexpr int N = 2;
  typedef double2 V;
  static __device__ __forceinline__ void get(const V& v, double* o) { o[0] = v.x; o[1] = v.y; }
  static __device__ __forceinline__ V make(const double* o) { return make_double2(o[0], o[1]); }
};
constexpr int W_CTAS_PER_SM = 4;  // 64 registers: the pass's 2 x 3 vectors stay in registers

// With ESS (adaptive resampling) the carried log-weights are added: L = lambda + l.
template <class R, bool ESS = false>
__global__ void __launch_bounds__(BLOCK, W_CTAS_PER_SM) k_weights(FilterArgs<R> a) {
  typedef WVec<R> VW;
  typedef typename VW::V V;
  constexpr int NV = VW::N;
  constexpr uint64_t CHUNK = 64 * NV;  // particles per warp pass
  __shared__ R s_red[WARPS];
  const uint32_t t = a.ctl->t;
  const StateV<R> st = (t & 1) ? a.st[1] : a.st[0];
  // every thread reads y itself (no barrier), so that its first loads of the
  // state overlap that read (y may sit in host memory)
  const double y = a.y_src ? *a.y_src : a.y_val;
  if (blockIdx.x == 0 && threadIdx.x == 0) write_cycle_constants(a.ctl, y, a.a_sigma, a.a_tau, t + 1);
  const R yr = (R)y;
  const uint64_t n = a.n;
  const int lane = threadIdx.x & 31;
  const uint64_t gw = (uint64_t)blockIdx.x * WARPS + (threadIdx.x >> 5);
  const uint64_t nw = (uint64_t)gridDim.x * WARPS;
  (void)gw; (void)nw;
  MaxL<R> top;
  auto weigh = [&](R x, R s2, R t2, R lam) {
    R l = log_pred<R>(x, s2, t2, yr);
    if constexpr (ESS) l = lam + l;
    top.take(l);
    return l;
  };
  auto chunk = [&](uint64_t cb) {  // the warp's chunk of CHUNK particles from cb
    if (cb + CHUNK <= n) {
      const uint64_t i0 = cb + (uint64_t)lane * NV, i1 = i0 + 32 * NV;
      const V x0 = *reinterpret_cast<const V*>(st.x + i0), x1 = *reinterpret_cast<const V*>(st.x + i1);
      const V s0 = *reinterpret_cast<const V*>(st.s2 + i0), s1 = *reinterpret_cast<const V*>(st.s2 + i1);
      const V u0 = *reinterpret_cast<const V*>(st.t2 + i0), u1 = *reinterpret_cast<const V*>(st.t2 + i1);
      R xv[2 * NV], sv[2 * NV], tv[2 * NV], lm[2 * NV], lv[2 * NV];
      VW::get(x0, xv); VW::get(x1, xv + NV);
      VW::get(s0, sv); VW::get(s1, sv + NV);
      VW::get(u0, tv); VW::get(u1, tv + NV);
      if constexpr (ESS) {
        VW::get(*reinterpret_cast<const V*>(a.lam + i0), lm);
        VW::get(*reinterpret_cast<const V*>(a.lam + i1), lm + NV);
      }
      if constexpr (sizeof(R) == 4) {
#pragma unroll
        for (int e = 0; e < 2 * NV; e += 2) {
          const float2 l = log_pred2(make_float2(xv[e], xv[e + 1]), make_float2(sv[e], sv[e + 1]),
                                     make_float2(tv[e], tv[e + 1]), yr);
          lv[e] = ESS ? lm[e] + l.x : l.x;
          lv[e + 1] = ESS ? lm[e + 1] + l.y : l.y;
          top.take(lv[e]);
          top.take(lv[e + 1]);
        }
      }
      *reinterpret_cast<V*>(a.ell + i0) = VW::make(lv);
      *reinterpret_cast<V*>(a.ell + i1) = VW::make(lv + NV);
    } else {
      for (uint64_t i = cb + lane; i < n; i += 32)
        a.ell[i] = weigh(st.x[i], st.s2[i], st.t2[i], ESS ? a.lam[i] : (R)0);
    }
  };
  const uint64_t nchunks = (n + CHUNK - 1) / CHUNK;
  if constexpr (sizeof(R) == 8) {
    // bound by the binary64 pipe, not by loads: one particle per lane, the
    // warps of a CTA far apart, so that few particles still reach every SM
    for (uint64_t i = spread_slot(); i < n; i += nw * 32)
      a.ell[i] = weigh(st.x[i], st.s2[i], st.t2[i], ESS ? a.lam[i] : (R)0);
  } else if (nchunks >= 4 * nw) {
    // Many chunks per warp: rounds of WARPS chunks (one per warp) go to
    // CTAs by ticket, each ticket taken a round ahead by thread 0, so that
    // CTAs on faster SMs take more rounds (the CTAs' finishing times under
    // the grid stride at N = 2^24 spread from 35 to 43 us).
    __shared__ uint32_t s_round[2];
    const uint64_t nrounds = (nchunks + WARPS - 1) / WARPS;
    uint64_t rd = blockIdx.x;
    uint32_t tk = 0;
    if (threadIdx.x == 0) tk = atomicAdd(&a.ctl->w_ticket, 1u);
    for (uint32_t q = 0; rd < nrounds; ++q) {
      const uint64_t ch = rd * WARPS + (threadIdx.x >> 5);
      if (ch < nchunks) chunk(ch * CHUNK);
      if (threadIdx.x == 0) {
        s_round[q & 1] = gridDim.x + tk;
        tk = atomicAdd(&a.ctl->w_ticket, 1u);
      }
      __syncthreads();
      rd = s_round[q & 1];
    }
  } else {
    for (uint64_t cb = gw * CHUNK; cb < n; cb += nw * CHUNK) chunk(cb);
  }
  if (top.bad) atomicOr(&a.ctl->err, ERR_NUMERIC);
  const R mx = block_max<R>(top.value(), s_red);
  if (threadIdx.x == 0 && mx > (R)-INFINITY) atomicMax(&a.ctl->maxenc, enc_max(mx));
}
// CTAs of the weights kernel for n particles: the resident maximum `cap`, or
// fewer when the particles make fewer chunks than the resident warps.
template <class R>
inline unsigned weights_grid(uint64_t n, uint64_t cap) {
  // binary32: one chunk per warp; binary64: 32 particles, so that a CTA has one warp's work
  const uint64_t per_cta = sizeof(R) == 8 ? 32ull : 64ull * WVec<R>::N * WARPS;
  const uint64_t ctas = (n + per_cta - 1) / per_cta;
  return (unsigned)(ctas < cap ? (ctas > 0 ? ctas : 1) : cap);
}

// ---------------------------------------------------------------------------
// Algorithm "Particle Filtering" (the bootstrap filter, known variances),
// Steps 1-2: propagate every particle blind, x_t = x~_{t-1} + sqrt(tau^2) Z
// (Box-Muller's first output of the draw (seed, filter, t, i, BOOT_STATE)),
// in place, then weigh it by p(y_t | x_t) = N(y_t; x_t, sigma^2): the
// predictive-weight kernel's l with tau^2 = 0, and its maximum.  Step 3 is
// the resampling of the particle-learning cycle; k_boot_gather then copies
// the ancestors.
// ---------------------------------------------------------------------------
template <class R>
__global__ void __launch_bounds__(BLOCK) k_boot_pw(FilterArgs<R> a) {
  __shared__ R s_red[WARPS];
  Ctl* c = a.ctl;
  const uint32_t t = c->t;
  const StateV<R> st = (t & 1) ? a.st[1] : a.st[0];
  const double y = a.y_src ? *a.y_src : a.y_val;
  const R yr = (R)y;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    c->y = y;
    c->yf = (float)y;
  }
  MaxL<R> top;
  const uint64_t stride = (uint64_t)gridDim.x * BLOCK;
  for (uint64_t i = sizeof(R) == 8 ? spread_slot() : (uint64_t)blockIdx.x * BLOCK + threadIdx.x; i < a.n; i += stride) {
    const R Z = bm_normal(draw(a.seed, a.filter, t, (uint32_t)i, P_BOOT_STATE, 0), (R)0);
    const R sv = sqrt_rn(st.t2[i]);
    const R xz = sv * Z;
    const R xp = st.x[i] + xz;
    st.x[i] = xp;
    const R l = log_pred<R>(xp, st.s2[i], (R)0, yr);
    top.take(l);
    a.ell[i] = l;
  }
  if (top.bad) atomicOr(&c->err, ERR_NUMERIC);
  const R mx = block_max<R>(top.value(), s_red);
  if (threadIdx.x == 0 && mx > (R)-INFINITY) atomicMax(&c->maxenc, enc_max(mx));
}

// ---------------------------------------------------------------------------
// Step 1b: the exact fixed-point CDF by a single-pass decoupled look-back scan
// (Merrill & Garland 2016).  Tiles are claimed through an atomic ticket so a
// tile's predecessors are always resident or finished; the look-back wait is
// bounded and reports ERR_TIMEOUT instead of hanging.
//
// Warp w of a tile owns elements [512 w, 512 w + 512) as 4 chunks of 128;
// lane l owns elements 4l..4l+3 of each chunk, so every load and store
// instruction of the warp covers one contiguous span.
// ---------------------------------------------------------------------------

// Sum of exp(l_i - m) for the log marginal likelihood: exact 2^-96 fixed
// point in FP32 mode (binary32 terms >= 2^-73 are integers there).
struct ESum32 {
  U128 s;
  __device__ __forceinline__ void zero() { s.hi = 0; s.lo = 0; }
  __device__ __forceinline__ void add(float e) {
    // e = 0 or e >= 2^-73: e * 2^96 = mant * 2^(exponent bits - 54), an
    // integer below 2^101 (e < 16 for a thread's partial); added without branches
    const uint32_t b = __float_as_uint(e);
    const uint32_t E = b >> 23;
    const uint64_t mant = E ? (uint64_t)((b & 0x7fffffu) | 0x800000u) : 0ull;
    const int sh = E > 54u ? (int)E - 54 : 0;
    const uint64_t lo = sh < 64 ? mant << sh : 0ull;
    const uint64_t hi = sh == 0 ? 0ull : (sh < 64 ? mant >> (64 - sh) : mant << (sh - 64));
    s = add128(s, U128{hi, lo});
  }
  __device__ __forceinline__ void add(const ESum32& o) { s = add128(s, o.s); }
  __device__ __forceinline__ ESum32 shfl_xor(int m) const {
    ESum32 r;
    r.s.hi = __shfl_xor_sync(0xffffffffu, s.hi, m);
    r.s.lo = __shfl_xor_sync(0xffffffffu, s.lo, m);
    return r;
  }
};
struct ESum64 {
  double s;
  __device__ __forceinline__ void zero() { s = 0.0; }
  __device__ __forceinline__ void add(double e) { s = s + e; }
  __device__ __forceinline__ void add(const ESum64& o) { s = s + o.s; }
  __device__ __forceinline__ ESum64 shfl_xor(int m) const {
    ESum64 r;
    r.s = __shfl_xor_sync(0xffffffffu, s, m);
    return r;
  }
};
template <class R> struct ESumT;
template <> struct ESumT<float> { typedef ESum32 T; };
template <> struct ESumT<double> { typedef ESum64 T; };

// Binary64: e_i = exp(l_i - m) for every particle, into the space of the CDF
// (the scan reads e and writes Q in its place; l stays for a propagation that
// carries L - m).  The exponential is 21 of the CDF's 23 operations on the
// binary64 pipe; here it runs one particle per lane on every SM, where a scan
// tile would do 4096 of them on one: systematic cycle at N = 16384 70.7 -> 41.8
// us, at N = 2^20 (256 tiles on 152 SMs) 329 -> 313 us.
static __global__ void __launch_bounds__(BLOCK) k_exp(FilterArgs<double> a) {
  const double m = dec_d(a.ctl->maxenc);
  double* const E = reinterpret_cast<double*>(a.Q);
  for (uint64_t i = spread_slot(); i < a.n; i += (uint64_t)gridDim.x * BLOCK) E[i] = exp_weight(a.ell[i] - m);
}

// Tile look-back by warp 0.  Returns the exclusive prefix of the tile (in
// lane 0).  `total` is the tile aggregate.  Each round reads a window of 128
// predecessors (four status words per lane, loads issued together), so a
// tile far from the last published prefix needs few round trips.
constexpr int LB_PER_LANE = 4;

__device__ __forceinline__ uint64_t spin_status(const uint64_t* p, bool* timed_out,
                                                uint32_t limit) {
  uint64_t v = ld_status(p);
  uint32_t spins = 0;
  while ((v >> 62) == 0) {
    if (++spins > limit) {
      *timed_out = true;
      return FLAG_P;
    }
    __nanosleep(32);
    v = ld_status(p);
  }
  return v;
}

// limit: polls of one status word before the wait gives up (ERR_TIMEOUT);
// withhold: a tile that publishes nothing (a failure-detection test makes its
// successors' waits run out this way; NO_TILE otherwise).
constexpr uint32_t NO_TILE = 0xffffffffu;
__device__ __forceinline__ uint64_t lookback(uint64_t* stat, uint32_t tile, uint64_t total,
                                             uint32_t* err, uint32_t limit = SPIN_LIMIT,
                                             uint32_t withhold = NO_TILE) {
  const int lane = threadIdx.x & 31;
  if (tile == withhold) return 0;
  if (tile == 0) {
    if (lane == 0) st_status(&stat[0], FLAG_P | total);
    return 0;
  }
  if (lane == 0) st_status(&stat[tile], FLAG_A | total);
  uint64_t excl = 0;
  int64_t look = (int64_t)tile - 1;
  bool timed_out = false;
  while (true) {
    // lane l covers distances LB_PER_LANE*l .. LB_PER_LANE*l + 3 below `look`
    uint64_t v[LB_PER_LANE];
#pragma unroll
    for (int k = 0; k < LB_PER_LANE; ++k) {
      const int64_t idx = look - (LB_PER_LANE * lane + k);
      v[k] = idx >= 0 ? ld_status(&stat[idx]) : FLAG_P;  // before tile 0: a zero prefix
    }
#pragma unroll
    for (int k = 0; k < LB_PER_LANE; ++k) {
      const int64_t idx = look - (LB_PER_LANE * lane + k);
      if ((v[k] >> 62) == 0) v[k] = spin_status(&stat[idx], &timed_out, limit);
    }
    int first_p = LB_PER_LANE;
#pragma unroll
    for (int k = LB_PER_LANE - 1; k >= 0; --k)
      if ((v[k] >> 62) == 2) first_p = k;
    const uint32_t pmask = __ballot_sync(0xffffffffu, first_p < LB_PER_LANE);
    const int stop_lane = pmask ? __ffs(pmask) - 1 : 32;
    uint64_t contrib = 0;
#pragma unroll
    for (int k = 0; k < LB_PER_LANE; ++k) {
      const bool take = lane < stop_lane || (lane == stop_lane && k <= first_p);
      if (take) contrib += v[k] & VAL_MASK;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) contrib += __shfl_xor_sync(0xffffffffu, contrib, o);
    excl += contrib;
    if (pmask) break;
    look -= 32 * LB_PER_LANE;
  }
  if (__any_sync(0xffffffffu, timed_out) && lane == 0) atomicOr(err, ERR_TIMEOUT);
  if (lane == 0) st_status(&stat[tile], FLAG_P | ((excl + total) & VAL_MASK));
  return excl;
}

// floor(w 2^s) of a caller's weight (negative and non-finite ones, which
// k_wmax has flagged: 0); below 2^k by the choice of s
__device__ __forceinline__ uint64_t quant_weight(float w, int s) {
  const uint32_t b = __float_as_uint(w);
  if (b >= 0x7F800000u) return 0;
  const uint32_t E = b >> 23;
  const uint32_t m = (b & 0x7fffffu) | (E ? 0x800000u : 0u);
  const int sh = (int)(E ? E : 1u) - 150 + s;
  return sh >= 0 ? (uint64_t)m << sh : (uint64_t)(m >> (-sh < 31 ? -sh : 31));
}

struct ScanArgs {
  const float* src;         // weights
  uint64_t* Q;
  uint64_t* stat;           // tile status, zero before the launch
  Ctl* ctl;
  uint64_t n;
  int k;
  int vec_ok;               // src is 16-byte aligned
  uint32_t spin_limit;      // look-back polls before giving up (SPIN_LIMIT)
  uint32_t withhold;        // a tile that publishes nothing (NO_TILE; failure tests)
};

// Thread-blocked scan: thread t of a tile owns the 16 consecutive elements
// [16 t, 16 t + 16), so the running sum is two integer adds per element and
// the warp / block scans run once per 16 elements.
constexpr int SCAN_PER = TILE / BLOCK;  // 16

static __global__ void __launch_bounds__(BLOCK, 4) k_scan(ScanArgs a) {
  __shared__ uint64_t s_stage[BLOCK * (SCAN_PER + 1)];
  __shared__ uint32_t s_tile;
  __shared__ uint64_t s_warp_tot[WARPS];
  __shared__ uint64_t s_excl;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_tile = atomicAdd(&a.ctl->ticket_w, 1u);
  __syncthreads();
  const uint32_t tile = s_tile;
  const uint64_t base = (uint64_t)tile * TILE + (uint64_t)threadIdx.x * SCAN_PER;
  // quantisation is relative to the power of two of the largest weight
  int e2;
  (void)frexpf(__uint_as_float((uint32_t)a.ctl->maxenc), &e2);
  const int escale = a.k - e2;

  const bool full = base + SCAN_PER <= a.n;
  uint64_t W[SCAN_PER];
  uint64_t run = 0;
#pragma unroll
  for (int q = 0; q < SCAN_PER / 4; ++q) {
    // four values at a time, consumed as soon as they arrive
    float v[4];
    if (full && a.vec_ok) {
      const float4 f = *reinterpret_cast<const float4*>(a.src + base + 4 * q);
      v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = (base + 4 * q + e < a.n) ? a.src[base + 4 * q + e] : 0.0f;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      run += quant_weight(v[e], escale);
      W[4 * q + e] = run;  // inclusive running sum
    }
  }
  // warp exclusive offsets of the thread totals, then the block
  const uint64_t tt = W[SCAN_PER - 1];
  const uint64_t tincl = warp_incl_scan(tt, lane);
  if (lane == 31) s_warp_tot[warp] = tincl;
  __syncthreads();
  if (warp == 0) {
    uint64_t wt = lane < WARPS ? s_warp_tot[lane] : 0;
    const uint64_t wincl = warp_incl_scan(wt, lane);
    if (lane < WARPS) s_warp_tot[lane] = wincl - wt;  // exclusive warp offsets
  }
  __syncthreads();
  // stage the tile-local inclusive prefix (padded rows of 17 words), so that
  // no per-element state is live across the look-back
  {
    const uint64_t toff = s_warp_tot[warp] + (tincl - tt);
#pragma unroll
    for (int e = 0; e < SCAN_PER; ++e) s_stage[threadIdx.x * (SCAN_PER + 1) + e] = W[e] + toff;
  }
  __syncthreads();
  if (warp == 0) {
    // tile total = last thread's staged inclusive value
    const uint64_t total = s_stage[(BLOCK - 1) * (SCAN_PER + 1) + SCAN_PER - 1];
    const uint64_t excl = lookback(a.stat, tile, total, &a.ctl->err, a.spin_limit, a.withhold);
    if (lane == 0) s_excl = excl;
  }
  __syncthreads();
  const uint64_t off = s_excl;
  const uint64_t tbase = (uint64_t)tile * TILE;
  if (tbase + TILE <= a.n) {
#pragma unroll
    for (int r = 0; r < TILE / (2 * BLOCK); ++r) {
      const int q = 2 * threadIdx.x + 2 * BLOCK * r;  // even: q and q+1 share a row
      const int si = (q >> 4) * (SCAN_PER + 1) + (q & 15);
      *reinterpret_cast<ulonglong2*>(a.Q + tbase + q) =
          make_ulonglong2(s_stage[si] + off, s_stage[si + 1] + off);
    }
  } else {
    for (int q = threadIdx.x; q < TILE; q += BLOCK)
      if (tbase + q < a.n) a.Q[tbase + q] = s_stage[(q >> 4) * (SCAN_PER + 1) + (q & 15)] + off;
  }
}

// Multinomial positions: spacing E_l = floor(-log(u_l) 2^31), u_l from draw
// (seed, filter, t, l >> 2, SPACING) word l & 3 (multi.cuh).
__device__ __forceinline__ uint64_t spacing_E(uint64_t seed, uint32_t filter, uint32_t t,
                                              uint64_t l, const U4& w) {
  const uint32_t word = (l & 3) == 0 ? w.a : (l & 3) == 1 ? w.b : (l & 3) == 2 ? w.c : w.d;
  const float u = unif_f32(word);
  const float L = det_log(u);
  const float x = -L * 0x1p31f;
  return f2u64_rz(x);
}

// ---------------------------------------------------------------------------
// Exact slot positions.  Systematic: slot j's key is j T + r (A = n), so slots
// are equally spaced and particle i owns the slots [R_{i-1}, R_i) with
// R_i = #{j : j T + r < n Q_i}.
// ---------------------------------------------------------------------------

__device__ __forceinline__ U128 sub128(U128 x, uint64_t y) {
  return U128{x.hi - (x.lo < y ? 1ull : 0ull), x.lo - y};
}
__device__ __forceinline__ U128 sub128(U128 x, U128 y) {
  return U128{x.hi - y.hi - (x.lo < y.lo ? 1ull : 0ull), x.lo - y.lo};
}

struct SysDiv {      // reciprocal of T for quotients below 2^32
  uint64_t T, m;     // m = floor((2^64 - 1) / (T >> s))
  int s;             // T >> s lies in [2^31, 2^32) (s = 0 if T < 2^32)
};
__device__ __forceinline__ SysDiv make_sysdiv(uint64_t T) {
  SysDiv d;
  d.T = T;
  const int bits = 64 - __clzll((long long)T);
  d.s = bits > 32 ? bits - 32 : 0;
  d.m = 0xffffffffffffffffull / (T >> d.s);
  return d;
}
// floor(Z / T) for Z < T * 2^32: reciprocal estimate, exact correction.
__device__ __forceinline__ uint64_t sys_floor_div(U128 Z, const SysDiv& d) {
  const uint64_t zs = d.s ? ((Z.lo >> d.s) | (Z.hi << (64 - d.s))) : Z.lo;
  uint64_t q = __umul64hi(zs, d.m);
  U128 P = mul64(q, d.T);
  for (int it = 0; it < 8 && lt128(Z, P); ++it) {
    --q;
    P = sub128(P, d.T);
  }
  for (int it = 0; it < 8; ++it) {
    const U128 P1 = add128(P, d.T);
    if (lt128(Z, P1)) break;
    ++q;
    P = P1;
  }
  return q;
}
// R(Q) = #{j in [0, n) : j T + r < n Q} = clamp(ceil((n Q - r) / T), 0, n).
__device__ __forceinline__ uint64_t sys_first_slot(uint64_t Qi, uint64_t n, uint64_t r,
                                                   const SysDiv& d) {
  const U128 X = mul64x32(Qi, (uint32_t)n);
  if (le128(X, U128{0, r})) return 0;
  const U128 Z = sub128(sub128(X, r), 1ull);  // ceil(Y/T) = floor((Y-1)/T) + 1
  const uint64_t q = sys_floor_div(Z, d) + 1;
  return q < n ? q : n;
}

// Stratified resampling (Section 3.1, one uniform in each of the n equal
// strata): slot j's position is P_j = j T + r_j with its own r_j in [0, T),
// r_j = floor(R_j T / 2^64) from word pair 2 (j mod 2), 2 (j mod 2) + 1 of the
// draw (seed, filter, t, floor(j/2), STRATIFIED); slot j goes to the particle
// i with n Q_{i-1} <= P_j < n Q_i.
__device__ __forceinline__ uint64_t strat_offset(uint64_t T, uint64_t seed, uint32_t filter,
                                                 uint32_t t, uint64_t j) {
  const U4 w = draw(seed, filter, t, (uint32_t)(j >> 1), P_STRATIFIED, 0);
  const uint64_t R = (j & 1) ? (((uint64_t)w.d << 32) | w.c) : (((uint64_t)w.b << 32) | w.a);
  return __umul64hi(R, T);
}
// #{j : P_j < n q}: with c = floor(n q / T), P_c is the only position in
// [c T, c T + T), so the count is c or c + 1.
__device__ __forceinline__ uint64_t strat_first(uint64_t q, uint64_t n, uint64_t T, const SysDiv& dv,
                                                uint64_t seed, uint32_t filter, uint32_t t) {
  const U128 X = mul64x32(q, (uint32_t)n);
  if (X.hi == 0 && X.lo == 0) return 0;
  const uint64_t c = sys_floor_div(X, dv);  // X <= n T < 2^32 T
  if (c >= n) return n;
  const U128 P = add128(mul64x32(T, (uint32_t)c), strat_offset(T, seed, filter, t, c));
  return lt128(P, X) ? c + 1 : c;
}
// ---------------------------------------------------------------------------
// The paper's Section 3.2 algorithms.
// Parallelized Cut-Point Search: L_i = ceil(n Q_i / T), and I_k = i for
// L_{i-1} <= k < L_i.  One thread per particle; L_{i-1} comes from the lane
// below, and a warp stores the ranges longer than 32 together.  (Inside a
// resampling k_slots builds the same table: L_i is its slot map with r = 0.)
// ---------------------------------------------------------------------------
static __global__ void __launch_bounds__(BLOCK) k_cutpoint_search(const uint64_t* Q, uint64_t n,
                                                           uint32_t* I) {
  const uint64_t i = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
  const uint64_t T = Q[n - 1];
  const int lane = threadIdx.x & 31;
  if (T == 0) {
    if (i < n) I[i] = (uint32_t)i;
    return;
  }
  const SysDiv dv = make_sysdiv(T);
  auto L = [&](uint64_t q) { return sys_first_slot(q, n, 0, dv); };  // at most n
  const uint64_t l1 = i < n ? L(Q[i]) : n;
  uint64_t l0 = __shfl_up_sync(0xffffffffu, l1, 1);
  if (lane == 0) l0 = i == 0 ? 0 : (i < n ? L(Q[i - 1]) : n);
  const uint64_t cnt = i < n && l1 > l0 ? l1 - l0 : 0;
  if (cnt <= 32)
    for (uint64_t k = l0; k < l0 + cnt; ++k) I[k] = (uint32_t)i;
  uint32_t heavy = __ballot_sync(0xffffffffu, cnt > 32);
  while (heavy) {
    const int l = __ffs(heavy) - 1;
    heavy &= heavy - 1;
    const uint64_t s0 = __shfl_sync(0xffffffffu, l0, l), s1 = __shfl_sync(0xffffffffu, l1, l);
    const uint32_t v = (uint32_t)__shfl_sync(0xffffffffu, i, l);
    for (uint64_t k = s0 + lane; k < s1; k += 32) I[k] = v;
  }
}

// Parallelized Cut-Point Method for the systematic positions j T + r (bucket
// j): start at I_j, climb while n Q_k <= j T + r.  (Multinomial: k_multi.)
struct PosArgs {
  const uint64_t* Q;
  uint32_t* anc;
  const uint32_t* I;      // cut-point table
  Ctl* ctl;
  const uint32_t* t_dev;
  uint32_t t_arg;
  uint64_t n;
  uint64_t seed;
  uint32_t filter;
  // adaptive resampling: when set and *gate == 0 this cycle does not
  // resample, and the kernel returns at once (NULL: always run)
  const uint32_t* gate;
};
static __global__ void __launch_bounds__(BLOCK) k_cutpoint_method_sys(PosArgs a) {
  if (a.gate && *a.gate == 0u) return;
  const uint64_t j = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (j >= a.n) return;
  const uint64_t T = a.ctl->keyT;
  if (T == 0) {  // empty CDF (flagged): keep every index in range
    a.anc[j] = (uint32_t)j;
    return;
  }
  const uint32_t t = a.t_dev ? *a.t_dev : a.t_arg;
  const U4 w = draw(a.seed, a.filter, t, 0, P_SYS_OFFSET, 0);
  const uint64_t r = __umul64hi(((uint64_t)w.b << 32) | w.a, T);
  uint64_t k = a.I[j];
  const U128 kb = add128(mul64x32(T, (uint32_t)j), r);
  while (k < a.n && le128(mul64x32(a.Q[k], (uint32_t)a.n), kb)) ++k;
  a.anc[j] = (uint32_t)(k < a.n ? k : a.n - 1);
}

// Explicit integer positions U_j in [0, T) (A = 1).
static __global__ void __launch_bounds__(BLOCK) k_cutpoint_method_explicit(
    const uint64_t* Q, uint64_t n, const uint32_t* I, const uint64_t* U, uint64_t m,
    uint32_t* anc) {
  const uint64_t j = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (j >= m) return;
  const uint64_t T = Q[n - 1];
  const uint64_t u = U[j];
  const uint64_t b = T == 0 ? 0 : u < T ? sys_floor_div(mul64x32(u, (uint32_t)n), make_sysdiv(T)) : n;
  uint64_t k = I[b < n ? b : n - 1];
  while (k < n && Q[k] <= u) ++k;
  anc[j] = (uint32_t)(k < n ? k : n - 1);
}

// Entry of slot x (relative to the window's base, a multiple of four) in
// k_slots' window of 16-bit entries: x with bits 1-3 XORed by bits 6-8, so that
// threads writing slots about eight apart, and warps reading consecutive slots,
// hit distinct banks.  The four slots 4g .. 4g + 3 keep one aligned group of four
// entries (in the order 0 1 2 3, or 2 3 0 1 when bit 1 is flipped), so the window
// is read out four slots per 8-byte load.
__device__ __forceinline__ uint32_t win_entry(uint32_t x) { return x ^ (((x >> 6) & 7u) << 1); }
// Correctly rounded conversion of a 128-bit integer to binary64: the top 64
// significant bits with a sticky bit for the rest, rounded once, scaled by an
// exact power of two.
__device__ __forceinline__ double u128_to_f64_rn(U128 v) {
  if (v.hi == 0) return __ull2double_rn(v.lo);
  const int lz = __clzll(v.hi);
  const int sh = 64 - lz;  // 1..64
  uint64_t top, rest;
  if (lz == 0) {
    top = v.hi;
    rest = v.lo;
  } else {
    top = (v.hi << lz) | (v.lo >> sh);
    rest = v.lo << lz;
  }
  const double d = __ull2double_rn(top | (rest != 0 ? 1ull : 0ull));
  return d * __longlong_as_double((long long)(1023 + sh) << 52);
}

}  // namespace pfk
#include "slots.cuh"
#include "multi.cuh"
namespace pfk {

// ---------------------------------------------------------------------------
// Steps 2-4: propagate x, update the sufficient statistics, draw theta.
// The last block to finish folds the log-ML partials, resets the per-cycle
// counters and advances t.
// ---------------------------------------------------------------------------
template <class R> struct ResidObs;
template <> struct ResidObs<float> {
  static __device__ __forceinline__ float f(double, float yr, float xj) { return yr - xj; }
};
template <> struct ResidObs<double> {
  static __device__ __forceinline__ double f(double y, double, double xj) { return y - xj; }
};

__device__ __forceinline__ double esum_value(const ESum32& e) {
  return __ull2double_rn(e.s.hi) * 0x1p-32 + __ull2double_rn(e.s.lo) * 0x1p-96;
}
__device__ __forceinline__ double esum_value(const ESum64& e) { return e.s; }

// Run by the last warp of k_propagate: fold the per-tile log-ML partials
// (lane-strided, then butterfly: a fixed order), accumulate the increment
// m + log(sum_i e_i) - log n - log(2 pi)/2, reset the per-cycle counters and
// advance t.
//
// With FUSE the propagation has also computed the next cycle's weights: the
// maximum it gathered becomes the next cycle's, and the constants that the
// weights kernel would write for the next cycle (observation y_{t+2},
// Marsaglia-Tsang constants of the shapes a0 + (t+2)/2) are written here, once
// every warp has read this cycle's.
//
// With ESS (adaptive resampling) the increment is normalised by the carried
// weights, log sum_i exp(lambda_i), instead of log n, and that sum for the
// next cycle is n after a resampling, else this cycle's sum of exp(L_i - m).
template <class R, bool FUSE = false, bool ESS = false>
__device__ void fold_cycle_warp(const FilterArgs<R>& a, uint32_t t) {
  typedef typename ESumT<R>::T ES;
  const int lane = threadIdx.x & 31;
  ES acc;
  acc.zero();
  const ES* const part = reinterpret_cast<const ES*>(a.part);
  if constexpr (sizeof(R) == 4) {
    // exact fixed-point partials: any grouping gives the same sum, so each
    // lane issues eight loads at once
    for (uint32_t b = lane; b < a.nparts; b += 256) {
      ES v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        v[q].zero();
        if (b + 32u * q < a.nparts) v[q] = part[b + 32u * q];
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) acc.add(v[q]);
    }
  } else {
    for (uint32_t b = lane; b < a.nparts; b += 32) acc.add(part[b]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc.add(acc.shfl_xor(o));
  if (lane == 0) {
    Ctl* c = a.ctl;
    const double m = sizeof(R) == 4 ? (double)dec_f((uint32_t)c->maxenc) : dec_d(c->maxenc);
    const double LOG_2PI = 0x1.d67f1c864beb5p+0;
    if constexpr (ESS) {
      const double S = esum_value(acc);
      const double inc = m + log(S) - log(c->slam) - 0.5 * LOG_2PI;
      c->logml = c->logml + inc;
      c->slam = c->resamp ? (double)a.n : S;
    } else {
      const double inc = m + log(esum_value(acc)) - log((double)a.n) - 0.5 * LOG_2PI;
      c->logml = c->logml + inc;
    }
    const unsigned long long ninf =
        sizeof(R) == 4 ? (unsigned long long)enc_f(-INFINITY) : enc_d(-INFINITY);
    if constexpr (FUSE) {
      // every warp's maximum was published before its completion count
      __threadfence();
      c->maxenc = atomicExch(&c->maxenc_nx, ninf);
      const double y = a.y_nx_src ? *a.y_nx_src : a.y_nx_val;
      write_cycle_constants(c, y, a.a_sigma, a.a_tau, t + 2);
    } else {
      c->maxenc = ninf;
    }
    c->ticket_w = 0;
    c->done_prop = 0;
    c->prop_ticket = 0;
    c->w_ticket = 0;
    __threadfence();
    c->t = t + 1;
  }
}

// A gamma draw that missed the Marsaglia-Tsang squeeze on its first attempt,
// finished after the warp's fast path (same arithmetic, later in time).
template <class R>
struct GammaItem {
  typename SuffT<R>::B b;  // updated sufficient statistic (the IG scale)
  R Z, U;                  // attempt-0 normal and uniform
  uint32_t j;              // slot
  uint32_t which;          // 0: sigma^2, 1: tau^2
};

// Per-warp queue of such draws.  A warp pushes at most 64 per pass and
// finishes them 32 at a time (one per lane) once 32 are queued, so no block
// barrier is needed and the lanes of a finishing round are all busy.
constexpr uint32_t WQ_CAP = 96;

template <class Item>
__device__ __forceinline__ void wq_push(Item* q, uint32_t& qn, bool dfr, const Item& itm,
                                        int lane) {
  const uint32_t m = __ballot_sync(0xffffffffu, dfr);
  if (dfr) q[qn + __popc(m & ((1u << lane) - 1u))] = itm;
  qn += __popc(m);
}

// Finish queued draws, 32 per round, while at least `lo` (>= 1) are queued;
// after each round (its writes ordered by the warp barrier) `post` runs on the
// lanes whose item has bit 1 of `which` set.
template <class R, class Fin, class Post>
__device__ __forceinline__ void wq_drain_post(GammaItem<R>* q, uint32_t& qn, uint32_t lo,
                                              int lane, Fin fin, Post post) {
  __syncwarp();
  while (qn >= lo) {
    const uint32_t take = qn < 32u ? qn : 32u;
    const uint32_t base = qn - take;
    const bool mine = (uint32_t)lane < take;
    GammaItem<R> itm;
    if (mine) {
      itm = q[base + lane];
      fin(itm);
    }
    __syncwarp();
    if (mine && (itm.which & 2u)) post(itm);
    qn = base;
    __syncwarp();
  }
}

// Finish queued draws, 32 per round, while at least `lo` (>= 1) are queued.
template <class Item, class Fin>
__device__ __forceinline__ void wq_drain(Item* q, uint32_t& qn, uint32_t lo, int lane, Fin fin) {
  __syncwarp();
  while (qn >= lo) {
    const uint32_t take = qn < 32u ? qn : 32u;
    const uint32_t base = qn - take;
    if ((uint32_t)lane < take) fin(q[base + lane]);
    qn = base;
    __syncwarp();
  }
}

// The propagation's shared reciprocal 1 / s of s = sigma^2 + tau^2 and
// sqrt(V), V = (sigma^2 tau^2) / s, of a slot pair.
__device__ __forceinline__ void state_scale2(float2 sa, float2 ta, float2 s, float2* ri, float2* sv) {
  const float2 p = mul2(sa, ta);
  if (pair_safe(sa, ta)) {  // then s and V lie within [2^-81, 2^41] too
    *ri = rcp_rn2(s);
    *sv = sqrt_rn2(mul2(p, *ri));
  } else {
    *ri = make_float2(__frcp_rn(s.x), __frcp_rn(s.y));
    const float2 V = mul2(p, *ri);
    *sv = make_float2(sqrtf(V.x), sqrtf(V.y));
  }
}
// The inverse-gamma quotients b / G of a slot pair.  b is 0 or in [2^-32, 2^32);
// an accepted draw has G = d v^3 with v above 0.04 (the squeeze bounds |Z|) and
// below 4, so for shapes below 2^60 both operands and the quotient are far from
// the ends of the range (the quotient of a draw that missed the squeeze is not
// used).  wide: a larger shape (the same in every thread).
__device__ __forceinline__ bool ig_wide(float ds, float dt) { return !(ds < 0x1p60f && dt < 0x1p60f); }
__device__ __forceinline__ float2 ig2(float2 b, float2 G, bool wide) {
  if (wide) return make_float2(b.x / G.x, b.y / G.y);
  return div_rn2(b, G);
}

// The next cycle's weight of one slot: l = log p(y_{t+2} | x, sigma^2, tau^2),
// the weights kernel's arithmetic; its maximum and finiteness are tracked.
template <class R>
__device__ __forceinline__ void weigh_next(R* ell, uint64_t j, R x, R s2, R t2, R yn, R& mx,
                                           bool& bad) {
  const R l = log_pred<R>(x, s2, t2, yn);
  ell[j] = l;
  bad |= !(l < (R)INFINITY);
  mx = fmax(mx, l);
}

// Store a next-cycle weight computed elsewhere and track it.
template <class R>
__device__ __forceinline__ void keep_next(R* ell, uint64_t j, R l, R& mx, bool& bad) {
  ell[j] = l;
  bad |= !(l < (R)INFINITY);
  mx = fmax(mx, l);
}

// Publish a warp's maximum of the next cycle's weights (lane 0 only), before
// the warp's completion count.
template <class R>
__device__ __forceinline__ void publish_next_max(Ctl* c, R mx, int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) {
    if (mx > (R)-INFINITY) atomicMax(&c->maxenc_nx, enc_max(mx));
    __threadfence();
  }
}

// One ancestor's record, gathered ahead of its use.
template <class R>
struct Gathered {
  R x, s2, t2;
  typename SuffT<R>::B bs, bt;
};
template <class R>
__device__ __forceinline__ Gathered<R> gather_rec(const StateV<R>& src, uint32_t an) {
  Gathered<R> g;
  g.x = src.x[an];
  g.s2 = src.s2[an];
  g.t2 = src.t2[an];
  g.bs = src.bs[an];
  g.bt = src.bt[an];
  return g;
}

// Persistent grid: a thread handles the slots spread_slot() + k * stride.  The
// ancestor index is loaded two slots ahead and the ancestor's record one slot
// ahead, so the dependent index -> gather latency overlaps the arithmetic of the
// current slot.
//
// With FUSE the kernel also computes the next cycle's predictive weights
// l_j = log p(y_{t+2} | x'_j, sigma^2'_j, tau^2'_j) and their maximum, which
// the next cycle then uses instead of running the weights kernel.  A slot
// whose gamma draw missed the squeeze is weighed by the drain round that
// finishes its last queued draw (bit 1 of `which` on that item), reading its
// new state back after the round's warp barrier.  Every value is the one the
// weights kernel would give.
template <class R, bool LEARN, bool FUSE = false, bool ESS = false>
__global__ void __launch_bounds__(BLOCK, 3) k_propagate(FilterArgs<R> a) {
  typedef GammaItem<R> Item;
  __shared__ Item s_q[WARPS][WQ_CAP];
  const Ctl* c = a.ctl;
  const uint32_t t = c->t;
  const StateV<R> src = (t & 1) ? a.st[1] : a.st[0];
  const StateV<R> dst = (t & 1) ? a.st[0] : a.st[1];
  const double y = c->y;
  R yr, ds, cs, dt, ct, ks, kt;
  if constexpr (sizeof(R) == 4) {
    yr = c->yf; ds = c->mtf[0]; cs = c->mtf[1]; dt = c->mtf[2]; ct = c->mtf[3];
    ks = c->mtf[4]; kt = c->mtf[5];
  } else {
    yr = y; ds = c->mtd[0]; cs = c->mtd[1]; dt = c->mtd[2]; ct = c->mtd[3];
    ks = c->mtd[4]; kt = c->mtd[5];
  }
  const int lane = threadIdx.x & 31;
  Item* const wq = s_q[threadIdx.x >> 5];
  uint32_t qn = 0;  // warp-uniform
  const uint64_t n = a.n;
  const uint64_t stride = (uint64_t)gridDim.x * BLOCK;
  const uint64_t iters = (n + stride - 1) / stride;
  auto clampi = [&](uint32_t v) { return v < n ? v : (uint32_t)(n - 1); };
  // adaptive resampling: without a resampling every slot is its own ancestor
  bool rs = true;
  R mR = 0;
  if constexpr (ESS) {
    rs = c->resamp != 0;
    if constexpr (sizeof(R) == 4) mR = dec_f((uint32_t)c->maxenc);
    else mR = dec_d(c->maxenc);
  }
  auto ancx = [&](uint64_t k) -> uint32_t {
    if constexpr (ESS) {
      if (!rs) return (uint32_t)k;
    }
    return clampi(a.anc[k]);
  };
  // the carried log-weight of slot j: 0 after a resampling, else L_j - m
  auto carry = [&](uint64_t k) {
    if (rs) {
      a.lam[k] = (R)0;
    } else {
      a.lam[k] = a.ell[k] - mR;
      a.anc[k] = (uint32_t)k;
    }
  };
  bool fail = false;
  // next cycle's weights (FUSE)
  R yn = 0;
  if constexpr (FUSE) yn = (R)(a.y_nx_src ? *a.y_nx_src : a.y_nx_val);
  R mxn = (R)-INFINITY;
  bool badn = false;
  auto finish = [&](const Item& itm) {
    const bool sig = (itm.which & 1u) == 0;
    const R G = gamma_mt_from<R>(sig ? ds : dt, sig ? cs : ct, sig ? ks : kt, itm.Z, itm.U, a.seed,
                                 a.filter, t, itm.j, sig ? P_GAMMA_SIGMA : P_GAMMA_TAU, &fail);
    const R v = SuffOps<R>::ig(itm.b, G);
    if (sig) dst.s2[itm.j] = v;
    else dst.t2[itm.j] = v;
  };
  auto weigh_late = [&](const Item& itm) {  // FUSE: the slot's state is final
    weigh_next<R>(a.ell, itm.j, dst.x[itm.j], dst.s2[itm.j], dst.t2[itm.j], yn, mxn, badn);
  };
  uint64_t j = spread_slot();
  uint32_t an = j < n ? ancx(j) : 0;
  uint32_t an_next = j + stride < n ? ancx(j + stride) : 0;
  Gathered<R> cur = gather_rec<R>(src, an);
  for (uint64_t it = 0; it < iters; ++it, j += stride) {
    // prefetch: the index two slots ahead, the record one slot ahead
    const uint32_t an_next2 = j + 2 * stride < n ? ancx(j + 2 * stride) : 0;
    const Gathered<R> nxt = gather_rec<R>(src, an_next);
    bool defer_s = false, defer_t = false;
    typename SuffT<R>::B bsn = 0, btn = 0;
    R Zs = 0, Us = 0, Zt = 0, Ut = 0;
    R xj = 0, s2n = 0, t2n = 0;
    if (j < n) {
      const R xa = cur.x, sa = cur.s2, ta = cur.t2;
      // V and mu share one correctly rounded reciprocal of s
      const R s = sa + ta;
      const R ri = div_rn((R)1, s);
      const R p = sa * ta;
      const R V = p * ri;
      const R n2 = yr * ta;
      const R nn = fmaR(xa, sa, n2);
      const R mu = nn * ri;
      const R sv = sqrt_rn(V);
      R Z;
      theta_draws_rk<R>(a.rk, a.filter, t, (uint32_t)j, &Z, &Zs, &Us, &Zt, &Ut);
      xj = fmaR(sv, Z, mu);
      dst.x[j] = xj;
      if (LEARN) {
        const R rs = ResidObs<R>::f(y, yr, xj);
        const R rt = xj - xa;
        bsn = SuffOps<R>::add_half_square(cur.bs, rs, &fail);
        btn = SuffOps<R>::add_half_square(cur.bt, rt, &fail);
        dst.bs[j] = bsn;
        dst.bt[j] = btn;
        R Gs, Gt;
        if (gamma_mt_squeeze<R>(ds, cs, ks, Zs, Us, &Gs)) dst.s2[j] = s2n = SuffOps<R>::ig(bsn, Gs);
        else defer_s = true;
        if (gamma_mt_squeeze<R>(dt, ct, kt, Zt, Ut, &Gt)) dst.t2[j] = t2n = SuffOps<R>::ig(btn, Gt);
        else defer_t = true;
      } else {
        dst.s2[j] = s2n = sa;
        dst.t2[j] = t2n = ta;
        dst.bs[j] = cur.bs;
        dst.bt[j] = cur.bt;
      }
      if (FUSE && !defer_s && !defer_t) weigh_next<R>(a.ell, j, xj, s2n, t2n, yn, mxn, badn);
      if constexpr (ESS) carry(j);
    }
    if constexpr (LEARN && FUSE) {
      // the sigma^2 item sits below the tau^2 item of its slot, so it is
      // finished in the same round or a later one: it weighs the slot when
      // both were deferred
      wq_push(wq, qn, defer_s, Item{bsn, Zs, Us, (uint32_t)j, 2u}, lane);
      wq_push(wq, qn, defer_t, Item{btn, Zt, Ut, (uint32_t)j, defer_s ? 1u : 3u}, lane);
      wq_drain_post(wq, qn, 32u, lane, finish, weigh_late);
    } else if constexpr (LEARN) {
      // queue the draws that missed the squeeze; the warp finishes them 32
      // at a time
      wq_push(wq, qn, defer_s, Item{bsn, Zs, Us, (uint32_t)j, 0u}, lane);
      wq_push(wq, qn, defer_t, Item{btn, Zt, Ut, (uint32_t)j, 1u}, lane);
      wq_drain(wq, qn, 32u, lane, finish);
    }
    cur = nxt;
    an_next = an_next2;
  }
  if constexpr (LEARN && FUSE) wq_drain_post(wq, qn, 1u, lane, finish, weigh_late);
  else if (LEARN) wq_drain(wq, qn, 1u, lane, finish);
  (void)an;
  if (__any_sync(0xffffffffu, fail || badn) && lane == 0) atomicOr(&a.ctl->err, ERR_NUMERIC);
  // Without FUSE the fold reads only what earlier kernels wrote (tile
  // partials, the control block), so the completion count needs no fence;
  // every warp has read t before its increment.  With FUSE each warp's
  // maximum is fenced before its count.
  if constexpr (FUSE) publish_next_max<R>(a.ctl, mxn, lane);
  bool last = false;
  if (lane == 0) last = atomicAdd(&a.ctl->done_prop, 1u) == gridDim.x * WARPS - 1;
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last) fold_cycle_warp<R, FUSE, ESS>(a, t);
}

// ---------------------------------------------------------------------------
// k_propagate for binary32 state, two slots per thread per pass: the pair
// 2i, 2i + 1, which shares its second draw (theta_draws2), shares each paired
// FMUL2 / FFMA2, its quotients and roots among them (state_scale2, ig2), while
// additions, comparisons and the fixed-point statistics run per lane.  Per slot the operations are those of
// the scalar propagation, in the same order, so the results are the same bits.
// ---------------------------------------------------------------------------
constexpr uint32_t WQ2_CAP = 160;  // 31 queued + 4 pushes of 32 per pass
// k_propagate2's units of 64 slots: with DYN handed out by ticket, PROP_GRAB
// at a time.  Tickets even out the warps' finishing times, but each batch waits
// for an atomic and costs the address arithmetic of an arbitrary unit, so they
// pay only where a warp has many units: the launch takes DYN from PROP_DYN units
// per warp (PROP_DYN_ESS with adaptive resampling), learning forms only.  Cycle
// in us, fixed / by ticket: N = 2^22 105.9 / 111.0, 2^23 193.4 / 196.6, 2^24
// 366.1 / 365.7, 2^25 709.6 / 700.4; adaptive 2^22 121.6 / 126.0, 10^7 260.4 /
// 260.1, 2^24 419.2 / 413.8.  Fixed is the faster at every size with FUSE (2^22
// 108.0 / 119.0, 2^24 365.0 / 387.6, 2^26 1390 / 1453) and with known variances
// (2^22 88.6 / 96.3, 2^24 299.7 / 314.7, 2^26 1140 / 1210), which therefore have
// no ticket form.
constexpr uint32_t PROP_GRAB = 4;
constexpr uint32_t PROP_DYN = 68, PROP_DYN_ESS = 44;

// With FUSE, the next cycle's weights as in k_propagate, the two slots of a
// pass weighed by paired operations.
// 3 CTAs per SM (up to 85 registers, no spills): measured faster at N = 2^24
// than 4 CTAs at 64 registers, where the plain form spills.
// As 128 threads x 7 CTAs the cycle of 2^24 takes 0.4 % less, but the adaptive
// one of 2^20 4 % and the fused one of 2.6 million 3 % more.
template <bool LEARN, bool FUSE = false, bool ESS = false, bool DYN = false>
__global__ void __launch_bounds__(BLOCK, 3) k_propagate2(FilterArgs<float> a) {
  static_assert(!DYN || (LEARN && !FUSE), "tickets: learning forms without FUSE");
  typedef GammaItem<float> Item;
  __shared__ Item s_q[WARPS][WQ2_CAP];
  const Ctl* c = a.ctl;
  const uint32_t t = c->t;
  const StateV<float> src = (t & 1) ? a.st[1] : a.st[0];
  const StateV<float> dst = (t & 1) ? a.st[0] : a.st[1];
  const float yr = c->yf, ds = c->mtf[0], cs = c->mtf[1], dt = c->mtf[2], ct = c->mtf[3];
  const float ks = c->mtf[4], kt = c->mtf[5];
  const bool wide = ig_wide(ds, dt);
  const int lane = threadIdx.x & 31;
  Item* const wq = s_q[threadIdx.x >> 5];
  uint32_t qn = 0;  // warp-uniform
  const uint64_t n = a.n;
  auto clampi = [&](uint32_t v) { return v < n ? v : (uint32_t)(n - 1); };
  // adaptive resampling: without a resampling every slot is its own ancestor
  bool rs = true;
  float mR = 0.0f;
  if constexpr (ESS) {
    rs = c->resamp != 0;
    mR = dec_f((uint32_t)c->maxenc);
  }
  // the carried log-weight of slot j: 0 after a resampling, else L_j - m
  auto carry = [&](uint64_t k) {
    if (rs) {
      a.lam[k] = 0.0f;
    } else {
      a.lam[k] = a.ell[k] - mR;
      a.anc[k] = (uint32_t)k;
    }
  };
  bool fail = false;
  // next cycle's weights (FUSE)
  float yn = 0.0f;
  if constexpr (FUSE) yn = (float)(a.y_nx_src ? *a.y_nx_src : a.y_nx_val);
  float mxn = -INFINITY;
  bool badn = false;
  auto finish = [&](const Item& itm) {
    const bool sig = (itm.which & 1u) == 0;
    const float G = gamma_mt_from<float>(sig ? ds : dt, sig ? cs : ct, sig ? ks : kt, itm.Z,
                                         itm.U, a.seed, a.filter, t, itm.j,
                                         sig ? P_GAMMA_SIGMA : P_GAMMA_TAU, &fail);
    const float v = SuffOps<float>::ig(itm.b, G);
    if (sig) dst.s2[itm.j] = v;
    else dst.t2[itm.j] = v;
  };
  auto weigh_late = [&](const Item& itm) {  // FUSE: the slot's state is final
    weigh_next<float>(a.ell, itm.j, dst.x[itm.j], dst.s2[itm.j], dst.t2[itm.j], yn, mxn, badn);
  };
  // Slots go out in units of 64: lane l of a warp takes the pair j0 = 64 u +
  // 2 l, j1 = j0 + 1 of unit u (the two slots that share a draw), so its
  // ancestor load and its stores are 8 or 16 bytes wide.  Without DYN, pass
  // p of warp w (of the grid's W) is unit p W + w.  With DYN (many units per
  // warp) a warp takes PROP_GRAB consecutive units per ticket, each ticket
  // taken a batch ahead of its use, so that a warp on a slower SM (or with
  // more draws that missed the squeeze) takes fewer of them and the kernel
  // ends with its work: under the fixed assignment the CTAs' finishing times
  // at N = 2^24 spread from 187 to 234 us.  A slot's arithmetic does not
  // depend on the warp that computes it.
  const uint64_t nunits = (n + 63) / 64;
  const uint64_t stride = (uint64_t)gridDim.x * BLOCK * 2;  // slots per pass
  const uint64_t iters = (n + stride - 1) / stride;
  unsigned long long tick = 0;  // lane 0: the ticket of the next batch
  uint64_t u = 0;
  uint64_t j0 = 2 * ((uint64_t)blockIdx.x * BLOCK + threadIdx.x);
  if constexpr (DYN) {
    if (lane == 0) tick = atomicAdd(&a.ctl->prop_ticket, (unsigned long long)PROP_GRAB);
    u = __shfl_sync(0xffffffffu, tick, 0);
    if (lane == 0) tick = atomicAdd(&a.ctl->prop_ticket, (unsigned long long)PROP_GRAB);
    j0 = u * 64 + 2 * (uint64_t)lane;
  }
  (void)nunits; (void)iters; (void)u;
  // the ancestors of the pair starting at slot j (even; clamped into range)
  auto anc_pair = [&](uint64_t j) -> uint2 {
    if constexpr (ESS) {  // (past the end: the last slot, a valid address)
      if (!rs) return make_uint2(clampi((uint32_t)j), clampi((uint32_t)j + 1u));
    }
    if (j + 1 < n) {
      const uint2 v = *reinterpret_cast<const uint2*>(a.anc + j);
      return make_uint2(clampi(v.x), clampi(v.y));
    }
    return make_uint2(j < n ? clampi(a.anc[j]) : 0u, 0u);
  };
  uint2 an = anc_pair(j0);
  Gathered<float> c0 = gather_rec<float>(src, an.x);
  Gathered<float> c1 = gather_rec<float>(src, an.y);
  for (uint64_t it = 0; DYN ? u < nunits : it < iters; ++it) {  // (the same in every lane)
    // the next pair: the next pass's; with DYN the next unit of the batch,
    // or the first of the batch taken a batch ago (then the ticket of the
    // batch after it)
    uint64_t jn = j0 + stride;
    uint64_t un = u + 1;
    if constexpr (DYN) {
      if (un % PROP_GRAB == 0) {
        un = __shfl_sync(0xffffffffu, tick, 0);
        if (lane == 0 && un < nunits) tick = atomicAdd(&a.ctl->prop_ticket, (unsigned long long)PROP_GRAB);
      }
      jn = un * 64 + 2 * (uint64_t)lane;
    }
    const uint64_t j1 = j0 + 1;
    const bool v0 = j0 < n, v1 = j1 < n;
    // the next unit's records, gathered ahead
    const uint2 na = anc_pair(jn);
    const Gathered<float> n0 = gather_rec<float>(src, na.x);
    const Gathered<float> n1 = gather_rec<float>(src, na.y);
    // the last unit may be partial: a warp skips it when no lane has a slot
    if (__any_sync(0xffffffffu, v0)) {
      const float2 xa = make_float2(c0.x, c1.x), sa = make_float2(c0.s2, c1.s2);
      const float2 ta = make_float2(c0.t2, c1.t2);
      // V and mu share one correctly rounded reciprocal of s = sigma^2 + tau^2
      const float2 sm = addp(sa, ta);
      float2 ri, sv;
      state_scale2(sa, ta, sm, &ri, &sv);
      const float2 nn = fma2(xa, sa, mul2(splat2(yr), ta));
      const float2 mu = mul2(nn, ri);
      float2 Z, Zs, Us, Zt, Ut;
      theta_draws2(a.rk, a.filter, t, (uint32_t)(j0 >> 1), &Z, &Zs, &Us, &Zt, &Ut);
      const float2 xj = fma2(sv, Z, mu);
      if (v1) {
        *reinterpret_cast<float2*>(dst.x + j0) = xj;
      } else if (v0) {
        dst.x[j0] = xj.x;
      }
      bool ds0 = false, dt0 = false, ds1 = false, dt1 = false;
      uint64_t bs0 = 0, bt0 = 0, bs1 = 0, bt1 = 0;
      if (LEARN) {
        const float2 rs = addp(splat2(yr), make_float2(-xj.x, -xj.y));
        const float2 rt = addp(xj, make_float2(-xa.x, -xa.y));
        // b + r^2 / 2 in 2^-32 fixed point, per SuffOps<float>::add_half_square
        const float2 ws = mul2(mul2(rs, rs), splat2(0x1p31f));
        const float2 wt = mul2(mul2(rt, rt), splat2(0x1p31f));
        bool f0 = false, f1 = false;
        auto addb = [&](uint64_t b, float v, bool* f) -> uint64_t {
          if (!(v < 0x1p63f)) {
            *f = true;
            return b;
          }
          return b + SuffOps<float>::incr(v);
        };
        bs0 = addb(c0.bs, ws.x, &f0);
        bt0 = addb(c0.bt, wt.x, &f0);
        bs1 = addb(c1.bs, ws.y, &f1);
        bt1 = addb(c1.bt, wt.y, &f1);
        fail |= (v0 && f0) || (v1 && f1);
        if (v1) {
          *reinterpret_cast<ulonglong2*>(dst.bs + j0) = make_ulonglong2(bs0, bs1);
          *reinterpret_cast<ulonglong2*>(dst.bt + j0) = make_ulonglong2(bt0, bt1);
        } else if (v0) {
          dst.bs[j0] = bs0;
          dst.bt[j0] = bt0;
        }
        // Marsaglia-Tsang squeeze for sigma^2 (x lanes: slot j0, j1) and tau^2
        const float2 vs = fma2(splat2(cs), Zs, splat2(1.0f)), vt = fma2(splat2(ct), Zt, splat2(1.0f));
        const float2 v3s = mul2(mul2(vs, vs), vs), v3t = mul2(mul2(vt, vt), vt);
        const float2 Z2s = mul2(Zs, Zs), Z2t = mul2(Zt, Zt);
        const float2 thrs = fma2(splat2(-ks), mul2(Z2s, Z2s), splat2(1.0f));
        const float2 thrt = fma2(splat2(-kt), mul2(Z2t, Z2t), splat2(1.0f));
        const float2 Gs = mul2(splat2(ds), v3s), Gt = mul2(splat2(dt), v3t);
        const bool as0 = vs.x > 0.0f && Us.x < thrs.x, as1 = vs.y > 0.0f && Us.y < thrs.y;
        const bool at0 = vt.x > 0.0f && Ut.x < thrt.x, at1 = vt.y > 0.0f && Ut.y < thrt.y;
        // inverse gamma: (b 2^-32) / G, per SuffOps<float>::ig.  The divisions
        // run for every lane (no branch around them); a draw that missed the
        // squeeze stores nothing here and is finished from the warp's queue.
        const float2 bsf = fma2(make_float2(__uint2float_rn((uint32_t)bs0), __uint2float_rn((uint32_t)bs1)),
                                splat2(0x1p-32f),
                                make_float2(__uint2float_rn((uint32_t)(bs0 >> 32)),
                                            __uint2float_rn((uint32_t)(bs1 >> 32))));
        const float2 btf = fma2(make_float2(__uint2float_rn((uint32_t)bt0), __uint2float_rn((uint32_t)bt1)),
                                splat2(0x1p-32f),
                                make_float2(__uint2float_rn((uint32_t)(bt0 >> 32)),
                                            __uint2float_rn((uint32_t)(bt1 >> 32))));
        const float2 qs = ig2(bsf, Gs, wide), qt = ig2(btf, Gt, wide);
        const float q0 = qs.x, r0 = qt.x, q1 = qs.y, r1 = qt.y;
        ds0 = v0 && !as0; dt0 = v0 && !at0; ds1 = v1 && !as1; dt1 = v1 && !at1;
        if (v1 && as0 && as1) {
          *reinterpret_cast<float2*>(dst.s2 + j0) = make_float2(q0, q1);
        } else {
          if (v0 && as0) dst.s2[j0] = q0;
          if (v1 && as1) dst.s2[j1] = q1;
        }
        if (v1 && at0 && at1) {
          *reinterpret_cast<float2*>(dst.t2 + j0) = make_float2(r0, r1);
        } else {
          if (v0 && at0) dst.t2[j0] = r0;
          if (v1 && at1) dst.t2[j1] = r1;
        }
        // 1 for a deferred draw: the paired weight of that slot is discarded,
        // and a normal operand keeps the log and the division on their fast paths
        const float s20 = as0 ? q0 : 1.0f, t20 = at0 ? r0 : 1.0f;
        const float s21 = as1 ? q1 : 1.0f, t21 = at1 ? r1 : 1.0f;
        // queue the draws that missed the squeeze (rare: K Z^4 is small for
        // the shapes of a running filter); the warp finishes them 32 at a time
        const bool any_def = __any_sync(0xffffffffu, ds0 || dt0 || ds1 || dt1);
        if constexpr (FUSE) {
          // both slots weighed paired; a slot with a deferred draw is weighed
          // by the drain round that finishes it (its sigma^2 item lies below
          // its tau^2 item, so it weighs when both were deferred)
          const float2 l = log_pred2(xj, make_float2(s20, s21), make_float2(t20, t21), yn);
          if (v0 && !ds0 && !dt0) keep_next(a.ell, j0, l.x, mxn, badn);
          if (v1 && !ds1 && !dt1) keep_next(a.ell, j1, l.y, mxn, badn);
          if (any_def) {
            wq_push(wq, qn, ds0, Item{bs0, Zs.x, Us.x, (uint32_t)j0, 2u}, lane);
            wq_push(wq, qn, dt0, Item{bt0, Zt.x, Ut.x, (uint32_t)j0, ds0 ? 1u : 3u}, lane);
            wq_push(wq, qn, ds1, Item{bs1, Zs.y, Us.y, (uint32_t)j1, 2u}, lane);
            wq_push(wq, qn, dt1, Item{bt1, Zt.y, Ut.y, (uint32_t)j1, ds1 ? 1u : 3u}, lane);
            wq_drain_post(wq, qn, 32u, lane, finish, weigh_late);
          }
        } else {
          (void)s20; (void)t20; (void)s21; (void)t21;
          if (any_def) {
            wq_push(wq, qn, ds0, Item{bs0, Zs.x, Us.x, (uint32_t)j0, 0u}, lane);
            wq_push(wq, qn, dt0, Item{bt0, Zt.x, Ut.x, (uint32_t)j0, 1u}, lane);
            wq_push(wq, qn, ds1, Item{bs1, Zs.y, Us.y, (uint32_t)j1, 0u}, lane);
            wq_push(wq, qn, dt1, Item{bt1, Zt.y, Ut.y, (uint32_t)j1, 1u}, lane);
            wq_drain(wq, qn, 32u, lane, finish);
          }
        }
      } else {
        if (v0) { dst.s2[j0] = sa.x; dst.t2[j0] = ta.x; dst.bs[j0] = c0.bs; dst.bt[j0] = c0.bt; }
        if (v1) { dst.s2[j1] = sa.y; dst.t2[j1] = ta.y; dst.bs[j1] = c1.bs; dst.bt[j1] = c1.bt; }
        if constexpr (FUSE) {
          const float2 l = log_pred2(xj, sa, ta, yn);
          if (v0) keep_next(a.ell, j0, l.x, mxn, badn);
          if (v1) keep_next(a.ell, j1, l.y, mxn, badn);
        }
      }
      if constexpr (ESS) {
        if (v0) carry(j0);
        if (v1) carry(j1);
      }
    }
    c0 = n0;
    c1 = n1;
    u = un;
    j0 = jn;
  }
  if constexpr (LEARN && FUSE) wq_drain_post(wq, qn, 1u, lane, finish, weigh_late);
  else if (LEARN) wq_drain(wq, qn, 1u, lane, finish);
  if (__any_sync(0xffffffffu, fail || badn) && lane == 0) atomicOr(&a.ctl->err, ERR_NUMERIC);
  if constexpr (FUSE) publish_next_max<float>(a.ctl, mxn, lane);
  bool last = false;
  if (lane == 0) last = atomicAdd(&a.ctl->done_prop, 1u) == gridDim.x * WARPS - 1;
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last) fold_cycle_warp<float, FUSE, ESS>(a, t);
}

// ---------------------------------------------------------------------------
// The bootstrap filter's Step 3 completed: the resampled particles are the
// propagated ones at the ancestors (in place in the current buffer), copied
// into the other buffer; the last warp folds the log-ML increment and
// advances t, as in the propagation kernels.
// ---------------------------------------------------------------------------
template <class R>
__global__ void __launch_bounds__(BLOCK) k_boot_gather(FilterArgs<R> a) {
  const uint32_t t = a.ctl->t;
  const StateV<R> src = (t & 1) ? a.st[1] : a.st[0];
  const StateV<R> dst = (t & 1) ? a.st[0] : a.st[1];
  const uint64_t n = a.n;
  // (grid-stride and one completion count per CTA: a count per warp of a grid of
  // all slots, 32,768 atomics on one word at N = 2^20, held the kernel at 37 us)
  const uint64_t stride = (uint64_t)gridDim.x * BLOCK;
#pragma unroll 2
  for (uint64_t j = (uint64_t)blockIdx.x * BLOCK + threadIdx.x; j < n; j += stride) {
    uint32_t an = a.anc[j];
    an = an < n ? an : (uint32_t)(n - 1);
    dst.x[j] = src.x[an];
    dst.s2[j] = src.s2[an];
    dst.t2[j] = src.t2[an];
    dst.bs[j] = src.bs[an];
    dst.bt[j] = src.bt[an];
  }
  __syncthreads();  // every warp has read t
  if (threadIdx.x >= 32) return;
  bool last = false;
  if (threadIdx.x == 0) last = atomicAdd(&a.ctl->done_prop, 1u) == gridDim.x - 1;
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last) fold_cycle_warp<R>(a, t);
}

// ---------------------------------------------------------------------------
// Posterior summaries (on demand): population means and variances of x,
// sigma^2 and tau^2, from sums of v - c and (v - c)^2 with c the value of
// particle 0 (a shift against cancellation).  Each thread sums its
// EST_PER_THREAD consecutive particles (vector loads) and each warp its
// lanes by a shuffle tree in the working precision; the warps of a block are
// joined in binary64, and the last block to finish folds the block partials
// in binary64 (each thread a fixed stride of blocks, then a shuffle tree):
// the result is run-to-run deterministic and binary64 arithmetic runs per
// block, not per particle (binary64 is a small fraction of the binary32 rate
// on this part).
// ---------------------------------------------------------------------------
constexpr int EST_PER_THREAD = 16;

// The control block's prefix up to the per-cycle constants (t, error word,
// counters, log-ML, summaries) written to the mapped host mirror, one 8-byte
// word per thread (called by every thread of the block, after a barrier that
// follows the writes to the control block); the host reads the mirror after
// synchronising with the stream, which orders these writes.
constexpr int SUMMARY_WORDS = (int)(offsetof(Ctl, y) / 8);
__device__ __forceinline__ void publish_summary(const Ctl* c, Ctl* mirror) {
  static_assert(offsetof(Ctl, y) % 8 == 0 && SUMMARY_WORDS <= 32, "prefix of whole words");
  if (!mirror || threadIdx.x >= SUMMARY_WORDS) return;
  reinterpret_cast<unsigned long long*>(mirror)[threadIdx.x] =
      __ldcg(reinterpret_cast<const unsigned long long*>(c) + threadIdx.x);
}
// After publish_summary, by the whole block: the host's sequence number to
// io->seq_out, ordered after every mirror word (each writer's system-scope
// fence, the block barrier, a release store).
__device__ __forceinline__ void publish_done(EstIO* io) {
  if (!io) return;
  __threadfence_system();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long sq = *reinterpret_cast<volatile unsigned long long*>(&io->seq_in);
    asm volatile("st.release.sys.global.u64 [%0], %1;" ::"l"(&io->seq_out), "l"(sq) : "memory");
  }
}

// Means and variances from the shifted sums (sum of v - c, sum of (v - c)^2
// per quantity) over n particles, one reciprocal of n.
__device__ __forceinline__ void est_finish(const double* tot, double n, const double* cs,
                                           double* out) {
  const double inv_n = div_rn(1.0, n);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const double m1 = tot[2 * q] * inv_n;
    const double m2 = tot[2 * q + 1] * inv_n;
    out[2 * q] = cs[q] + m1;
    out[2 * q + 1] = m2 - m1 * m1;
  }
}

template <class R>
__device__ __forceinline__ void est_add(R* loc, R v0, R v1, R v2, R c0, R c1, R c2) {
  const R dx = v0 - c0, ds = v1 - c1, dt = v2 - c2;
  loc[0] += dx; loc[1] += dx * dx;
  loc[2] += ds; loc[3] += ds * ds;
  loc[4] += dt; loc[5] += dt * dt;
}

// The sums of block b of BLOCK x EST_PER_THREAD particles, to part_est (the
// state is read through L2: the caller may have written it in this launch).
template <class R>
__device__ __forceinline__ void est_block(const StateV<R>& st, uint64_t n, uint32_t b, R c0, R c1,
                                          R c2, double (*s_sum)[WARPS], double* part_est) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  {
    R loc[6] = {0, 0, 0, 0, 0, 0};
    const uint64_t base = ((uint64_t)b * BLOCK + threadIdx.x) * EST_PER_THREAD;
    if constexpr (sizeof(R) == 4) {
      if (base + EST_PER_THREAD <= n) {
        float4 X[EST_PER_THREAD / 4], S[EST_PER_THREAD / 4], T[EST_PER_THREAD / 4];
#pragma unroll
        for (int q = 0; q < EST_PER_THREAD / 4; ++q) {
          X[q] = __ldcg(reinterpret_cast<const float4*>(st.x + base + 4 * q));
          S[q] = __ldcg(reinterpret_cast<const float4*>(st.s2 + base + 4 * q));
          T[q] = __ldcg(reinterpret_cast<const float4*>(st.t2 + base + 4 * q));
        }
#pragma unroll
        for (int q = 0; q < EST_PER_THREAD / 4; ++q) {
          est_add<float>(loc, X[q].x, S[q].x, T[q].x, c0, c1, c2);
          est_add<float>(loc, X[q].y, S[q].y, T[q].y, c0, c1, c2);
          est_add<float>(loc, X[q].z, S[q].z, T[q].z, c0, c1, c2);
          est_add<float>(loc, X[q].w, S[q].w, T[q].w, c0, c1, c2);
        }
      } else {
        for (uint64_t i = base; i < n; ++i)
          est_add<R>(loc, __ldcg(st.x + i), __ldcg(st.s2 + i), __ldcg(st.t2 + i), c0, c1, c2);
      }
    } else {
#pragma unroll 4
      for (int e = 0; e < EST_PER_THREAD; ++e) {
        const uint64_t i = base + e;
        if (i < n) est_add<R>(loc, __ldcg(st.x + i), __ldcg(st.s2 + i), __ldcg(st.t2 + i), c0, c1, c2);
      }
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      R v = loc[q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) s_sum[q][warp] = (double)v;
    }
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double v = 0;
    for (int w = 0; w < WARPS; ++w) v += s_sum[threadIdx.x][w];
    part_est[(uint64_t)b * 6 + threadIdx.x] = v;
  }
  __syncthreads();  // (s_sum is reused; the sums are visible to the block)
}

// The sums of nblk blocks folded into s_tot: thread i sums blocks i, i + BLOCK,
// ... (a fixed assignment), then a shuffle tree per warp and the warps in order.
__device__ __forceinline__ void est_fold_sums(const double* part_est, uint32_t nblk,
                                              double (*s_sum)[WARPS], double* s_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // (a warp without a block adds zeros, which change no sum: it is left out)
  const int nw = nblk >= BLOCK ? WARPS : (int)((nblk + 31) / 32);
  if (warp < nw) {
    double v[6] = {0, 0, 0, 0, 0, 0};
    for (uint32_t b = threadIdx.x; b < nblk; b += BLOCK) {
#pragma unroll
      for (int q = 0; q < 6; ++q) v[q] += __ldcg(part_est + (uint64_t)b * 6 + q);
    }
    if (nblk > 1) {
#pragma unroll
      for (int q = 0; q < 6; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
      }
    }
    // (s_sum was last read before the caller's barrier)
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < 6; ++q) s_sum[q][warp] = v[q];
    }
  }
  __syncthreads();
  if (threadIdx.x < 6) {  // the warps in order, one quantity per thread
    double v = 0;
    for (int w = 0; w < nw; ++w) v += s_sum[threadIdx.x][w];
    s_tot[threadIdx.x] = v;
  }
  __syncthreads();
}

// The fold, and the summaries written and published.
template <class R>
__device__ __forceinline__ void est_fold(const FilterArgs<R>& a, uint32_t t, uint32_t nblk, R c0, R c1,
                                         R c2, double (*s_sum)[WARPS], double* s_tot) {
  est_fold_sums(a.part_est, nblk, s_sum, s_tot);
  if (threadIdx.x == 0) {
    const double cs[3] = {(double)c0, (double)c1, (double)c2};
    a.ctl->est[0] = (double)t;
    est_finish(s_tot, (double)a.n, cs, a.ctl->est + 1);
    a.ctl->est[7] = a.ctl->logml;
    a.ctl->done_est = 0;
  }
  __syncthreads();
  publish_summary(a.ctl, a.ctl_mirror);
  publish_done(a.io);
}

template <class R>
__global__ void __launch_bounds__(BLOCK) k_estimate(FilterArgs<R> a) {
  __shared__ double s_sum[6][WARPS];
  __shared__ double s_tot[6];
  __shared__ bool s_last;
  const uint32_t t = a.ctl->t;
  const StateV<R> st = (t & 1) ? a.st[1] : a.st[0];
  const R c0 = st.x[0], c1 = st.s2[0], c2 = st.t2[0];
  est_block<R>(st, a.n, blockIdx.x, c0, c1, c2, s_sum, a.part_est);
  if (threadIdx.x == 0) {  // (the block's sums were written before its last barrier)
    __threadfence();
    s_last = atomicAdd(&a.ctl->done_est, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  est_fold<R>(a, t, gridDim.x, c0, c1, c2, s_sum, s_tot);
}

// Posterior summaries under adaptive resampling: the particles weighted by
// w_i = exp(lambda_i) (the CDF's deterministic exp).  Per block: sums of w,
// w (v - c) and w (v - c)^2 with c the value of particle 0, in binary64; the
// last block folds the block partials in block order.
template <class R>
__global__ void __launch_bounds__(BLOCK) k_estimate_w(FilterArgs<R> a) {
  __shared__ double s_sum[7][WARPS];
  __shared__ bool s_last;
  const uint32_t t = a.ctl->t;
  const StateV<R> st = (t & 1) ? a.st[1] : a.st[0];
  const R c0 = st.x[0], c1 = st.s2[0], c2 = st.t2[0];
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  const uint64_t base = ((uint64_t)blockIdx.x * BLOCK + threadIdx.x) * EST_PER_THREAD;
  for (int e = 0; e < EST_PER_THREAD; ++e) {
    const uint64_t i = base + e;
    if (i < a.n) {
      R wr;
      (void)quant_exp(a.lam[i], a.k, &wr);
      const double w = (double)wr;
      const double dx = (double)(st.x[i] - c0), ds = (double)(st.s2[i] - c1),
                   dt = (double)(st.t2[i] - c2);
      acc[0] += w;
      acc[1] += w * dx; acc[2] += w * (dx * dx);
      acc[3] += w * ds; acc[4] += w * (ds * ds);
      acc[5] += w * dt; acc[6] += w * (dt * dt);
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    double v = acc[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s_sum[q][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x < 7) {
    double v = 0;
    for (int w = 0; w < WARPS; ++w) v += s_sum[threadIdx.x][w];
    a.part_est[(uint64_t)blockIdx.x * 7 + threadIdx.x] = v;
  }
  __syncthreads();  // all seven sums, before the count that announces them
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&a.ctl->done_est, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (threadIdx.x < 7) {
    double v = 0;
    for (uint32_t b = 0; b < gridDim.x; ++b) v += __ldcg(a.part_est + (uint64_t)b * 7 + threadIdx.x);
    s_sum[threadIdx.x][0] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double sw = s_sum[0][0];
    const double cs[3] = {(double)c0, (double)c1, (double)c2};
    a.ctl->est[0] = (double)t;
    for (int q = 0; q < 3; ++q) {
      const double m1 = s_sum[1 + 2 * q][0] / sw;
      const double m2 = s_sum[2 + 2 * q][0] / sw;
      a.ctl->est[1 + 2 * q] = cs[q] + m1;
      a.ctl->est[2 + 2 * q] = m2 - m1 * m1;
    }
    a.ctl->est[7] = a.ctl->logml;
    a.ctl->done_est = 0;
  }
  __syncthreads();
  publish_summary(a.ctl, a.ctl_mirror);
  publish_done(a.io);
}

// Maximum of binary32 input weights (pf_resample): non-negative floats order
// as their bit patterns (-0 is a zero weight).  With vec, 32-byte aligned w: a
// thread's eight weights per load, two loads in flight.
static __global__ void __launch_bounds__(BLOCK) k_wmax(const float* w, uint64_t n, Ctl* ctl, int vec) {
  __shared__ uint32_t s_red[WARPS];
  uint32_t mx = 0;
  bool bad = false;
  auto take = [&](float v) {
    if (!(v >= 0.0f) || !(v < INFINITY)) bad = true;
    else mx = max(mx, __float_as_uint(fabsf(v)));
  };
  const uint64_t nt = (uint64_t)gridDim.x * BLOCK, id = (uint64_t)blockIdx.x * BLOCK + threadIdx.x;
  const uint64_t n8 = vec ? n / 8 : 0;
  for (uint64_t i = id; i < n8; i += 2 * nt) {
    float v[16];
    const bool two = i + nt < n8;
    ld8(w + 8 * i, v);
    if (two) ld8(w + 8 * (i + nt), v + 8);
#pragma unroll
    for (int e = 0; e < 8; ++e) take(v[e]);
    if (two) {
#pragma unroll
      for (int e = 8; e < 16; ++e) take(v[e]);
    }
  }
  for (uint64_t i = 8 * n8 + id; i < n; i += nt) take(w[i]);
  if (bad) atomicOr(&ctl->err, ERR_WEIGHTS);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_red[warp] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < WARPS; ++i) mx = max(mx, s_red[i]);
    mx = max(mx, s_red[0]);
    atomicMax(&ctl->maxenc, (unsigned long long)mx);
  }
}

}  // namespace pfk
