// The CDF and the resampling of a cycle (Steps 1b-1c) in two launches over
// tiles of 2048 particles:
//   k_sums   the exact sum of each tile's quantised weights; the last CTA
//            turns the sums into exclusive prefixes and writes the total T
//            and the constants of the slot map;
//   k_slots  each tile's CDF values from its prefix, the number of slots
//            below each, and the ancestors of the tile's slots, stored out
//            coalesced.
// For the systematic and stratified schemes the number of slots below a CDF
// value, R(Q), is a function of Q alone (slot_below), so a particle's slots
// [R(Q_{i-1}), R(Q_i)) need no search and no walk over its neighbours.
//
// Both kernels are plain launches of many short CTAs.  Neither is bound by HBM:
// at N = 2^22 k_sums (36 instructions per particle, 16 us) has 13 % of the DRAM
// throughput and issues in 44 % of cycles, k_slots (86 instructions, 19 us) 12 %
// and 61 %; what is left is the latency of each CTA's loads and block scans.
// At 2^24 they take 43 and 61 us; below 2^18 launch latency and the last CTA's
// prefix count.  They replaced one
// cooperative launch of resident CTAs over fixed tile ranges, whose grid
// barrier waited for the slowest CTA and whose per-thread walk was serial.
#pragma once
#include "device.cuh"

namespace pfk {

constexpr int SLOT_PER = 8;                      // particles per thread of k_slots
constexpr int SLOT_TILE = BLOCK * SLOT_PER;      // 2048 particles per tile
constexpr int SUM_PER = 16;                      // particles per thread of k_sums
constexpr int SUM_TILE = BLOCK * SUM_PER;        // 4096: two tiles per CTA
constexpr int SUM_SUB = SUM_TILE / SLOT_TILE;
constexpr uint32_t SLOT_WIN = 2 * SLOT_TILE;     // window slots
constexpr int SLOT_RUNS = 512;                   // runs per tile held in shared memory

// What the weights are read from.
enum SlotSrc : int {
  SRC_LOG = 0,  // binary32 l_i, relative to the maximum in the control block
  SRC_E32 = 1,  // binary32 e_i = exp(l_i - max)
  SRC_E64 = 2,  // binary64 e_i (k_exp), in the space of Q
  SRC_W = 3,    // binary32 weights of the caller (pf_resample)
};
// bytes of the tile prefixes of n particles (a multiple of four tiles), and
// with the heavy list after them (an entry has more than SLOT_WIN - 32 slots)
constexpr size_t pre_bytes(uint64_t n) {
  return ((n + SLOT_TILE - 1) / SLOT_TILE + 3) / 4 * 32;
}
constexpr size_t pre_heavy_bytes(uint64_t n) { return pre_bytes(n) + (n / (SLOT_WIN - 32) + 1) * 8; }
enum SlotPos : int { SLOTS_NONE = 0, SLOTS_SYS = 1, SLOTS_STRAT = 2 };

struct SlotArgs {
  const void* src;
  float* e_out;           // k_sums from l: e_i, or NULL
  uint64_t* Q;            // CDF out, or NULL
  uint32_t* anc;
  uint64_t* pre;          // per tile: its sum, then its exclusive prefix (padded to pre_bytes)
  void* part;             // log-ML partials: the last one is written by the last CTA (binary32)
  void* part_blk;         // per CTA of k_sums (binary32: scratch; binary64: the partials)
  U128* sq;               // per CTA of k_sums: sum of W^2 (adaptive resampling)
  Ctl* ctl;
  const uint32_t* t_dev;
  uint32_t t_arg;
  uint64_t n;
  uint32_t ntiles;        // of SLOT_TILE
  int k;                  // CDF shift
  uint64_t seed;
  uint32_t filter;
  double ess_frac;
  void* heavy;            // heavy list, or NULL (NONE: no windows)
  const double* l;        // binary64: the l_i, for the tiles of the heavy list
  uint32_t* host_err;     // mapped host word for pf_resample's errors, or NULL
  int multi;              // multinomial: S_n is known (k_spacing_sums ran before)
  int cut;                // k_slots builds the cut-point table in anc: the slot map with r = 0
  const uint32_t* gate;   // *gate == 0: this cycle does not resample (NULL: it does)
  int src_vec, anc_vec;   // src is 32-byte and anc 16-byte aligned
};

// 256-bit loads and stores (sm_100+): a thread's eight binary32 values, or
// four 64-bit ones, are one instruction and one full sector.
__device__ __forceinline__ void ld8(const float* p, float* v) {
  asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p) : "memory");
}
__device__ __forceinline__ void st8(float* p, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void ld4(const double* p, double* v) {
  asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
               : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void ld4(const uint64_t* p, uint64_t* v) {
  asm volatile("ld.global.v4.b64 {%0,%1,%2,%3}, [%4];"
               : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void st4(uint64_t* p, uint64_t a, uint64_t b, uint64_t c, uint64_t d) {
  asm volatile("st.global.v4.b64 [%0], {%1,%2,%3,%4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

// The further windows of a tile of weight `sum` that other CTAs store (k_sums
// lists it), 0: its own CTA stores all its windows, up to OWN past the first.
// The estimate of its slots is within 32 of them, so a last window may turn out
// empty.  A window by the tile's own CTA takes 0.9 us, the tile built once more by
// another 2.5, in binary64, where that takes the exponentials again, 5.
template <int SRC>
struct HeavyRule {
  static constexpr uint32_t OWN = SRC == SRC_E64 ? 6 : 0;
  float per_slot;
  uint64_t most;  // a tile of at most this is not listed
  __device__ __forceinline__ HeavyRule(uint64_t T, uint64_t n) {
    const float Tf = __ull2float_rn(T), nf = (float)n;
    per_slot = nf / Tf;
    most = f2u64_rz(Tf * ((float)((OWN + 1) * SLOT_WIN - 16) / nf));
  }
  __device__ __forceinline__ uint32_t operator()(uint64_t sum) const {
    return sum > most ? (uint32_t)((__ull2float_rn(sum) * per_slot + 40.0f) * (1.0f / SLOT_WIN)) : 0u;
  }
};

template <int SRC> struct SrcT { typedef float R; };
template <> struct SrcT<SRC_E64> { typedef double R; };

// Eight consecutive values from `base`; past n: values of weight zero.
template <int SRC>
__device__ __forceinline__ void load8(const SlotArgs& a, uint64_t base, typename SrcT<SRC>::R* v) {
  typedef typename SrcT<SRC>::R R;
  const R* p = reinterpret_cast<const R*>(a.src) + base;
  if (base + 8 <= a.n && a.src_vec) {
    if constexpr (SRC == SRC_E64) {
      ld4(p, v);
      ld4(p + 4, v + 4);
    } else {
      ld8(p, v);
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = base + e < a.n ? p[e] : (SRC == SRC_LOG ? (R)-INFINITY : (R)0);
  }
}

// What quantisation is relative to: the maximum of l, or the power of two of
// the weights' maximum.
template <int SRC>
struct Quant {
  typedef typename SrcT<SRC>::R R;
  R m;
  int k, s;
  __device__ __forceinline__ Quant(const SlotArgs& a) : m(0), k(a.k), s(0) {
    if constexpr (SRC == SRC_LOG) m = dec_f((uint32_t)a.ctl->maxenc);
    if constexpr (SRC == SRC_W) {
      int e;
      (void)frexpf(__uint_as_float((uint32_t)a.ctl->maxenc), &e);
      s = a.k - e;
    }
  }
  // e in the place of eight sources l, two at a time
  __device__ __forceinline__ void exps(R* v) const {
    if constexpr (SRC == SRC_LOG) {
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const float2 x = exp_weight2(make_float2(v[e] - m, v[e + 1] - m));
        v[e] = x.x;
        v[e + 1] = x.y;
      }
    }
  }
  // W from e, or from a weight
  __device__ __forceinline__ uint64_t operator()(R v) const {
    if constexpr (SRC == SRC_W) return quant_weight(v, s);
    else return quant_from_e(v, k);
  }
};

// floor((hi 2^64 + lo) / d) for hi < d, d >= 2^63 (two 32-bit digits)
static __device__ __noinline__ uint64_t div_2by1(uint64_t hi, uint64_t lo, uint64_t d) {
  const uint64_t dh = d >> 32, dl = d & 0xffffffffull;
  uint64_t q[2];
  uint64_t r = hi;
  for (int i = 0; i < 2; ++i) {
    const uint64_t x = i == 0 ? lo >> 32 : lo & 0xffffffffull;
    uint64_t qh = r / dh, rh = r - qh * dh;  // digit estimate, at most two too large
    while (qh >= (1ull << 32) || qh * dl > ((rh << 32) | x)) {
      --qh;
      rh += dh;
      if (rh >= (1ull << 32)) break;
    }
    r = ((r << 32) | x) - qh * d;  // mod 2^64
    q[i] = qh;
  }
  return (q[0] << 32) | q[1];
}

// The slot map.  R(Q), the number of slot positions below n Q (systematic:
// j T + r; stratified: j T + r_j), from the fixed-point value X of n Q / T in
// units of 2^-32: X = Q' rho / 2^64 with Q' = Q 2^z and rho = n 2^(96 - z) / T
// rounded down, z the least shift that keeps rho below 2^64 (0 unless most of
// the mass is on few particles).  X, from three partial
// products, is low by less than 4.  Systematic: R = ceil((n Q - r) / T) and
// with r32 = floor(r 2^32 / T), Y = X - r32 is off by less than 4, so
// R = (Y >> 32) + 1 unless Y is within 4 of a whole number.  Stratified: with
// c = X >> 32, slot c is below n Q when r_c / T < frac(n Q / T); r_c / T is the
// leading 32 bits u of slot c's uniform to within a unit, so R = c + (frac > u)
// unless they are within 5.  The doubtful cases take the exact divisions of
// slot_below_exact: one in 2^29, and Q = 0 and Q = T, which the stratified map and
// the cut-point table meet in every call and which are told apart there (by
// divisions, with the thread's other values, they made a cycle of 8193 particles
// 2 to 4 us longer).  A high product per particle where a walk would carry a
// 64-bit remainder from one particle to the next and compare it with T, 2 T
// and 3 T.
// Stratified: the 32-bit uniforms of the slots a tile can reach come from a
// shared-memory table, half a Philox block per slot (slots past the table, in
// a tile of heavy particles, draw their own).
struct SlotMap {
  uint64_t rho, r32;
  const uint32_t* u;      // stratified: slots [u0, u0 + nu)
  uint32_t u0, nu;
  uint64_t seed;
  uint32_t filter, t;
};
static __device__ __noinline__ uint32_t strat_u32(uint32_t c, uint64_t seed, uint32_t filter, uint32_t t) {
  const U4 w = draw(seed, filter, t, c >> 1, P_STRATIFIED, 0);
  return (c & 1u) ? w.d : w.b;
}
// X of Q 2^z
__device__ __forceinline__ uint64_t slot_x(uint64_t q, uint64_t rho) {
  const uint32_t qh = (uint32_t)(q >> 32), ql = (uint32_t)q;
  const uint32_t rh = (uint32_t)(rho >> 32), rl = (uint32_t)rho;
  return (uint64_t)qh * rh + __umulhi(qh, rl) + __umulhi(ql, rh);
}
// R of Q 2^z; *close falls below 8 when R is doubtful
template <int POS>
__device__ __forceinline__ uint32_t slot_below(uint64_t q, const SlotMap& m, uint32_t* close) {
  const uint64_t X = slot_x(q, m.rho);
  if constexpr (POS == SLOTS_SYS) {
    const uint64_t Y = X - m.r32;
    *close = min(*close, (uint32_t)Y + 5u);
    return (uint32_t)(Y >> 32) + 1u;
  } else {
    const uint32_t c = (uint32_t)(X >> 32), f = (uint32_t)X;
    const uint32_t i = c - m.u0;
    // (a value as close to a whole number as Q = T is doubtful whatever u is)
    const uint32_t u = i < m.nu ? m.u[i] : f + 8u < 8u ? 0u : strat_u32(c, m.seed, m.filter, m.t);
    *close = min(*close, min(f + 8u, f - u + 5u));
    return c + (f > u ? 1u : 0u);
  }
}

// R of one of a thread's values when one or more of them are doubtful: the ends and
// the others without a division.
template <int POS>
static __device__ __noinline__ uint32_t slot_below_exact(uint64_t q, const Ctl* c, uint64_t n,
                                                         uint64_t seed, uint32_t filter, uint32_t t) {
  const uint64_t T = c->keyT;
  if (q == 0) return 0;
  if (q == T) return (uint32_t)n;
  SlotMap m;
  m.rho = c->slot_rho;
  m.r32 = c->slot_r32;
  m.u = nullptr;
  m.u0 = m.nu = 0;
  m.seed = seed;
  m.filter = filter;
  m.t = t;
  uint32_t close = ~0u;
  const uint32_t v = slot_below<POS>(q << c->slot_z, m, &close);
  if (close >= 8u) return v;
  const SysDiv dv = make_sysdiv(T);
  if (POS == SLOTS_SYS) return (uint32_t)sys_first_slot(q, n, c->keyR, dv);
  return (uint32_t)strat_first(q, n, T, dv, seed, filter, t);
}

// The last CTA of k_sums (out of line: its registers are not the others').
template <int SRC, bool ESS>
static __device__ __noinline__ void sums_last(const SlotArgs& a, uint64_t* s_tot,
                                              typename ESumT<typename SrcT<SRC>::R>::T* s_es, U128* s_sq) {
  typedef typename SrcT<SRC>::R R;
  typedef typename ESumT<R>::T ES;
  constexpr bool HAS_E = SRC != SRC_W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // exclusive prefixes of the tile sums, a contiguous run of
  // tiles per thread (up to 8 of them, N <= 2^22, kept in registers)
  constexpr uint32_t KEEP = 8;
  // (a multiple of four: the tiles' sums move four at a time, pre is padded)
  const uint32_t per = (((a.ntiles + BLOCK - 1) / BLOCK) + 3u) & ~3u;
  const uint32_t t0 = threadIdx.x * per < a.ntiles ? threadIdx.x * per : a.ntiles;
  const uint32_t t1 = t0 + per < a.ntiles ? t0 + per : a.ntiles;
  uint64_t mine = 0, kept[KEEP];
  // four sums from tile i (zero past the last)
  auto four = [&](uint32_t i, uint64_t* v) {
    v[0] = v[1] = v[2] = v[3] = 0;
    if (i < t1) ld4(a.pre + i, v);
#pragma unroll
    for (int q = 1; q < 4; ++q)
      if (i + q >= t1) v[q] = 0;
  };
#pragma unroll
  for (uint32_t i = 0; i < KEEP; i += 4) four(t0 + i, kept + i);
#pragma unroll
  for (uint32_t i = 0; i < KEEP; ++i) mine += kept[i];
#pragma unroll 4
  for (uint32_t i = t0 + KEEP; i < t1; i += 4) {
    uint64_t v[4];
    four(i, v);
    mine += (v[0] + v[1]) + (v[2] + v[3]);
  }
  const uint64_t incl = warp_incl_scan(mine, lane);
  if (lane == 31) s_tot[warp] = incl;
  ES es;
  es.zero();
  if constexpr (HAS_E && sizeof(R) == 4) {  // exact, so in any order
    const ES* const pb = reinterpret_cast<const ES*>(a.part_blk);
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < gridDim.x; i += BLOCK) {
      ES p;
      p.s.hi = __ldcg(&pb[i].s.hi);
      p.s.lo = __ldcg(&pb[i].s.lo);
      es.add(p);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) es.add(es.shfl_xor(o));
    if (lane == 0) s_es[warp] = es;
  }
  if constexpr (ESS) {
    U128 sq{0, 0};
    for (uint32_t i = threadIdx.x; i < gridDim.x; i += BLOCK) {
      U128 p;
      p.hi = __ldcg(&a.sq[i].hi);
      p.lo = __ldcg(&a.sq[i].lo);
      sq = add128(sq, p);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      U128 u;
      u.hi = __shfl_xor_sync(0xffffffffu, sq.hi, o);
      u.lo = __shfl_xor_sync(0xffffffffu, sq.lo, o);
      sq = add128(sq, u);
    }
    if (lane == 0) s_sq[warp] = sq;
  }
  __syncthreads();
  uint64_t run = incl - mine, T = 0;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) {
    if (w < warp) run += s_tot[w];
    T += s_tot[w];
  }
  // (a group's entries past the last tile are padding)
  bool heavy = false;
  const HeavyRule<SRC> rule(T, a.n);
  auto put4 = [&](uint32_t i, const uint64_t* v) {
#pragma unroll
    for (int q = 0; q < 4; ++q) heavy |= v[q] > rule.most;
    const uint64_t r1 = run + v[0], r2 = r1 + v[1], r3 = r2 + v[2];
    if (i < t1) st4(a.pre + i, run, r1, r2, r3);
    run = r3 + v[3];
  };
#pragma unroll
  for (uint32_t i = 0; i < KEEP; i += 4) put4(t0 + i, kept + i);
#pragma unroll 4
  for (uint32_t i = t0 + KEEP; i < t1; i += 4) {
    uint64_t v[4];
    four(i, v);
    put4(i, v);
  }
  // the constants, by one thread of each of four warps
  Ctl* const c = a.ctl;
  if (threadIdx.x == 0) {
    c->done_sums = 0;
    c->keyT = T;
    if (T == 0) atomicOr(&c->err, ERR_NUMERIC);
    if (SRC == SRC_W && a.host_err) *a.host_err = c->err | (c->maxenc == 0 ? ERR_WEIGHTS : 0u);
    if constexpr (HAS_E && sizeof(R) == 4) {
      es = s_es[0];
      for (int w = 1; w < WARPS; ++w) es.add(s_es[w]);
      reinterpret_cast<ES*>(a.part)[0] = es;
    }
  }
  if constexpr (ESS) {
    if (threadIdx.x == 32) {
      // ESS = T^2 / sum W^2 against ess_frac n (Kong, Liu & Wong 1994), as
      // A * A < (ess_frac * n) * B in binary64, A and B the exact sums each
      // rounded to nearest once
      U128 b = s_sq[0];
      for (int w = 1; w < WARPS; ++w) b = add128(b, s_sq[w]);
      const double A = __ull2double_rn(T);
      const double Bd = u128_to_f64_rn(b);
      const double lhs = A * A;
      const double f = a.ess_frac * (double)a.n;
      const double rhs = f * Bd;
      c->resamp = lhs < rhs ? 1u : 0u;
    }
  }
  if (T == 0) return;  // (the same in every thread)
  const int z = __clzll((long long)T);
  const uint64_t Tz = T << z;
  if (threadIdx.x == 64) {
    // rho = n 2^(96 + zs) / Tz with zs = z where that stays below 2^64 (the
    // quotient n 2^96 / Tz is below n 2^33): the shift of Q that is left is z - zs
    const int room = 31 - (64 - __clzll((long long)a.n));  // n 2^33 2^room <= 2^64
    const int zs = z < room ? z : room;
    c->slot_z = z - zs;
    c->slot_rho = div_2by1(a.n << (32 + zs), 0, Tz);
  }
  if (threadIdx.x == 96) {
    const uint32_t t = a.t_dev ? *a.t_dev : a.t_arg;
    const U4 wr = draw(a.seed, a.filter, t, 0, P_SYS_OFFSET, 0);
    const uint64_t r = a.cut ? 0ull : __umul64hi(((uint64_t)wr.b << 32) | wr.a, T);
    c->keyR = r;
    c->slot_r32 = div_2by1((r << z) >> 32, (r << z) << 32, Tz);
  }
  // multinomial: the constants of the slots' positions (k_multi).  With A = S_n,
  // P = floor((S 2^z) rho / 2^64), rho = floor(T 2^64 / (A 2^z)), A 2^z in
  // [2^63, 2^64); and the cut-point bucket n S / A in units of 2^-32 likewise
  if (a.multi && (threadIdx.x == 128 || threadIdx.x == 160)) {
    const uint64_t A = c->keyS;
    const int az = __clzll((long long)A);
    if (threadIdx.x == 128) {
      c->multi_z = az;
      c->multi_rho = div_2by1(T, 0, A << az);
    } else {
      c->bucket_rho = div_2by1(a.n << 32, 0, A << az);
    }
  }
  if (!a.heavy) return;
  const bool any = __syncthreads_or(heavy);  // (the prefixes and constants are written)
  if (!any) {
    if (threadIdx.x == 0) c->heavy_chunks = 0;
    return;
  }
  // The heavy list: the tiles whose further windows other CTAs store, in tile
  // order, with the number of their first chunk (a chunk is one such window).
  auto each = [&](auto f) {
    for (uint32_t i = t0; i < t1; ++i)
      if (const uint32_t k = rule((i + 1 < a.ntiles ? a.pre[i + 1] : T) - a.pre[i])) f(i, k);
  };
  uint64_t cnt = 0;  // entries, then chunks
  each([&](uint32_t, uint32_t k) { cnt += (1ull << 32) + k; });
  const uint64_t ci = warp_incl_scan(cnt, lane);
  if (lane == 31) s_tot[warp] = ci;
  __syncthreads();
  uint64_t at = ci - cnt, all = 0;
  for (int w = 0; w < WARPS; ++w) {
    if (w < warp) at += s_tot[w];
    all += s_tot[w];
  }
  each([&](uint32_t i, uint32_t k) {
    reinterpret_cast<uint2*>(a.heavy)[at >> 32] = make_uint2(i, (uint32_t)at);
    at += (1ull << 32) + k;
  });
  if (threadIdx.x == 0) {
    c->heavy_count = (uint32_t)(all >> 32);
    c->heavy_chunks = (uint32_t)all;
  }
}

template <int SRC, bool ESS>
__global__ void __launch_bounds__(BLOCK, 4) k_sums(SlotArgs a) {
  typedef typename SrcT<SRC>::R R;
  typedef typename ESumT<R>::T ES;
  constexpr bool HAS_E = SRC != SRC_W;
  __shared__ uint64_t s_tot[WARPS];
  __shared__ ES s_es[WARPS];
  __shared__ U128 s_sq[WARPS];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t base = (uint64_t)blockIdx.x * SUM_TILE + (uint64_t)threadIdx.x * SUM_PER;
  R v[SUM_PER];
  load8<SRC>(a, base, v);
  load8<SRC>(a, base + 8, v + 8);
  const Quant<SRC> quant(a);
  uint64_t tot = 0;
  U128 sq{0, 0};
  R ep = (R)0;  // sum of e over the thread's 16 particles, in order
#pragma unroll
  for (int h = 0; h < SUM_PER / 8; ++h) {
    R* const ex = v + 8 * h;
    quant.exps(ex);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint64_t w = quant(ex[e]);
      tot += w;
      if constexpr (HAS_E) ep = ep + ex[e];
      if constexpr (ESS) sq = add128(sq, mul64(w, w));
    }
    if constexpr (SRC == SRC_LOG) {
      if (a.e_out) {  // e in l's place: k_slots needs no exponential
        const uint64_t b = base + 8 * h;
        if (b + 8 <= a.n) {
          st8(a.e_out + b, ex);
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (b + e < a.n) a.e_out[b + e] = ex[e];
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if (lane == 0) s_tot[warp] = tot;
  if constexpr (HAS_E) {
    ES es;
    es.zero();
    es.add(ep);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) es.add(es.shfl_xor(o));
    if (lane == 0) s_es[warp] = es;
  }
  if constexpr (ESS) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      U128 u;
      u.hi = __shfl_xor_sync(0xffffffffu, sq.hi, o);
      u.lo = __shfl_xor_sync(0xffffffffu, sq.lo, o);
      sq = add128(sq, u);
    }
    if (lane == 0) s_sq[warp] = sq;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int h = 0; h < SUM_SUB; ++h) {
      uint64_t s = 0;
      for (int w = 0; w < WARPS / SUM_SUB; ++w) s += s_tot[h * (WARPS / SUM_SUB) + w];
      const uint32_t tile = blockIdx.x * SUM_SUB + h;
      if (tile < a.ntiles) a.pre[tile] = s;
    }
    if constexpr (HAS_E) {
      ES es = s_es[0];
      for (int w = 1; w < WARPS; ++w) es.add(s_es[w]);
      reinterpret_cast<ES*>(a.part_blk)[blockIdx.x] = es;
    }
    if constexpr (ESS) {
      U128 b = s_sq[0];
      for (int w = 1; w < WARPS; ++w) b = add128(b, s_sq[w]);
      a.sq[blockIdx.x] = b;
    }
    __threadfence();
    s_last = atomicAdd(&a.ctl->done_sums, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  sums_last<SRC, ESS>(a, s_tot, s_es, s_sq);
}

// Rare part of marking: the group starts [from, to) of a particle of more than
// five slots in the window, as a run of the whole CTA when long.
constexpr uint32_t RUN_MIN = 64;  // slots of a run
static __device__ __noinline__ void mark_rest(uint32_t from, uint32_t to, uint16_t mk, uint16_t* win,
                                              uint32_t (*runs)[3], uint32_t* nruns) {
  if (to - from > RUN_MIN) {
    const uint32_t kr = atomicAdd(nruns, 1u);
    if (kr < SLOT_RUNS) {
      runs[kr][0] = from;
      runs[kr][1] = to;
      runs[kr][2] = mk;
      return;
    }
  }
  for (uint32_t q = from; q < to; q += 4u) win[win_entry(q)] = mk;
}

// The slots [j, Rs[0]), [Rs[0], Rs[1]), ... of a thread's particles marked in the
// window of WIN slots from wb; mk0: the first particle's mark.  When the window
// holds them all and none has more than five (for a whole warp):
__device__ __forceinline__ void win_mark(uint16_t* win, uint32_t wb, uint32_t j, const uint32_t* Rs, uint32_t mk0) {
  uint32_t x = j - wb;
#pragma unroll
  for (int e = 0; e < SLOT_PER; ++e) {
    const uint32_t xe = Rs[e] - wb, g = (x + 4u) & ~3u;
    if (xe > x) win[win_entry(x)] = (uint16_t)(mk0 + e);
    if (xe > g) win[win_entry(g)] = (uint16_t)(mk0 + e);
    x = xe;
  }
}
// else each particle's slots clipped to the window
template <uint32_t WIN>
__device__ __forceinline__ void win_mark_clipped(uint16_t* win, uint32_t (*runs)[3], uint32_t* nruns, uint32_t wb,
                                                 uint32_t j, const uint32_t* Rs, uint32_t mk0) {
  uint32_t x = j < wb ? 0u : min(j - wb, WIN);
#pragma unroll
  for (int e = 0; e < SLOT_PER; ++e) {
    const uint32_t xe = Rs[e] < wb ? 0u : min(Rs[e] - wb, WIN), g = (x + 4u) & ~3u;
    const uint16_t mk = (uint16_t)(mk0 + e);
    if (xe > x) win[win_entry(x)] = mk;
    if (xe > g) win[win_entry(g)] = mk;
    if (xe > g + 4u) mark_rest(g + 4u, xe, mk, win, runs, nruns);
    x = xe;
  }
}
// the runs that marking left, by the whole CTA of NT threads (after a barrier)
template <int NT>
__device__ __forceinline__ void win_runs(uint16_t* win, const uint32_t (*runs)[3], const uint32_t* nruns) {
  const uint32_t nr = *nruns < SLOT_RUNS ? *nruns : SLOT_RUNS;
  if (!nr) return;
  for (uint32_t q = 0; q < nr; ++q) {
    const uint32_t en = runs[q][1];
    for (uint32_t y = runs[q][0] + 4u * threadIdx.x; y < en; y += 4u * NT) win[win_entry(y)] = (uint16_t)runs[q][2];
  }
  __syncthreads();
}
// the window's slots [ws, wend), four per 16-byte store where vec (the partial
// groups at either end slot by slot); tb: the tile's first particle
template <int NT>
__device__ __forceinline__ void win_store(const uint16_t* win, uint32_t* anc, uint32_t wb, uint32_t ws, uint32_t wend,
                                          uint32_t tb, bool vec) {
  const uint32_t tb32 = tb - 1u;
  const uint32_t ng = wend > ws ? (wend - wb + 3u) >> 2 : 0u;
  for (uint32_t g = threadIdx.x; g < ng; g += NT) {
    const uint32_t x0 = g << 2;
    const uint32_t sw = ((x0 >> 6) & 7u) << 1;
    const uint2 w = *reinterpret_cast<const uint2*>(win + (x0 ^ (sw & 12u)));
    const uint32_t lo = (sw & 2u) ? w.y : w.x, hi = (sw & 2u) ? w.x : w.y;
    const uint32_t slot = wb + x0;
    const uint32_t e0 = lo & 0xffffu, e1 = max(e0, lo >> 16);
    const uint32_t e2 = max(e1, hi & 0xffffu), e3 = max(e2, hi >> 16);
    const uint4 o4 = make_uint4(tb32 + e0, tb32 + e1, tb32 + e2, tb32 + e3);
    if (slot >= ws && slot + 4u <= wend && vec) {
      *reinterpret_cast<uint4*>(anc + slot) = o4;
    } else {
      if (slot >= ws && slot < wend) anc[slot] = o4.x;
      if (slot + 1u >= ws && slot + 1u < wend) anc[slot + 1u] = o4.y;
      if (slot + 2u >= ws && slot + 2u < wend) anc[slot + 2u] = o4.z;
      if (slot + 3u >= ws && slot + 3u < wend) anc[slot + 3u] = o4.w;
    }
  }
}

// Binary64: an exponential of a heavy tile, taken again from l by another CTA than
// the tile's, which may have written Q over k_exp's values already.
static __device__ __noinline__ double heavy_exp64(const SlotArgs& a, uint64_t i) {
  return i < a.n ? exp_weight(a.l[i] - dec_d(a.ctl->maxenc)) : 0.0;
}

// One CTA per tile.  Thread t takes particles [8 t, 8 t + 8) of the tile.  The
// ancestors of the tile's slots are built in a shared-memory window of one
// 16-bit entry per slot (at least two slots per particle of the tile), cleared
// first: a particle marks (its offset in the tile + 1) its first slot and every
// multiple of four among its others, so that each aligned group of four slots
// starts with a mark and a thread completes its group by a running maximum
// and stores it as 16 bytes.  Two predicated stores cover a particle of up to
// five slots, whatever its neighbours own; writing every slot took a divergent
// path per heavy particle (k_slots at N = 2^24 on weights of log-spread 1:
// 112 -> 64 us).
//
// A tile of more slots than its window (binary64: than seven) holds leaves the
// others to the CTAs of the heavy list (k_sums): CTA b < heavy_chunks, after its
// own tile, rebuilds the heavy tile of chunk b and stores that window.  With all
// the mass on one particle of 2^23 the kernel takes 43 us (binary64 55), by one
// CTA window after window 2.5 ms.  Binary64 overwrites its source with Q, so there
// the heavy tile is rebuilt from l.
template <int SRC, int POS>
__global__ void __launch_bounds__(BLOCK, 4) k_slots(SlotArgs a) {
  typedef typename SrcT<SRC>::R R;
  constexpr int P = POS == SLOTS_NONE ? SLOTS_SYS : POS;
  __shared__ uint64_t s_warp[WARPS];
  __shared__ uint32_t s_run[SLOT_RUNS][3];
  __shared__ uint32_t s_nruns, s_end;
  __shared__ alignas(16) uint16_t s_win[SLOT_WIN];
  __shared__ alignas(8) uint32_t s_u[POS == SLOTS_STRAT ? SLOT_WIN : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t n = a.n;
  const Ctl* const c = a.ctl;
  const Quant<SRC> quant(a);
  uint32_t tile = blockIdx.x, wsel = 0;
  for (int pass = 0;; ++pass) {
    const uint64_t tbase = (uint64_t)tile * SLOT_TILE;
    const uint64_t base = tbase + (uint64_t)threadIdx.x * SLOT_PER;
    R v[SLOT_PER];
    if constexpr (SRC == SRC_E64) {
      if (pass == 0) {
        load8<SRC>(a, base, v);
      } else {
#pragma unroll
        for (int e = 0; e < SLOT_PER; ++e) v[e] = heavy_exp64(a, base + e);
      }
    } else {
      load8<SRC>(a, base, v);
    }
    uint64_t run[SLOT_PER];
    uint64_t acc = 0;
    quant.exps(v);
#pragma unroll
    for (int e = 0; e < SLOT_PER; ++e) {
      acc += quant(v[e]);
      run[e] = acc;
    }
    const uint64_t incl = warp_incl_scan(acc, lane);
    if (lane == 31) s_warp[warp] = incl;
    auto clear = [&]() {
      if (threadIdx.x == 0) s_nruns = 0;
#pragma unroll
      for (uint32_t i = 0; i < SLOT_WIN; i += 8 * BLOCK)
        *reinterpret_cast<uint4*>(s_win + i + 8 * threadIdx.x) = make_uint4(0u, 0u, 0u, 0u);
    };
    if constexpr (POS != SLOTS_NONE) clear();
    const uint64_t pre = a.pre[tile];
    __syncthreads();
    uint64_t woff = (lane & 7) < warp ? s_warp[lane & 7] : 0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) woff += __shfl_xor_sync(0xffffffffu, woff, o);
    uint64_t q0 = pre + woff + incl - acc;  // Q just before this thread's particles
    if (a.Q && pass == 0) {
      if (base + SLOT_PER <= n) {
        st4(a.Q + base, q0 + run[0], q0 + run[1], q0 + run[2], q0 + run[3]);
        st4(a.Q + base + 4, q0 + run[4], q0 + run[5], q0 + run[6], q0 + run[7]);
      } else {
#pragma unroll
        for (int e = 0; e < SLOT_PER; ++e)
          if (base + e < n) a.Q[base + e] = q0 + run[e];
      }
    }
    if constexpr (POS == SLOTS_NONE) return;
    if (a.gate && *a.gate == 0u) return;
    if (c->keyT == 0) {  // empty CDF (flagged): keep every index in range
#pragma unroll
      for (int e = 0; e < SLOT_PER; ++e)
        if (base + e < n) a.anc[base + e] = (uint32_t)(base + e);
      return;
    }
    SlotMap m;
    m.rho = c->slot_rho;
    m.r32 = c->slot_r32;
    m.seed = a.seed;
    m.filter = a.filter;
    m.t = a.t_dev ? *a.t_dev : a.t_arg;
    const int z = c->slot_z;
    uint64_t p0 = pre;
    if (z) {  // (the same in every thread; rare)
      p0 <<= z;
      q0 <<= z;
#pragma unroll
      for (int e = 0; e < SLOT_PER; ++e) run[e] <<= z;
    }
    if constexpr (POS == SLOTS_STRAT) {
      uint64_t tot = s_warp[lane & 7];
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      m.u = s_u;
      m.u0 = (uint32_t)(slot_x(p0, m.rho) >> 32) & ~1u;
      const uint32_t last = (uint32_t)(slot_x(p0 + (tot << z), m.rho) >> 32);
      m.nu = min(((last - m.u0) | 1u) + 1u, SLOT_WIN);
      for (uint32_t i = 2u * threadIdx.x; i < m.nu; i += 2u * BLOCK) {
        const U4 w = draw(m.seed, m.filter, m.t, (m.u0 + i) >> 1, P_STRATIFIED, 0);
        *reinterpret_cast<uint2*>(s_u + i) = make_uint2(w.b, w.d);
      }
      __syncthreads();
    }
    uint32_t close = ~0u, close0 = ~0u;
    uint32_t S0 = slot_below<P>(p0, m, &close0);  // the tile's first slot
    if (close0 < 8u) S0 = slot_below_exact<P>(pre, c, n, m.seed, m.filter, m.t);
    uint32_t Rs[SLOT_PER];
    uint32_t j = slot_below<P>(q0, m, &close);
#pragma unroll
    for (int e = 0; e < SLOT_PER; ++e) Rs[e] = slot_below<P>(q0 + run[e], m, &close);
    if (close < 8u) {
      j = slot_below_exact<P>(q0 >> z, c, n, m.seed, m.filter, m.t);
      for (int e = 0; e < SLOT_PER; ++e)
        Rs[e] = slot_below_exact<P>((q0 + run[e]) >> z, c, n, m.seed, m.filter, m.t);
    }
    if (threadIdx.x == BLOCK - 1) s_end = Rs[SLOT_PER - 1];
    const uint32_t mk0 = threadIdx.x * SLOT_PER + 1u;
    uint32_t most = Rs[0] - j;
#pragma unroll
    for (int e = 1; e < SLOT_PER; ++e) most = max(most, Rs[e] - Rs[e - 1]);
    // the window's base: slots in aligned groups of four
    uint32_t wb = (S0 & ~3u) + wsel * SLOT_WIN;
    while (true) {
      if (!__any_sync(0xffffffffu, most > 5u || j < wb || Rs[SLOT_PER - 1] - wb > SLOT_WIN))
        win_mark(s_win, wb, j, Rs, mk0);
      else
        win_mark_clipped<SLOT_WIN>(s_win, s_run, &s_nruns, wb, j, Rs, mk0);
      __syncthreads();
      win_runs<BLOCK>(s_win, s_run, &s_nruns);
      win_store<BLOCK>(s_win, a.anc, wb, max(S0, wb), min(s_end, wb + SLOT_WIN), (uint32_t)tbase, a.anc_vec);
      wb += SLOT_WIN;
      if (HeavyRule<SRC>::OWN == 0 || pass == 1 || s_end <= wb) break;
      const uint64_t next = tile + 1 < a.ntiles ? a.pre[tile + 1] : c->keyT;
      if (HeavyRule<SRC>(c->keyT, n)(next - pre)) break;
      __syncthreads();  // the window has been read
      clear();
      __syncthreads();
    }
    if (pass == 1 || blockIdx.x >= c->heavy_chunks) return;
    // the heavy tile of chunk blockIdx.x: the last entry whose first chunk is
    // not above it
    const uint2* const list = reinterpret_cast<const uint2*>(a.heavy);
    uint32_t lo = 0, hi = c->heavy_count - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (list[mid].y <= blockIdx.x) lo = mid;
      else hi = mid - 1;
    }
    tile = list[lo].x;
    wsel = 1 + blockIdx.x - list[lo].y;
    __syncthreads();  // shared memory has been read
  }
}

}  // namespace pfk
