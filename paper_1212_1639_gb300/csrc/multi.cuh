// Multinomial resampling (Section 3.1) against a finished CDF, from sorted
// uniforms U_(j) = S_j / S_n with S the running sum of exponential spacings
// E_l = floor(-log(u_l) 2^31) (Carpenter, Clifford & Fearnhead 1999; u_l from
// draw (seed, filter, t, l >> 2, SPACING) word l & 3):
//   k_spacing_sums  the sums of 2048 spacings each, their prefixes, S_n;
//   k_multi_split   per tile of 2048 slots, the particles below its start;
//   k_multi         per tile: its spacings again, their scan, and each slot's
//                   ancestor a_j = #{i : Q_i S_n <= S_j T}.
// The spacings are drawn twice (a quarter Philox block and a logarithm per
// slot) instead of stored once and read once as 64-bit prefixes: 55 instructions
// against 16 bytes.  A slot's position is brought to the CDF's scale once,
// P_j = S_j T / S_n, so that the search compares 64-bit words: the merge it
// replaces formed and compared 128-bit keys for every particle and slot
// (N = 2^24: k_partition 51 and k_merge 201 us, spacing scan 109 beside the
// weights and the CDF).
#pragma once
#include "device.cuh"
#include "slots.cuh"

namespace pfk {

constexpr int MULTI_PER = 8;                     // slots per thread
constexpr int MULTI_TILE = BLOCK * MULTI_PER;    // 2048: k_slots' tile too
constexpr uint32_t MULTI_CAP = 4096;             // particles of a tile staged in shared memory
static_assert(MULTI_TILE == SLOT_TILE, "the CDF's tile prefixes serve the split search");

struct MultiArgs {
  const uint64_t* Q;
  const uint64_t* pre;     // per CDF tile: its exclusive prefix (k_sums)
  uint64_t* spre;          // per slot tile: its sum, then its exclusive prefix
  uint32_t* splits;        // per slot tile (and one more): particles below its start
  uint32_t* anc;
  const uint32_t* I;       // cut-point table (k_multi<true>)
  Ctl* ctl;
  const uint32_t* t_dev;
  uint32_t t_arg;
  uint32_t ntiles;
  uint64_t n;
  uint64_t seed;
  uint32_t filter;
  const uint32_t* gate;    // *gate == 0: this cycle does not resample (NULL: it does)
  int anc_vec;             // anc is 32-byte aligned
};

// The 8 spacings from slot l0 (a multiple of 8), as running sums; slots past n
// add nothing.
__device__ __forceinline__ void spacings8(const MultiArgs& a, uint32_t t, uint64_t l0, uint64_t* run) {
  uint64_t acc = 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const U4 w = draw(a.seed, a.filter, t, (uint32_t)(l0 >> 2) + h, P_SPACING, 0);
    const float2 L0 = det_log2(unif_f32_2(w.a, w.b)), L1 = det_log2(unif_f32_2(w.c, w.d));
    const float L[4] = {L0.x, L0.y, L1.x, L1.y};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      // floor(-L 2^31) from L's bits: |L| in [2^-24, 17), so a right shift of
      // the significand from 12 above
      const uint32_t b = __float_as_uint(L[e]) & 0x7fffffffu;
      const uint64_t E = ((uint64_t)((b & 0x7fffffu) | 0x800000u) << 12) >> (131 - (int)(b >> 23));
      acc += l0 + 4 * h + e < a.n ? E : 0ull;
      run[4 * h + e] = acc;
    }
  }
}

static __global__ void __launch_bounds__(BLOCK, 4) k_spacing_sums(MultiArgs a) {
  __shared__ uint64_t s_tot[WARPS];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t t = a.t_dev ? *a.t_dev : a.t_arg;
  uint64_t run[MULTI_PER];
  spacings8(a, t, (uint64_t)blockIdx.x * MULTI_TILE + threadIdx.x * MULTI_PER, run);
  uint64_t tot = run[MULTI_PER - 1];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if (lane == 0) s_tot[warp] = tot;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t s = 0;
    for (int w = 0; w < WARPS; ++w) s += s_tot[w];
    a.spre[blockIdx.x] = s;
    __threadfence();
    s_last = atomicAdd(&a.ctl->done_spc, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the last CTA: exclusive prefixes, four tiles at a time (spre is padded)
  const uint32_t per = (((a.ntiles + BLOCK - 1) / BLOCK) + 3u) & ~3u;
  const uint32_t t0 = threadIdx.x * per < a.ntiles ? threadIdx.x * per : a.ntiles;
  const uint32_t t1 = t0 + per < a.ntiles ? t0 + per : a.ntiles;
  auto four = [&](uint32_t i, uint64_t* v) {
    v[0] = v[1] = v[2] = v[3] = 0;
    if (i < t1) ld4(a.spre + i, v);
#pragma unroll
    for (int q = 1; q < 4; ++q)
      if (i + q >= t1) v[q] = 0;
  };
  uint64_t mine = 0;
#pragma unroll 4
  for (uint32_t i = t0; i < t1; i += 4) {
    uint64_t v[4];
    four(i, v);
    mine += (v[0] + v[1]) + (v[2] + v[3]);
  }
  const uint64_t incl = warp_incl_scan(mine, lane);
  if (lane == 31) s_tot[warp] = incl;
  __syncthreads();
  uint64_t at = incl - mine, all = 0;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) {
    if (w < warp) at += s_tot[w];
    all += s_tot[w];
  }
#pragma unroll 4
  for (uint32_t i = t0; i < t1; i += 4) {
    uint64_t v[4];
    four(i, v);
    st4(a.spre + i, at, at + v[0], at + v[0] + v[1], at + v[0] + v[1] + v[2]);
    at += (v[0] + v[1]) + (v[2] + v[3]);
  }
  if (threadIdx.x == 0) {  // S_n = S_{n-1} + E_n
    const U4 w = draw(a.seed, a.filter, t, (uint32_t)(a.n >> 2), P_SPACING, 0);
    a.ctl->keyS = all + spacing_E(a.seed, a.filter, t, a.n, w);
    a.ctl->done_spc = 0;
  }
}

// The largest i in [lo, hi] with i == lo or below(i), for below() true then
// false in i, by a warp-wide 32-ary search.
template <class F>
__device__ __forceinline__ uint64_t warp_last(uint64_t lo, uint64_t hi, F below) {
  const int lane = threadIdx.x & 31;
  while (hi > lo) {
    const uint64_t span = hi - lo;
    const uint64_t q = lo + 1 + (span * (uint64_t)lane) / 32;
    const uint32_t m = __ballot_sync(0xffffffffu, below(q));
    if (m == 0) {
      hi = lo;
    } else {
      const int kstar = 31 - __clz(m);
      const uint64_t qk = __shfl_sync(0xffffffffu, q, kstar);
      const uint64_t qn = __shfl_sync(0xffffffffu, q, kstar < 31 ? kstar + 1 : 31);
      lo = qk;
      if (kstar < 31) hi = qn - 1;
    }
  }
  return lo;
}

// #{i : Q_i S_n <= S T} for S the spacings before slot tile s, by one warp: the
// CDF tile by its prefix, then the particle in the tile.  Past the last tile: the
// first particle whose CDF value is T (no ancestor lies beyond it).
__device__ __forceinline__ uint32_t multi_split(const MultiArgs& a, uint32_t s, uint64_t T, uint64_t A) {
  const bool end = s == a.ntiles;
  const U128 key = mul64(end ? T - 1 : a.spre[s], end ? 1ull : T);
  const uint64_t f = end ? 1ull : A;
  const uint64_t tile = warp_last(0, a.ntiles - 1, [&](uint64_t i) { return le128(mul64(a.pre[i], f), key); });
  const uint64_t b = tile * SLOT_TILE, e = b + SLOT_TILE < a.n ? b + SLOT_TILE : a.n;
  return (uint32_t)warp_last(b, e, [&](uint64_t q) { return le128(mul64(a.Q[q - 1], f), key); });
}
// splits[s] of every tile and of the end, one warp each.
static __global__ void __launch_bounds__(BLOCK) k_multi_split(MultiArgs a) {
  if (a.gate && *a.gate == 0u) return;
  const uint64_t T = a.ctl->keyT, A = a.ctl->keyS;
  if (T == 0) return;  // empty CDF (flagged)
  const uint32_t s = blockIdx.x * WARPS + (threadIdx.x >> 5);
  if (s > a.ntiles) return;
  const uint32_t i = multi_split(a, s, T, A);
  if ((threadIdx.x & 31) == 0) a.splits[s] = i;
}
// Up to this many slot tiles two warps of each tile's CTA search for its splits
// themselves, beside the other warps' spacings, and k_multi_split is not launched.
// Cycle in us, launched / own: N = 16,384 37.0 / 34.9, 2^18 40.8 / 39.0, 2^20 61.0 /
// 56.8, 2^21 92.8 / 91.6, 2^22 151.6 / 153.8, 2^24 521 / 542.
constexpr uint32_t MULTI_OWN = 1024;

// The exact ancestor of a slot at S, not before particle i.
static __device__ __noinline__ uint32_t multi_exact(const uint64_t* Q, uint64_t n, uint64_t S, uint64_t T,
                                                    uint64_t A, uint32_t i) {
  const U128 key = mul64(S, T);
  while (i < n && le128(mul64(Q[i], A), key)) ++i;
  return i;
}

// One CTA per tile of 2048 slots, thread t slots [8 t, 8 t + 8).  The tile's
// ancestors are in [splits[s], splits[s + 1]]; that part of the CDF is staged in
// shared memory when it has at most MULTI_CAP particles, else searched in global
// memory.  A thread finds its first slot's ancestor by bisection and steps on
// from slot to slot, bisecting again past 16 particles.  P is low by less than
// 4, so an ancestor whose next CDF value is within that of P takes the exact
// comparison.  CUT: the paper's Section 3.2 method instead -- start at the
// cut-point table's entry of the slot's bucket and climb.
// OWN: the CTA's first two warps search for its splits (MULTI_OWN).
template <bool CUT, bool OWN = false>
__global__ void __launch_bounds__(BLOCK, 4) k_multi(MultiArgs a) {
  __shared__ uint64_t s_q[CUT ? 1 : MULTI_CAP + 1];
  __shared__ uint64_t s_warp[WARPS];
  __shared__ uint32_t s_split[OWN ? 2 : 1];
  if (a.gate && *a.gate == 0u) return;
  const Ctl* const c = a.ctl;
  const uint64_t n = a.n, T = c->keyT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t j0 = (uint64_t)blockIdx.x * MULTI_TILE + threadIdx.x * MULTI_PER;
  if (T == 0) {  // empty CDF (flagged): keep every index in range
    for (int e = 0; e < MULTI_PER; ++e)
      if (j0 + e < n) a.anc[j0 + e] = (uint32_t)(j0 + e);
    return;
  }
  const uint32_t t = a.t_dev ? *a.t_dev : a.t_arg;
  const uint64_t A = c->keyS, rho = c->multi_rho;
  const int z = c->multi_z;
  uint32_t i0 = 0, i1 = 0;
  bool staged = false;
  auto stage = [&]() {
    staged = i1 - i0 <= MULTI_CAP;
    if (staged)
      for (uint32_t i = threadIdx.x; i < i1 - i0; i += BLOCK) s_q[i] = a.Q[i0 + i];
    if (threadIdx.x == 0) s_q[staged ? i1 - i0 : 0] = ~0ull;
  };
  if constexpr (!CUT) {
    if constexpr (!OWN) {
      i0 = a.splits[blockIdx.x];
      i1 = a.splits[blockIdx.x + 1];
      stage();
    } else if (warp < 2) {
      const uint32_t v = multi_split(a, blockIdx.x + warp, T, A);
      if (lane == 0) s_split[warp] = v;
    }
  }
  uint64_t run[MULTI_PER];
  spacings8(a, t, j0, run);
  const uint64_t incl = warp_incl_scan(run[MULTI_PER - 1], lane);
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if constexpr (OWN) {
    i0 = s_split[0];
    i1 = s_split[1];
    stage();
    __syncthreads();
  }
  uint64_t off = (lane & 7) < warp ? s_warp[lane & 7] : 0;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) off += __shfl_xor_sync(0xffffffffu, off, o);
  const uint64_t S0 = a.spre[blockIdx.x] + off + incl - run[MULTI_PER - 1];
  uint32_t out[MULTI_PER];
  auto keep = [&](int e, uint64_t P, uint64_t nextq, uint32_t an) {  // nextq: the first CDF value above P
    if (nextq - P < 5ull) an = multi_exact(a.Q, n, S0 + run[e], T, A, an);
    out[e] = an < n ? an : (uint32_t)(n - 1);
  };
  if constexpr (CUT) {
    // four slots' table entries, then their CDF values, then their climbs step by
    // step together, so that the loads of four are in flight at once (one slot
    // after the other a cycle of 8193 particles was 10 us longer)
    const uint64_t brho = c->bucket_rho;
#pragma unroll
    for (int h = 0; h < MULTI_PER; h += 4) {
      uint64_t P[4], nextq[4];
      uint32_t i[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        // bucket floor(n S / A): X is low by less than 4 units of 2^-32, and a
        // bucket one too low only starts the climb earlier
        const uint64_t S = (S0 + run[h + e]) << z;
        P[e] = slot_x(S, rho);
        const uint32_t b = (uint32_t)(slot_x(S, brho) >> 32);
        i[e] = a.I[b < n ? b : n - 1];
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) nextq[e] = a.Q[i[e]];
      bool more = true;
      while (more) {
        more = false;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (nextq[e] <= P[e] && i[e] + 1 < n) {
            nextq[e] = a.Q[++i[e]];
            more = true;
          }
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j0 + h + e < n) keep(h + e, P[e], nextq[e], i[e]);
    }
  } else if (staged) {
    uint32_t i = 0;
    const uint32_t cnt = i1 - i0;
    auto bisect = [&](uint64_t P) {
      uint32_t hi = cnt;
      while (i < hi) {
        const uint32_t mid = (i + hi) >> 1;
        if (s_q[mid] <= P) i = mid + 1;
        else hi = mid;
      }
    };
#pragma unroll
    for (int e = 0; e < MULTI_PER; ++e) {
      const uint64_t P = slot_x((S0 + run[e]) << z, rho);
      if (j0 + e < n) {
        if (e == 0) {
          bisect(P);
        } else {
          uint32_t steps = 0;
          while (steps < 16u && s_q[i] <= P) {
            ++i;
            ++steps;
          }
          if (steps == 16u) bisect(P);
        }
        keep(e, P, s_q[i], i0 + i);
      }
    }
  } else {
    // in global memory: the eight bisections step by step together, so that
    // their loads are in flight at once
    uint64_t P[MULTI_PER];
    uint32_t lo[MULTI_PER], hi[MULTI_PER];
#pragma unroll
    for (int e = 0; e < MULTI_PER; ++e) {
      P[e] = slot_x((S0 + run[e]) << z, rho);
      lo[e] = i0;
      hi[e] = i1;
    }
    for (uint32_t w = i1 - i0; w; w >>= 1) {  // (a range of w halves to at most w / 2)
#pragma unroll
      for (int e = 0; e < MULTI_PER; ++e) {
        if (lo[e] < hi[e]) {
          const uint32_t mid = (lo[e] + hi[e]) >> 1;
          if (a.Q[mid] <= P[e]) lo[e] = mid + 1;
          else hi[e] = mid;
        }
      }
    }
#pragma unroll
    for (int e = 0; e < MULTI_PER; ++e)
      if (j0 + e < n) keep(e, P[e], a.Q[lo[e]], lo[e]);
  }
  if (j0 + MULTI_PER <= n && a.anc_vec) {
    float v[MULTI_PER];
#pragma unroll
    for (int e = 0; e < MULTI_PER; ++e) v[e] = __uint_as_float(out[e]);
    st8(reinterpret_cast<float*>(a.anc + j0), v);
  } else {
#pragma unroll
    for (int e = 0; e < MULTI_PER; ++e)
      if (j0 + e < n) a.anc[j0 + e] = out[e];
  }
}

}  // namespace pfk
