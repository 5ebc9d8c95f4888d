// Whole cycles of a small filter in one launch: one thread-block cluster holds
// the filter, CTA r of G the particles and slots [r m, (r + 1) m), and goes
// through Steps 1-4 with cluster barriers, several observations per launch.
//
// A filter of a few thousand particles is bound by latency: the general cycle's
// four to eight launches cost 23-30 us (binary32) and 35-41 us (binary64) at
// N = 1024 whatever the arithmetic.  Here a cycle is four cluster barriers, two
// trips to L2 (the state, the ancestor's record) and a search in distributed
// shared memory.  Microseconds per cycle of a block of observations, general /
// here: binary32 systematic 23 / 9.8 at N = 1024, 25 / 17.9 at 8192; binary32
// multinomial 30 / 10.7 and 35 / 19.3; binary64 multinomial 41 / 18.2 at 1024,
// 44 / 34.7 at 4096 (8192: 60, so binary64 stops at 4096: eight SMs' binary64
// pipes against 152).
//
// Every value is the general path's: the same operations per particle, and the
// log-ML and summary sums over the same groups in the same order.
#pragma once
#include "kernels.cuh"

namespace pfk {

constexpr int SMALL_M = 1024;          // particles per CTA, at most
constexpr int SMALL_K = SMALL_M / BLOCK;
constexpr uint32_t SMALL_Y = 64;       // observations of one launch
constexpr uint32_t SMALL_GMAX = 8;     // CTAs per cluster (the portable size)

enum SmallPos : int { SP_SYS = 0, SP_STRAT = 1, SP_MULTI = 2 };

struct SmallArgs {
  int pos;                 // SmallPos (the cut-point schemes give the same ancestors)
  int learn, ess, boot;    // boot: Algorithm "Particle Filtering"
  int est;                 // the summaries after the last cycle
  uint32_t m;              // particles per CTA, a multiple of 32
  uint32_t steps;
  double ess_frac;
  const double* y_dev;     // device-resident observations, or NULL
  double y[SMALL_Y];       // else observations by value
};

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_nctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t dsm_addr(const void* p, uint32_t rank) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ uint64_t dsm_u64(uint32_t addr) {
  uint64_t v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t dsm_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float dsm_real(const float* p, uint32_t rank) {
  return __uint_as_float(dsm_u32(dsm_addr(p, rank)));
}
__device__ __forceinline__ double dsm_real(const double* p, uint32_t rank) {
  return from_bits(dsm_u64(dsm_addr(p, rank)));
}

// Block exclusive scan of one 64-bit value per thread; *total in every thread.
// Two barriers; s is read until the next barrier of the block.
__device__ __forceinline__ uint64_t small_scan(uint64_t v, uint64_t* s, uint64_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t incl = warp_incl_scan(v, lane);
  if (lane == 31) s[warp] = incl;
  __syncthreads();
  uint64_t off = (lane & 7) < warp ? s[lane & 7] : 0, all = s[lane & 7];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    off += __shfl_xor_sync(0xffffffffu, off, o);
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  *total = all;
  return off + incl - v;
}

// The number of particles whose key Q A is not above each of K slots' keys,
// for Q in the cluster's distributed shared memory (m per CTA, q): first over
// the CTAs by their last values cum, then by bisection in that CTA's part.  The
// K bisections go step by step together, so that their loads overlap.
template <int K, class F>
__device__ __forceinline__ void cluster_search(const uint64_t* q, const uint64_t* cum, uint32_t G,
                                               uint32_t m, uint32_t n, const U128* kb, F above,
                                               uint32_t* out) {
  uint32_t at[K], lo[K], hi[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    lo[k] = 0;
    hi[k] = G - 1;
  }
  for (uint32_t w = G - 1; w; w >>= 1) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t mid = (lo[k] + hi[k]) >> 1;
      const bool up = lo[k] < hi[k], ab = above(cum[mid], kb[k]);
      if (up && ab) hi[k] = mid;
      if (up && !ab) lo[k] = mid + 1;
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t rr = lo[k], b = rr * m;
    at[k] = dsm_addr(q, rr);
    out[k] = b;
    lo[k] = 0;
    hi[k] = b < n ? (b + m < n ? m : n - b) : 0u;
  }
  for (uint32_t w = m; w; w >>= 1) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t mid = (lo[k] + hi[k]) >> 1;
      const bool up = lo[k] < hi[k];
      const bool ab = up && above(dsm_u64(at[k] + 8 * mid), kb[k]);
      if (up && ab) hi[k] = mid;
      if (up && !ab) lo[k] = mid + 1;
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = out[k] + lo[k] < n ? out[k] + lo[k] : n - 1;
}

template <class R>
struct SmallSmem {
  R e[SMALL_M];                 // e_i
  uint64_t q[SMALL_M];          // W_i, then Q_i (read by the whole cluster)
  uint64_t s[SMALL_M];          // multinomial: S_j of the CTA's slots
  R ep[SMALL_M / 16];           // sums of 16 consecutive e (read by rank 0)
  uint64_t warp[WARPS], warp2[WARPS];
  uint64_t cum[SMALL_GMAX];     // Q at the end of each CTA's particles
  R red[WARPS];
  R gmax;                       // read by the whole cluster, as are tot, stot and sq
  uint64_t tot, stot;
  U128 sq;
  U128 sqw[WARPS];
  double c[6];
  uint64_t En;                  // multinomial: spacing n
  typename ESumT<R>::T es[SMALL_GMAX * SMALL_M / 512];
  double est_sum[6][WARPS];
  double est_tot[6];
};

template <class R>
__global__ void __launch_bounds__(BLOCK) k_small(FilterArgs<R> a, SmallArgs sa) {
  typedef typename ESumT<R>::T ES;
  __shared__ SmallSmem<R> sm;
  const uint32_t tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_ctarank(), G = cluster_nctarank();
  const uint32_t n = (uint32_t)a.n, m = sa.m;
  const uint32_t lo = rank * m < n ? rank * m : n;
  const uint32_t cnt = lo + m < n ? m : n - lo;
  Ctl* const c = a.ctl;
  const uint32_t t0 = c->t;
  double logml = 0.0, slam = 0.0;  // rank 0, thread 0
  if (rank == 0 && tid == 0) {
    logml = c->logml;
    slam = c->slam;
  }
  const bool learn = sa.learn != 0, ess = sa.ess != 0;
  bool fail = false, rs = true;
  for (uint32_t step = 0; step < sa.steps; ++step) {
    const uint32_t t = t0 + step;
    const double y = sa.y_dev ? sa.y_dev[step] : sa.y[step];
    const R yr = (R)y;
    const StateV<R> src = (t & 1) ? a.st[1] : a.st[0];
    const StateV<R> dst = (t & 1) ? a.st[0] : a.st[1];
    // Step 1: weights of the CTA's particles (thread t: t, t + 256, ...)
    R l[SMALL_K];
    MaxL<R> top;
#pragma unroll
    for (int k = 0; k < SMALL_K; ++k) {
      const uint32_t i = tid + k * BLOCK;
      l[k] = (R)-INFINITY;
      if (i < cnt) {
        const uint32_t g = lo + i;
        const R s2 = __ldcg(src.s2 + g), t2 = __ldcg(src.t2 + g);
        R x = __ldcg(src.x + g);
        if (sa.boot) {  // propagate blind, in place (k_boot_pw)
          const R Z = bm_normal(draw(a.seed, a.filter, t, g, P_BOOT_STATE, 0), (R)0);
          const R xz = sqrt_rn(t2) * Z;
          x = x + xz;
          src.x[g] = x;
        }
        l[k] = log_pred<R>(x, s2, sa.boot ? (R)0 : t2, yr);
        if (ess) l[k] = a.lam[g] + l[k];
        top.take(l[k]);
      }
    }
    fail |= top.bad;
    {
      R v = top.value();
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (lane == 0) sm.red[warp] = v;
    }
    __syncthreads();
    if (tid == 0) {
      R v = sm.red[0];
      for (int w = 1; w < WARPS; ++w) v = fmax(v, sm.red[w]);
      sm.gmax = v;
    }
    // meanwhile: the cycle's Marsaglia-Tsang constants, and the multinomial
    // spacings of the CTA's slots (thread t: slots 4 t .. 4 t + 3)
    if (warp == WARPS - 1 && lane < 2) {
      double d, cc, K;
      mt_constants((lane ? a.a_tau : a.a_sigma) + 0.5 * (double)(t + 1), &d, &cc, &K);
      sm.c[2 * lane] = d; sm.c[2 * lane + 1] = cc; sm.c[4 + lane] = K;
    }
    uint64_t Es[SMALL_K], er = 0;
    if (sa.pos == SP_MULTI) {
      const uint32_t l0 = lo + SMALL_K * tid;  // a multiple of four
      U4 w = {0, 0, 0, 0};
      if (l0 < n && SMALL_K * tid < cnt) w = draw(a.seed, a.filter, t, l0 >> 2, P_SPACING, 0);
#pragma unroll
      for (int e = 0; e < SMALL_K; ++e) {
        if (SMALL_K * tid + e < cnt) er += spacing_E(a.seed, a.filter, t, l0 + e, w);
        Es[e] = er;
      }
      if (tid == BLOCK - 1)
        sm.En = spacing_E(a.seed, a.filter, t, n, draw(a.seed, a.filter, t, n >> 2, P_SPACING, 0));
    }
    cluster_sync_all();  // 1: every CTA's maximum
    R mx = (uint32_t)lane < G ? dsm_real(&sm.gmax, lane) : (R)-INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    // e and W; zero past the CTA's particles
#pragma unroll
    for (int k = 0; k < SMALL_K; ++k) {
      const uint32_t i = tid + k * BLOCK;
      const R e = i < cnt ? exp_weight(l[k] - mx) : (R)0;
      sm.e[i] = e;
      sm.q[i] = quant_from_e(e, a.k);
    }
    __syncthreads();
    uint64_t run[SMALL_K], acc = 0;  // thread t: particles 4 t .. 4 t + 3
    U128 sq{0, 0};
#pragma unroll
    for (int e = 0; e < SMALL_K; ++e) {
      const uint64_t w = sm.q[SMALL_K * tid + e];
      acc += w;
      run[e] = acc;
      if (ess) sq = add128(sq, mul64(w, w));
    }
    if (tid < SMALL_M / 16) {  // log-ML: sums over 16 consecutive particles, in order
      R v = (R)0;
      for (int e = 0; e < 16; ++e) v = v + sm.e[16 * tid + e];
      sm.ep[tid] = v;
    }
    if (ess) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        U128 u;
        u.hi = __shfl_xor_sync(0xffffffffu, sq.hi, o);
        u.lo = __shfl_xor_sync(0xffffffffu, sq.lo, o);
        sq = add128(sq, u);
      }
      if (lane == 0) sm.sqw[warp] = sq;
    }
    uint64_t tot, stot = 0, sexcl = 0;
    const uint64_t qexcl = small_scan(acc, sm.warp, &tot);
    if (sa.pos == SP_MULTI) sexcl = small_scan(er, sm.warp2, &stot);
    if (tid == 0) {
      sm.tot = tot;
      sm.stot = stot;
      if (ess) {
        U128 b = sm.sqw[0];
        for (int w = 1; w < WARPS; ++w) b = add128(b, sm.sqw[w]);
        sm.sq = b;
      }
    }
    cluster_sync_all();  // 2: every CTA's sums
    uint64_t T, A = n, pre, spre = 0;
    {
      const uint64_t v = (uint32_t)lane < G ? dsm_u64(dsm_addr(&sm.tot, lane)) : 0ull;
      const uint64_t in = warp_incl_scan(v, lane);
      T = __shfl_sync(0xffffffffu, in, 31);
      pre = __shfl_sync(0xffffffffu, in - v, rank);
      if (warp == 0 && (uint32_t)lane < G) sm.cum[lane] = in;
    }
    if (sa.pos == SP_MULTI) {
      const uint64_t v = (uint32_t)lane < G ? dsm_u64(dsm_addr(&sm.stot, lane)) : 0ull;
      const uint64_t in = warp_incl_scan(v, lane);
      A = __shfl_sync(0xffffffffu, in, 31) + sm.En;
      spre = __shfl_sync(0xffffffffu, in - v, rank);
    }
    rs = true;
    if (ess) {
      U128 b{0, 0};
      for (uint32_t r = 0; r < G; ++r) {
        U128 v;
        v.hi = dsm_u64(dsm_addr(&sm.sq.hi, r));
        v.lo = dsm_u64(dsm_addr(&sm.sq.lo, r));
        b = add128(b, v);
      }
      const double Ad = __ull2double_rn(T);
      const double Bd = u128_to_f64_rn(b);
      const double lhs = Ad * Ad;
      const double f = sa.ess_frac * (double)a.n;
      const double rhs = f * Bd;
      rs = lhs < rhs;
    }
    fail |= T == 0;
    // the CDF: in place for the search, and out
    const uint64_t q0 = pre + qexcl;
#pragma unroll
    for (int e = 0; e < SMALL_K; ++e) {
      const uint32_t i = SMALL_K * tid + e;
      sm.q[i] = q0 + run[e];
      if (sa.pos == SP_MULTI) sm.s[i] = spre + sexcl + Es[e];
      if (i < cnt) a.Q[lo + i] = q0 + run[e];
    }
    cluster_sync_all();  // 3: every CTA's CDF (and this CTA's S and cum)
    // log-ML (rank 0): the general path's order -- 32 sums of 16 per warp
    // tile, eight of those per tile of 4096, the tiles over the lanes
    if (rank == 0) {
      const uint32_t n512 = (n + 511) / 512;
      for (uint32_t g = warp; g < n512; g += WARPS) {
        const uint32_t i = g * 512 + lane * 16;  // first of the lane's 16 particles
        R v = (R)0;
        if (i < n) v = dsm_real(&sm.ep[(i % m) / 16], i / m);
        ES es;
        es.zero();
        es.add(v);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) es.add(es.shfl_xor(o));
        if (lane == 0) sm.es[g] = es;
      }
      __syncthreads();
      if (warp == 0) {
        ES es;
        es.zero();
        if ((uint32_t)lane * 8 < n512) {
          es = sm.es[lane * 8];
          for (uint32_t g = lane * 8 + 1; g < n512 && g < lane * 8 + 8u; ++g) es.add(sm.es[g]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) es.add(es.shfl_xor(o));
        if (lane == 0) {
          const double LOG_2PI = 0x1.d67f1c864beb5p+0;
          const double S = esum_value(es);
          if (ess) {
            const double inc = (double)mx + log(S) - log(slam) - 0.5 * LOG_2PI;
            logml = logml + inc;
            slam = rs ? (double)a.n : S;
          } else {
            const double inc = (double)mx + log(S) - log((double)a.n) - 0.5 * LOG_2PI;
            logml = logml + inc;
          }
        }
      }
    }
    // Steps 2-4, the CTA's slots.  The ancestor of slot j is the number of
    // particles whose key Q_i A is not above the slot's key B_j: first over the
    // CTAs, then by bisection in that CTA's shared memory.
    uint64_t r = 0;
    if (sa.pos == SP_SYS) {
      const U4 w = draw(a.seed, a.filter, t, 0, P_SYS_OFFSET, 0);
      r = __umul64hi(((uint64_t)w.b << 32) | w.a, T);
    }
    const bool multi = sa.pos == SP_MULTI;
    auto above = [&](uint64_t q, const U128& kb) {  // Q A > B
      return lt128(kb, multi ? mul64(q, A) : mul64x32(q, n));
    };
    uint32_t an[SMALL_K];
    if (rs && T > 0) {
      U128 kb[SMALL_K];
#pragma unroll
      for (int k = 0; k < SMALL_K; ++k) {
        const uint32_t i = tid + k * BLOCK, j = lo + i;
        kb[k] = U128{0, 0};
        if (i < cnt) {
          if (sa.pos == SP_SYS) kb[k] = add128(mul64x32(T, j), r);
          else if (sa.pos == SP_STRAT) kb[k] = add128(mul64x32(T, j), strat_offset(T, a.seed, a.filter, t, j));
          else kb[k] = mul64(sm.s[i], T);
        }
      }
      if (m <= BLOCK) {
        cluster_search<1>(sm.q, sm.cum, G, m, n, kb, above, an);
      } else {
#pragma unroll
        for (int k = 0; k < SMALL_K; k += 2)
          if (k * BLOCK < m) cluster_search<2>(sm.q, sm.cum, G, m, n, kb + k, above, an + k);
      }
    } else {
#pragma unroll
      for (int k = 0; k < SMALL_K; ++k) an[k] = lo + tid + k * BLOCK;
    }
#pragma unroll
    for (int k = 0; k < SMALL_K; ++k) {
      const uint32_t i = tid + k * BLOCK;
      if (i < cnt) a.anc[lo + i] = an[k];
    }
    const R ds = (R)sm.c[0], cs = (R)sm.c[1], dt = (R)sm.c[2], ct = (R)sm.c[3];
    const R ks = (R)sm.c[4], kt = (R)sm.c[5];
    Gathered<R> rec[SMALL_K];
#pragma unroll
    for (int k = 0; k < SMALL_K; ++k) {
      const uint32_t i = tid + k * BLOCK;
      if (i < cnt) {
        const uint32_t g = an[k];
        rec[k].x = __ldcg(src.x + g);
        rec[k].s2 = __ldcg(src.s2 + g);
        rec[k].t2 = __ldcg(src.t2 + g);
        rec[k].bs = __ldcg(src.bs + g);
        rec[k].bt = __ldcg(src.bt + g);
      }
    }
#pragma unroll 1
    for (int k = 0; k < SMALL_K; ++k) {
      const uint32_t i = tid + k * BLOCK, j = lo + i;
      if (i < cnt) {
        Gathered<R> cur = rec[0];
#pragma unroll
        for (int q = 1; q < SMALL_K; ++q)
          if (q == k) cur = rec[q];
        const R xa = cur.x, s2 = cur.s2, t2 = cur.t2;
        if (sa.boot) {  // Step 3: the ancestor as it is
          dst.x[j] = xa;
          dst.s2[j] = s2;
          dst.t2[j] = t2;
          dst.bs[j] = cur.bs;
          dst.bt[j] = cur.bt;
          continue;
        }
        // V and mu share one correctly rounded reciprocal of s
        const R s = s2 + t2;
        const R ri = div_rn((R)1, s);
        const R p = s2 * t2;
        const R V = p * ri;
        const R n2 = yr * t2;
        const R nn = fmaR(xa, s2, n2);
        const R mu = nn * ri;
        const R sv = sqrt_rn(V);
        R Z, Zs, Us, Zt, Ut;
        theta_draws_rk<R>(a.rk, a.filter, t, j, &Z, &Zs, &Us, &Zt, &Ut);
        const R xj = fmaR(sv, Z, mu);
        dst.x[j] = xj;
        if (learn) {
          const R es_ = ResidObs<R>::f(y, yr, xj);
          const R et = xj - xa;
          const auto bsn = SuffOps<R>::add_half_square(cur.bs, es_, &fail);
          const auto btn = SuffOps<R>::add_half_square(cur.bt, et, &fail);
          dst.bs[j] = bsn;
          dst.bt[j] = btn;
          R Gs, Gt;
          if (!gamma_mt_squeeze<R>(ds, cs, ks, Zs, Us, &Gs))
            Gs = gamma_mt_from<R>(ds, cs, ks, Zs, Us, a.seed, a.filter, t, j, P_GAMMA_SIGMA, &fail);
          if (!gamma_mt_squeeze<R>(dt, ct, kt, Zt, Ut, &Gt))
            Gt = gamma_mt_from<R>(dt, ct, kt, Zt, Ut, a.seed, a.filter, t, j, P_GAMMA_TAU, &fail);
          dst.s2[j] = SuffOps<R>::ig(bsn, Gs);
          dst.t2[j] = SuffOps<R>::ig(btn, Gt);
        } else {
          dst.s2[j] = s2;
          dst.t2[j] = t2;
          dst.bs[j] = cur.bs;
          dst.bt[j] = cur.bt;
        }
      }
    }
    if (ess) {  // the carried log-weights: 0 after a resampling, else L - max
#pragma unroll
      for (int k = 0; k < SMALL_K; ++k) {
        const uint32_t i = tid + k * BLOCK;
        if (i < cnt) a.lam[lo + i] = rs ? (R)0 : l[k] - mx;
      }
    }
    // a failure goes to the error word before the last barrier, which orders it
    // before rank 0 publishes that word with the summaries
    if (step + 1 == sa.steps && __syncthreads_or(fail) && tid == 0) atomicOr(&c->err, ERR_NUMERIC);
    cluster_sync_all();  // 4: the new state, before the next cycle reads it
  }
  const uint32_t t1 = t0 + sa.steps;
  if (rank == 0 && tid == 0) {
    c->t = t1;
    c->logml = logml;
    c->slam = slam;
    c->resamp = rs ? 1u : 0u;
  }
  if (!sa.est) return;
  // the summaries: CTA b takes k_estimate's block b, rank 0 folds
  const StateV<R> st = (t1 & 1) ? a.st[1] : a.st[0];
  const R c0 = __ldcg(st.x), c1 = __ldcg(st.s2), c2 = __ldcg(st.t2);
  const uint32_t nblk = (n + BLOCK * EST_PER_THREAD - 1) / (BLOCK * EST_PER_THREAD);
  for (uint32_t b = rank; b < nblk; b += G) est_block<R>(st, a.n, b, c0, c1, c2, sm.est_sum, a.part_est);
  if (nblk > 1) cluster_sync_all();
  if (rank != 0) return;
  est_fold<R>(a, t1, nblk, c0, c1, c2, sm.est_sum, sm.est_tot);
}

// ---------------------------------------------------------------------------
// Resampling of a small weight vector (n <= RES_N) by one cluster, all schemes:
// the quantisation (W_i = floor(w_i 2^(k - e)), max w = f 2^e), the exact CDF and
// the positions of the general path, each slot's ancestor by the same search as
// above -- one launch instead of three to six, no scratch.  Errors go to *err
// (negative / non-finite / all-zero weights: ERR_WEIGHTS).
// ---------------------------------------------------------------------------
// RES_N is what eight CTAs hold.  Against the general path, microseconds per call
// on even weights, here / there: systematic 27.6 / 35.0 at 8192, 31.5 / 34.7 at
// 12,000, 34.3 / 35.6 at 16,384; stratified 35.5 / 42.3, multinomial 37.4 / 54.2
// and the cut-point schemes 34.2 / 44.5 at 16,384 (all mass on one particle,
// where every CTA searches one CTA's memory: systematic 39.9 / 38.0).
constexpr int RES_K = 8;
template <int N> struct Int { static constexpr int value = N; };
constexpr uint32_t RES_M = RES_K * BLOCK;
constexpr uint64_t RES_N = (uint64_t)RES_M * SMALL_GMAX;

static __global__ void __launch_bounds__(BLOCK) k_small_resample(const float* w, uint32_t n, uint32_t m,
                                                          int pos, int kshift, uint64_t seed,
                                                          uint32_t filter, uint32_t t, uint32_t* anc,
                                                          uint32_t* err) {
  __shared__ uint64_t s_q[RES_M], s_s[RES_M];
  __shared__ uint64_t s_warp[WARPS], s_warp2[WARPS], s_cum[SMALL_GMAX];
  __shared__ uint64_t s_tot, s_stot, s_En;
  __shared__ uint32_t s_red[WARPS], s_max;  // s_max: the CTA's largest weight; ~0: a bad one
  const uint32_t tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_ctarank(), G = cluster_nctarank();
  const uint32_t lo = rank * m < n ? rank * m : n;
  const uint32_t cnt = lo + m < n ? m : n - lo;
  float v[RES_K];
  uint32_t mx = 0;
#pragma unroll
  for (int k = 0; k < RES_K; ++k) {
    const uint32_t i = tid + k * BLOCK;
    v[k] = i < cnt ? w[lo + i] : 0.0f;
    mx = max(mx, (!(v[k] >= 0.0f) || !(v[k] < INFINITY)) ? ~0u : __float_as_uint(fabsf(v[k])));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) s_red[warp] = mx;
  // meanwhile: multinomial spacings of the CTA's slots (thread t: 8 t .. 8 t + 7)
  uint64_t Es[RES_K], er = 0;
  if (pos == SP_MULTI) {
#pragma unroll
    for (int h = 0; h < RES_K / 4; ++h) {
      const uint32_t l0 = lo + RES_K * tid + 4 * h;  // a multiple of four
      U4 d = {0, 0, 0, 0};
      if (RES_K * tid + 4 * h < cnt) d = draw(seed, filter, t, l0 >> 2, P_SPACING, 0);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (RES_K * tid + 4 * h + e < cnt) er += spacing_E(seed, filter, t, l0 + e, d);
        Es[4 * h + e] = er;
      }
    }
    if (tid == BLOCK - 1) s_En = spacing_E(seed, filter, t, n, draw(seed, filter, t, n >> 2, P_SPACING, 0));
  }
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < WARPS; ++i) mx = max(mx, s_red[i]);
    s_max = mx;
  }
  cluster_sync_all();  // 1: every CTA's maximum
  mx = __reduce_max_sync(0xffffffffu, (uint32_t)lane < G ? dsm_u32(dsm_addr(&s_max, lane)) : 0u);
  const bool wrong = mx == 0u || mx == ~0u;  // (the same in the whole cluster)
  if (!wrong) {
    int e2;
    (void)frexpf(__uint_as_float(mx), &e2);
#pragma unroll
    for (int k = 0; k < RES_K; ++k) s_q[tid + k * BLOCK] = quant_weight(v[k], kshift - e2);
  }
  __syncthreads();
  uint64_t run[RES_K], acc = 0;  // thread t: particles 8 t .. 8 t + 7
#pragma unroll
  for (int e = 0; e < RES_K; ++e) {
    acc += wrong ? 0ull : s_q[RES_K * tid + e];
    run[e] = acc;
  }
  uint64_t tot, stot = 0, sexcl = 0;
  const uint64_t qexcl = small_scan(acc, s_warp, &tot);
  if (pos == SP_MULTI) sexcl = small_scan(er, s_warp2, &stot);
  if (tid == 0) {
    s_tot = tot;
    s_stot = stot;
  }
  cluster_sync_all();  // 2: every CTA's sums (and its maximum has been read)
  if (wrong) {
    if (rank == 0 && tid == 0) *err = ERR_WEIGHTS;
    for (uint32_t i = tid; i < cnt; i += BLOCK) anc[lo + i] = lo + i;
    return;
  }
  uint64_t T, A = n, pre, spre = 0;
  {
    const uint64_t x = (uint32_t)lane < G ? dsm_u64(dsm_addr(&s_tot, lane)) : 0ull;
    const uint64_t in = warp_incl_scan(x, lane);
    T = __shfl_sync(0xffffffffu, in, 31);
    pre = __shfl_sync(0xffffffffu, in - x, rank);
    if (warp == 0 && (uint32_t)lane < G) s_cum[lane] = in;
  }
  const bool multi = pos == SP_MULTI;
  if (multi) {
    const uint64_t x = (uint32_t)lane < G ? dsm_u64(dsm_addr(&s_stot, lane)) : 0ull;
    const uint64_t in = warp_incl_scan(x, lane);
    A = __shfl_sync(0xffffffffu, in, 31) + s_En;
    spre = __shfl_sync(0xffffffffu, in - x, rank);
  }
  uint64_t r = 0;
  if (pos == SP_SYS) {
    const U4 d = draw(seed, filter, t, 0, P_SYS_OFFSET, 0);
    r = __umul64hi(((uint64_t)d.b << 32) | d.a, T);
  }
#pragma unroll
  for (int e = 0; e < RES_K; ++e) {
    s_q[RES_K * tid + e] = pre + qexcl + run[e];
    if (multi) s_s[RES_K * tid + e] = spre + sexcl + Es[e];
  }
  cluster_sync_all();  // 3: every CTA's CDF
  auto above = [&](uint64_t q, const U128& kb) {  // Q A > B
    return lt128(kb, multi ? mul64(q, A) : mul64x32(q, n));
  };
  U128 kb[RES_K];
#pragma unroll
  for (int k = 0; k < RES_K; ++k) {
    const uint32_t i = tid + k * BLOCK, j = lo + i;
    kb[k] = U128{0, 0};
    if (i < cnt) {
      if (pos == SP_SYS) kb[k] = add128(mul64x32(T, j), r);
      else if (pos == SP_STRAT) kb[k] = add128(mul64x32(T, j), strat_offset(T, seed, filter, t, j));
      else kb[k] = mul64(s_s[i], T);
    }
  }
  uint32_t an[RES_K];
  // as many searches as a thread has slots (with one, four and eight at choice:
  // 28.6 us instead of 25.0 at 4096, 36.7 instead of 30.5 at 8193)
  auto search = [&](auto K) { cluster_search<K.value>(s_q, s_cum, G, m, n, kb, above, an); };
  switch ((m + BLOCK - 1) / BLOCK) {
    case 1: search(Int<1>()); break;
    case 2: search(Int<2>()); break;
    case 3: search(Int<3>()); break;
    case 4: search(Int<4>()); break;
    case 5: search(Int<5>()); break;
    case 6: search(Int<6>()); break;
    case 7: search(Int<7>()); break;
    default: search(Int<8>());
  }
#pragma unroll
  for (int k = 0; k < RES_K; ++k) {
    const uint32_t i = tid + k * BLOCK;
    if (i < cnt) anc[lo + i] = an[k];
  }
  cluster_sync_all();  // 4: no CTA leaves while others search its part
}

}  // namespace pfk
