"""Performance cases: what programs built on this library spend their time in.

Five kinds of work, each through the public binding (pf.Filter, pf.resample,
pf.Batch):

  online    one filter, a summary read after every observation (step_estimate)
  run       one filter over a block of observations, then its summaries and
            particles (run, estimate, particles): offline learning, the paper's
            own experiment
  resample  ancestors for a weight vector of the caller's own (pf.resample):
            the paper's subject, used by filters of other models
  batch     many filters of uneven size advanced together, then every summary
  sparse    a batch of which a few filters at a time have a new observation:
            one cycle of a server, with the server's cluster launch

Sizes span 2^8 to 2^24 particles, in powers of two and ragged; options are the
schemes, both precisions, learned and known variances, the bootstrap filter and
adaptive resampling.  Every pass of a filter or batch takes its next block of
observations, so its state moves on as it does in use.
"""
import math

import numpy as np
import torch

from paper_1212_1639_gb300 import pf, synth

SCHEMES = ("multinomial", "systematic", "multinomial_cutpoint", "systematic_cutpoint", "stratified")
SUMMARY = ("x_mean", "x_var", "sigma2_mean", "sigma2_var", "tau2_mean", "tau2_var", "log_marglik")
BLOCKS = 48                # blocks of observations before a series runs backwards
MOST_EXACT = 9_000_000     # particle-steps that exact() computes in numpy


def _filter(kind, n, steps, warm, scheme="systematic", precision="fp32", **more):
    return dict(kind=kind, n=n, steps=steps, warm=warm, scheme=scheme, precision=precision,
                known=more.get("known", False), bootstrap=more.get("bootstrap", False),
                ess=more.get("ess", 0.0))


def listed():
    return [
        # a small filter behind a live feed: a summary per observation, launch latency
        dict(_filter("online", 1024, 32, 16), name="online_1k"),
        # the headline size, read after every observation
        dict(_filter("online", 1 << 20, 8, 16), name="online_1m"),
        # the at-scale filter over a block of a long series, working set above L2
        dict(_filter("run", 1 << 24, 8, 50), name="run_16m"),
        # the paper's run: 1,024 particles, 100 observations, binary64, multinomial
        dict(_filter("run", 1024, 100, 0, "multinomial", "fp64"), name="run_paper_1k_fp64"),
        # binary64 state at the headline size
        dict(_filter("run", 1 << 20, 4, 4, "systematic", "fp64"), name="run_1m_fp64"),
        # the paper's multinomial resampling at scale
        dict(_filter("run", 1 << 24, 4, 50, "multinomial"), name="run_16m_multinomial"),
        # stratified resampling, a ragged size
        dict(_filter("run", 1_000_003, 8, 16, "stratified"), name="run_1m_stratified"),
        # resampling only when the effective sample size asks for it, ragged
        dict(_filter("run", 2_600_003, 8, 16, ess=0.5), name="run_2m6_adaptive"),
        # resampling alone: a weight vector of a large filter of another model
        dict(kind="resample", n=1 << 24, scheme="systematic", spread=1.0, name="resample_16m"),
        # the paper's cut-point method (Section 3.2) on concentrated weights
        dict(kind="resample", n=1 << 20, scheme="multinomial_cutpoint", spread=1.0,
             name="resample_1m_cutpoint"),
        # thousands of series at once, every filter with a new observation
        dict(kind="batch", filters=4096, lo=256, hi=65536, steps=8, scheme="systematic",
             precision="fp32", name="batch_4096"),
        # a server's cycles: 80 of 2,000 resident streams have an observation
        dict(kind="sparse", filters=2000, lo=512, hi=131072, active=80, steps=8,
             scheme="systematic", precision="fp32", name="sparse_2000"),
    ]


def _log_int(rng, lo, hi):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, v))


def _size(rng, lo, hi):
    """Log-uniform; two in three as they fall (mostly odd shapes), one in three a power of two."""
    n = _log_int(rng, lo, hi)
    return 1 << int(round(math.log2(n))) if rng.random() < 1 / 3 else n


def draw(rng):
    kind = rng.choice(("online", "run", "run", "run", "resample", "resample", "batch", "sparse"))
    if kind == "resample":
        return dict(kind=kind, n=_size(rng, 1 << 8, 1 << 24), scheme=rng.choice(SCHEMES[:2] + SCHEMES),
                    spread=round(rng.choice((0.1, 1.0, 1.0, 5.0)) * rng.uniform(0.9, 1.1), 3))
    precision = rng.choice(("fp32", "fp32", "fp32", "fp64"))
    if kind in ("batch", "sparse"):
        filters = _log_int(rng, 16, 2000)
        hi = _log_int(rng, 4096, 65536 if precision == "fp32" else 16384)
        return dict(kind=kind, filters=filters, lo=_log_int(rng, 256, 1024), hi=hi,
                    steps=rng.randint(2, 8), scheme=rng.choice(("systematic", "systematic", "multinomial")),
                    precision=precision, **({"active": max(1, filters // rng.randint(4, 40))}
                                            if kind == "sparse" else {}))
    n = _size(rng, 1 << 8, (1 << 24 if kind == "run" else 1 << 21) if precision == "fp32" else 1 << 20)
    steps = max(2, min(rng.randint(4, 32), (1 << 25 if precision == "fp32" else 1 << 21) // n))
    option = rng.choice(("plain",) * 4 + ("known", "bootstrap", "ess"))
    return _filter(kind, n, steps, rng.choice((0, 8, 32)), rng.choice(SCHEMES[:2] + ("systematic", "stratified") + SCHEMES),
                   precision, known=option in ("known", "bootstrap"), bootstrap=option == "bootstrap",
                   ess=round(rng.uniform(0.3, 0.7), 2) if option == "ess" else 0.0)


def _series(seed, T, count=1):
    """T observations of `count` local-level series: T x count, running forwards and then
    backwards over the same values, so that it can be repeated without a jump."""
    rng = np.random.default_rng([int(seed), T, count])
    x = np.cumsum(rng.standard_normal((T, count)) * math.sqrt(0.1), axis=0)
    y = x + rng.standard_normal((T, count))
    return np.concatenate([y, y[::-1]])


def _observations(case, seed):
    y = np.ascontiguousarray(_series(seed, BLOCKS * case["steps"])[:, 0])
    return y[len(y) - case["warm"]:], y


def _weights(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    lw = torch.randn(case["n"], device="cuda", dtype=torch.float64, generator=g) * case["spread"]
    w = torch.exp(lw - lw.max())
    return (w / w.sum()).float()


def _members(case, seed):
    ns, _, _ = synth.batch_specs(case["filters"], seed, case["lo"], case["hi"])
    return [dict(n=int(n), seed=int(seed) * 1000 + i, filter_id=i) for i, n in enumerate(ns)]


def _active(case, seed):
    rng = np.random.default_rng([int(seed), 0xAC])
    masks = np.zeros((2 * BLOCKS * case["steps"], case["filters"]), dtype=np.uint8)
    for m in masks:
        m[rng.choice(case["filters"], case["active"], replace=False)] = 1
    return masks


def prepare(case, seed):
    """What a program holds before the call: a filter that has taken its first observations,
    a weight vector, a batch with its filters admitted; and the observations to come."""
    if case["kind"] == "resample":
        return dict(case=case, seed=int(seed), t=0, w=_weights(case, seed))
    if case["kind"] in ("batch", "sparse"):
        b = pf.Batch(_members(case, seed), scheme=case["scheme"], precision=case["precision"])
        s = dict(case=case, i=0, batch=b, y=_series(seed, BLOCKS * case["steps"], case["filters"]))
        if case["kind"] == "sparse":
            s["masks"] = _active(case, seed)
            # the server's launch shape: large filters by clusters of 8 CTAs, as many as fit
            for grid in (408, 304, 152, 8):
                try:
                    b.set_shape(256, grid, 8, 16384)
                    break
                except pf.PfError:
                    continue
        b.sync()
        return s
    f = pf.Filter(case["n"], seed=int(seed), scheme=case["scheme"], precision=case["precision"],
                  known_variances=case["known"], ess_frac=case["ess"],
                  algorithm="bootstrap" if case["bootstrap"] else "pl")
    warm, y = _observations(case, seed)
    f.run(warm)
    f.sync()
    return dict(case=case, i=0, filter=f, y=y)


def _row(e):
    return [e[k] for k in SUMMARY]


def run(s):
    case = s["case"]
    if case["kind"] == "resample":
        s["t"] += 1
        return pf.resample(s["w"], s["seed"], t=s["t"], scheme=case["scheme"])
    k = case["steps"]
    at = s["i"] * k % len(s["y"])
    s["i"] += 1
    y = s["y"][at:at + k]
    if case["kind"] == "online":
        f = s["filter"]
        rows = [_row(f.step_estimate(v)) for v in y]
        return dict(summaries=np.array(rows), particles=f.particles())
    if case["kind"] == "run":
        f = s["filter"]
        f.run(y)
        return dict(summaries=np.array(_row(f.estimate())), particles=f.particles())
    b = s["batch"]
    if case["kind"] == "batch":
        for v in y:
            b.step(v)
        e = b.estimates()
        return dict(summaries=np.array([_row(e[i]) for i in range(case["filters"])]))
    rows = []
    for v, m in zip(y, s["masks"][at:at + k]):
        b.step(v, m)
        e = b.estimates(m)
        rows += [_row(e[i]) for i in np.flatnonzero(m)]
    return dict(summaries=np.array(rows))


def _particles(case):
    """Particle-steps of one pass."""
    if case["kind"] in ("online", "run"):
        return case["n"] * case["steps"]
    span = math.log(case["hi"] / case["lo"])
    mean = (case["hi"] - case["lo"]) / span if span > 0 else case["lo"]  # log-uniform sizes
    return case.get("active", case["filters"]) * mean * case["steps"]


def work(case):
    if case["kind"] == "resample":
        # a 32-bit weight in and a 32-bit ancestor out; scale, round, add, compare
        return dict(bytes=8.0 * case["n"], flops=4.0 * case["n"])
    # per particle and cycle: the state (x, two variances, two 64-bit statistics) in and out;
    # about 150 floating-point operations of the weight, the state draw and the two gamma draws
    # in binary32, 250 in binary64 (longer polynomials, one draw more)
    fp64 = case["precision"] == "fp64"
    p = _particles(case)
    return dict(bytes=p * 2 * (40 if fp64 else 28), flops=p * (250 if fp64 else 150))


# ---------------------------------------------------------------------------
# The same results in 64 bits, in numpy: the Philox counters of the library's
# documented layout, its draws, and the filter's formulas in binary64.
# ---------------------------------------------------------------------------
INIT_X, INIT_SIGMA, INIT_TAU, STATE, G_SIGMA, G_TAU, OFFSET, SPACING, STRATUM, BOOT = range(1, 11)


class _Draws:
    """Uniforms and normals of one filter's counters."""

    def __init__(self, seed, filter_id, fp64):
        self.key = (int(seed) & 0xFFFFFFFF, (int(seed) >> 32) & 0xFFFFFFFF)
        self.filter, self.fp64 = filter_id, fp64

    def words(self, j, t, purpose, attempt=0):
        m32 = np.uint64(0xFFFFFFFF)
        c0 = np.asarray(j, dtype=np.uint64)
        c1 = np.full_like(c0, t)
        c2 = np.full_like(c0, self.filter)
        c3 = np.full_like(c0, purpose | attempt << 8)
        k0, k1 = self.key
        for _ in range(10):
            p0, p1 = c0 * np.uint64(0xD2511F53), c2 * np.uint64(0xCD9E8D57)
            c0, c1, c2, c3 = (p1 >> np.uint64(32) ^ c1 ^ np.uint64(k0), p1 & m32,
                              p0 >> np.uint64(32) ^ c3 ^ np.uint64(k1), p0 & m32)
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        return c0, c1, c2, c3

    @staticmethod
    def u23(w):
        return (2.0 * (w >> np.uint64(9)) + 1.0) * 2.0 ** -24

    def normals(self, w):
        """Box-Muller's two outputs and the spare uniform of one block of words."""
        if self.fp64:
            u1 = (2.0 * ((w[1] << np.uint64(32) | w[0]) >> np.uint64(12)) + 1.0) * 2.0 ** -53
            u2, spare = (2.0 * w[2] + 1.0) * 2.0 ** -33, (2.0 * w[3] + 1.0) * 2.0 ** -33
        else:
            u1, u2, spare = self.u23(w[0]), self.u23(w[1]), self.u23(w[2])
        r = np.sqrt(-2.0 * np.log(u1))
        return r * np.cos(2 * np.pi * u2), r * np.sin(2 * np.pi * u2), spare

    def gamma(self, shape, j, t, purpose, Z=None, U=None):
        """Gamma(shape, 1) by Marsaglia and Tsang; attempt 0 on (Z, U) where they are given."""
        d = shape - 1.0 / 3.0
        c = 1.0 / math.sqrt(9.0 * d)
        out, todo = np.empty(len(j)), np.arange(len(j))
        for attempt in range(16):
            if attempt or Z is None:
                z, _, u = self.normals(self.words(j[todo], t, purpose, attempt))
            else:
                z, u = Z, U
            v3 = (1.0 + c * z) ** 3
            with np.errstate(invalid="ignore", divide="ignore"):
                ok = (v3 > 0) & (np.log(u) < 0.5 * z * z + d * (1.0 - v3 + np.log(v3)))
            out[todo[ok]] = d * v3[ok]
            todo = todo[~ok]
            if not len(todo):
                break
        return out


def _positions(scheme, D, n, t):
    """The n sorted positions in [0, 1)."""
    j = np.arange(n, dtype=np.float64)
    if scheme.startswith("systematic"):
        w = D.words([0], t, OFFSET)
        return (j + float(w[1][0] << np.uint64(32) | w[0][0]) * 2.0 ** -64) / n
    if scheme == "stratified":
        w = D.words(np.arange((n + 1) // 2), t, STRATUM)
        u = np.stack([w[1] << np.uint64(32) | w[0], w[3] << np.uint64(32) | w[2]], 1).reshape(-1)[:n]
        return (j + u * 2.0 ** -64) / n
    w = np.stack(D.words(np.arange(n // 4 + 1), t, SPACING), 1).reshape(-1)[:n + 1]
    S = np.cumsum(np.floor(-np.log(D.u23(w)) * 2.0 ** 31).astype(np.uint64))
    return S[:n] / float(S[n])


def _filter64(cfg, seed, filter_id, ys):
    """Cycles of one filter over ys: the summaries after each, and the particles after the last."""
    n, fp64, learn = cfg["n"], cfg["precision"] == "fp64", not cfg["known"]
    a0, b0, k = 3.0, 2.0, 61 - max(0, (n - 1).bit_length())
    D = _Draws(seed, filter_id, fp64)
    j = np.arange(n, dtype=np.uint64)
    x = math.sqrt(10.0) * D.normals(D.words(j, 0, INIT_X))[0]
    bs, bt = np.full(n, b0), np.full(n, b0)
    s2 = bs / D.gamma(a0, j, 0, INIT_SIGMA) if learn else np.full(n, 1.0)
    t2 = bt / D.gamma(a0, j, 0, INIT_TAU) if learn else np.full(n, 0.1)
    lam, log_ml, rows = np.zeros(n), 0.0, []
    for t, y in enumerate(ys):
        if cfg["bootstrap"]:
            x = x + np.sqrt(t2) * D.normals(D.words(j, t, BOOT))[0]
            s = s2
        else:
            s = s2 + t2
        L = lam - 0.5 * (np.log(s) + (y - x) ** 2 / s)
        m = L.max()
        e = np.where(L - m >= -50.0, np.exp(L - m), 0.0)
        log_ml += m + math.log(e.sum()) - math.log(np.exp(lam).sum()) - 0.5 * math.log(2 * math.pi)
        W = np.floor(e * 2.0 ** k).astype(np.uint64)
        Q = np.cumsum(W)
        again = not cfg["ess"] or float(Q[-1]) ** 2 < cfg["ess"] * n * (W.astype(np.float64) ** 2).sum()
        if again:
            # positions and CDF on the scale of n, where both are near whole numbers
            a = np.searchsorted(Q / float(Q[-1]), _positions(cfg["scheme"], D, n, t), side="right")
            a = np.minimum(a, n - 1)
        else:
            a = np.arange(n)
        lam = np.zeros(n) if again else L - m
        x, s2, t2, bs, bt = x[a], s2[a], t2[a], bs[a], bt[a]
        if not cfg["bootstrap"]:
            Z, Zs, Us = D.normals(D.words(j, t, STATE))
            if fp64:
                Zt, _, Ut = D.normals(D.words(j, t, STATE, 1))
            else:  # the two slots of a pair share the second block
                w = D.words(np.arange((n + 1) // 2), t, STATE, 1)
                zc, zs, _ = D.normals(w)
                Zt = np.stack([zc, zs], 1).reshape(-1)[:n]
                Ut = np.stack([D.u23(w[2]), D.u23(w[3])], 1).reshape(-1)[:n]
            s = s2 + t2
            xn = np.sqrt(s2 * t2 / s) * Z + (x * s2 + y * t2) / s
            if learn:
                bs, bt = bs + 0.5 * (y - xn) ** 2, bt + 0.5 * (xn - x) ** 2
                s2 = bs / D.gamma(a0 + 0.5 * (t + 1), j, t, G_SIGMA, Zs, Us)
                t2 = bt / D.gamma(a0 + 0.5 * (t + 1), j, t, G_TAU, Zt, Ut)
            x = xn
        w = np.exp(lam) / np.exp(lam).sum()
        row = []
        for v in (x, s2, t2):
            mean = float((w * v).sum())
            row += [mean, float((w * (v - mean) ** 2).sum())]
        rows.append(row + [log_ml])
    return np.array(rows), dict(x=x, sigma2=s2, tau2=t2, b_sigma=bs, b_tau=bt)


def exact(case, seed):
    """None where the outputs are whole numbers (ancestors, equal bit for bit) or the numpy
    cycles would take too long.  Particles whose weights (binary32 state) or sorted uniforms
    (multinomial: binary32 logarithms in both precisions) are defined in 32 bits have no value
    in 64: a resampling boundary that falls to the other side moves a slot to another particle.
    Only their summaries are given."""
    if case["kind"] == "resample":
        return None
    if case["kind"] in ("batch", "sparse"):
        members, ys = _members(case, seed), _series(seed, BLOCKS * case["steps"], case["filters"])
        masks = _active(case, seed) if case["kind"] == "sparse" else None
        per = max(1, case["steps"] * case.get("active", case["filters"]))
        if per > 2000 or case["steps"] * sum(c["n"] for c in members) > MOST_EXACT:
            return None
        cfg = dict(case, known=False, bootstrap=False, ess=0.0)
        got = []
        for i, c in enumerate(members):
            mine = [v for v in range(case["steps"]) if masks is None or masks[v][i]]
            r = _filter64(dict(cfg, n=c["n"]), c["seed"], i, ys[mine, i])[0] if mine else []
            got.append(dict(zip(mine, r)))
        if masks is None:
            return dict(summaries=np.array([g[case["steps"] - 1] for g in got]))
        return dict(summaries=np.array([got[i][v] for v in range(case["steps"])
                                        for i in np.flatnonzero(masks[v])]))
    if case["n"] * (case["steps"] + case["warm"]) > MOST_EXACT:
        return None
    warm, y = _observations(case, seed)
    rows, particles = _filter64(case, seed, 0, np.concatenate([warm, y[:case["steps"]]]))
    rows = rows[case["warm"]:]
    return dict(summaries=rows if case["kind"] == "online" else rows[-1],
                particles=particles if case["precision"] == "fp64"
                and not case["scheme"].startswith("multinomial") else None)
