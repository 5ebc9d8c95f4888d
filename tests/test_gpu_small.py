"""Cycles of a small filter in one cluster launch (k_small) against the CPU
oracle, bit for bit: sizes around a CTA's share (multiples of 32 per CTA of 8)
and the limits (8192 particles binary32, 4096 binary64), blocks of observations
longer than one launch takes (64), host and device observations, and cycles of
the other forms in between."""
import numpy as np
import pytest
import torch

from paper_1212_1639_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = {"fp32": [1, 2, 31, 33, 255, 256, 257, 1000, 4099, 8191, 8192, 8193],
         "fp64": [1, 33, 257, 1000, 4095, 4096, 4097]}


def _pair(pf, orc, n, scheme, prec, **kw):
    g = pf.Filter(n, scheme=scheme, precision=prec, **kw)
    return g, orc.Filter(orc.make_config(n, scheme=pf.SCHEMES[scheme], precision=int(prec == "fp64"), **kw))


def _same(g, o, prec):
    p, r = {k: v.cpu().numpy() for k, v in g.particles().items()}, o.state_raw()
    for k in ("x", "sigma2", "tau2"):
        assert np.array_equal(p[k], r[k]), k
    for k in ("b_sigma", "b_tau"):
        assert np.array_equal(p[k].view(np.uint64) if prec == "fp32" else p[k], r[k]), k
    assert np.array_equal(g.ancestors().cpu().numpy().view(np.uint32), o.ancestors())
    e, f = g.estimate(), o.estimate()
    assert e["t"] == f["t"]
    tol = 1e-5 if prec == "fp32" else 1e-12
    assert abs(e["log_marglik"] - f["log_marglik"]) <= tol * max(1.0, abs(f["log_marglik"]))


@pytest.mark.parametrize("scheme", ["systematic", "multinomial", "stratified"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_small_sizes(pf, orc, prec, scheme):
    _, y = synth.local_level_series(5, 6)
    for n in SIZES[prec]:
        g, o = _pair(pf, orc, n, scheme, prec, seed=n)
        g.run(y)
        for v in y:
            o.step(v)
        _same(g, o, prec)
        g.close()


@pytest.mark.parametrize("kw", [{}, {"ess_frac": 0.5}, {"known_variances": True, "sigma2": 0.4, "tau2": 0.2}])
def test_small_blocks_and_forms(pf, orc, kw):
    """130 observations as blocks of 70 (host) and 30 (device), single steps, step_estimate, step_ahead."""
    _, y = synth.local_level_series(6, 130)
    y = y.copy()
    y[40] += 12.0  # an outlier
    g, o = _pair(pf, orc, 777, "multinomial_cutpoint", "fp32", seed=3, **kw)
    g.run(y[:70])
    g.run(torch.from_numpy(y[70:100]).cuda())
    g.step(y[100])
    g.step_estimate(y[101])
    g.step_ahead(y[102], y[103])
    g.run(y[103:129])
    e = g.step_estimate(y[129])
    for v in y:
        o.step(v)
    _same(g, o, "fp32")
    assert e == g.estimate()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [1, 300, 4096, 10_000])
def test_small_and_general_bootstrap(pf, orc, n, prec):
    _, y = synth.local_level_series(8, 7)
    kw = dict(seed=n, known_variances=True, sigma2=0.8, tau2=0.3)
    g = pf.Filter(n, scheme="stratified", precision=prec, algorithm="bootstrap", **kw)
    o = orc.Filter(orc.make_config(n, scheme=pf.SCHEMES["stratified"], precision=int(prec == "fp64"), algorithm=1, **kw))
    g.run(y)
    for v in y:
        o.step(v)
    _same(g, o, prec)
