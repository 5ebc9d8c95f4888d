"""Multinomial resampling by slot tiles (k_spacing_sums, k_multi_split, k_multi)
and the cut-point schemes on the table of the slot map, against the CPU oracle,
bit for bit: around the tile size (2048), and on weights whose tiles of slots
span few, many (beyond the staged 4096) or almost all particles."""
import numpy as np
import pytest
import torch

from test_gpu_slots import _shapes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", ["multinomial", "multinomial_cutpoint", "systematic_cutpoint"])
@pytest.mark.parametrize("n", [1, 7, 2047, 2048, 2049, 4097, 16385, 9 * 2048, 100_003])
def test_resample_multinomial_and_cutpoint(pf, orc, n, scheme):
    rng = np.random.default_rng(n + 1)
    if n >= 16385:
        shapes = _shapes(n, rng)
    else:
        spread = np.exp(3.0 * rng.standard_normal(n)).astype(np.float32)
        gaps = np.where(np.arange(n) % 5 == 0, spread, 0).astype(np.float32)
        shapes = {"equal": np.ones(n, np.float32), "spread": spread, "gaps": gaps}
    for name, w in shapes.items():
        ref = orc.resample_weights(w, pf.SCHEMES[scheme], 31, 2, 7)
        got = pf.resample(torch.from_numpy(w).cuda(), seed=31, filter_id=2, t=7, scheme=scheme)
        got = got.cpu().numpy().view(np.uint32)
        assert np.array_equal(got, ref), (name, np.flatnonzero(got != ref)[:5])


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("scheme", ["multinomial", "multinomial_cutpoint"])
def test_filter_multinomial_above_the_cluster_limit(pf, orc, prec, scheme):
    n = 8192 + 2049
    kw = dict(seed=12, known_variances=True, sigma2=0.05, tau2=0.01)
    g = pf.Filter(n, scheme=scheme, precision=prec, **kw)
    o = orc.Filter(orc.make_config(n, scheme=pf.SCHEMES[scheme], precision=int(prec == "fp64"), **kw))
    for y in [0.3, 25.0, -0.2, -40.0]:
        g.step(y)
        o.step(y)
        assert np.array_equal(g.ancestors().cpu().numpy().view(np.uint32), o.ancestors())
    assert np.array_equal(g.particles()["x"].cpu().numpy(), o.state_raw()["x"])
