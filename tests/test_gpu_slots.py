"""Tile sums and slot map (k_sums, k_slots) against the CPU oracle, bit for bit,
where they can go wrong: around the tile sizes (2048 and 4096 particles), with
runs of zero weights, tiles of far more slots than their shared-memory window
(the heavy list) in either source precision, unaligned inputs and outputs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [16385, 8 * 2048 + 2047, 9 * 2048, 5 * 4096 + 1, 100_003, (1 << 18) + 5]


def _shapes(n, rng):
    """Weight vectors: flat, one particle, one tile, zeros before and after a few, two far heavy ones."""
    flat = rng.random(n).astype(np.float32) + np.float32(0.5)
    one = np.zeros(n, np.float32)
    one[n // 3] = 0.25
    tile = np.full(n, 1e-9, np.float32)
    tile[4096:6144] = rng.random(2048).astype(np.float32)
    late = np.zeros(n, np.float32)
    late[-2500:-100] = rng.random(2400).astype(np.float32)
    two = flat * np.float32(1e-3)
    two[[5, n - 1]] = [n * 0.4, n * 0.01]
    grid = np.zeros(n, np.float32)
    grid[::2048] = 1.0  # every tile's slots on its first particle
    return {"flat": flat, "one": one, "tile": tile, "late": late, "two": two, "grid": grid, "equal": np.ones(n, np.float32)}


@pytest.mark.parametrize("scheme", ["systematic", "stratified"])
@pytest.mark.parametrize("n", SIZES)
def test_resample_slots_match_oracle(pf, orc, n, scheme):
    rng = np.random.default_rng(n)
    code = pf.SCHEMES[scheme]
    for name, w in _shapes(n, rng).items():
        ref = orc.resample_weights(w, code, 77, 3, 5)
        wd = torch.from_numpy(w).cuda()
        got = pf.resample(wd, seed=77, filter_id=3, t=5, scheme=scheme).cpu().numpy().view(np.uint32)
        assert np.array_equal(got, ref), (name, np.flatnonzero(got != ref)[:5])
    # 4-byte aligned weights and output
    pad_w = torch.from_numpy(np.concatenate([[0.5], _shapes(n, rng)["two"]]).astype(np.float32)).cuda()[1:]
    pad_o = torch.full((n + 1,), -1, dtype=torch.int32, device="cuda")
    pf.resample(pad_w, seed=9, scheme=scheme, out=pad_o[1:])
    ref = orc.resample_weights(pad_w.cpu().numpy(), code, 9, 0, 0)
    assert np.array_equal(pad_o[1:].cpu().numpy().view(np.uint32), ref) and int(pad_o[0]) == -1


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("scheme", ["systematic", "stratified"])
@pytest.mark.parametrize("ess", [0.0, 0.5])
def test_filter_slots_with_outliers(pf, orc, prec, scheme, ess):
    """Observations far out concentrate the weights on few particles of few tiles."""
    n = 3 * 4096 + 2049
    ys = [0.3, 25.0, -0.2, -40.0, 18.0]
    kw = dict(seed=11, known_variances=True, sigma2=0.05, tau2=0.01, ess_frac=ess)
    g = pf.Filter(n, scheme=scheme, precision=prec, **kw)
    o = orc.Filter(orc.make_config(n, scheme=pf.SCHEMES[scheme], precision=int(prec == "fp64"), **kw))
    for y in ys:
        g.step(y)
        o.step(y)
        anc, Q = g.ancestors(with_cdf=True)
        assert np.array_equal(anc.cpu().numpy().view(np.uint32), o.ancestors())
        assert int(Q[-1]) > 0 and bool((Q[1:] >= Q[:-1]).all())
    assert np.array_equal(g.particles()["x"].cpu().numpy(), o.state_raw()["x"])
