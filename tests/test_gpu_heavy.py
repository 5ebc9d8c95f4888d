"""Cycles whose weights concentrate on few particles: tiles of far more slots
than the window they are built in.  Single filters hand the further windows to
other CTAs (binary64 takes the exponentials again from l there); a batched
filter's CTA stores the slots of a heavy particle straight."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# observations that leave one particle, a few, some thousands, all of them
YS = [40.0, -3.0, 0.2, 6.0, -60.0, 0.0, 11.0, 3.5]
KW = dict(known_variances=True, sigma2=0.02, tau2=0.05)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("scheme", ["systematic", "stratified", "systematic_cutpoint", "multinomial"])
@pytest.mark.parametrize("ess", [0.0, 0.5])
def test_filter_with_heavy_tiles(pf, orc, prec, scheme, ess):
    n = 150_001
    g = pf.Filter(n, seed=23, scheme=scheme, precision=prec, ess_frac=ess, **KW)
    o = orc.Filter(orc.make_config(n, seed=23, scheme=pf.SCHEMES[scheme], precision=int(prec == "fp64"),
                                   ess_frac=ess, **KW))
    fewest = n
    for y in YS:
        g.step(y)
        o.step(y)
        a = g.ancestors().cpu().numpy().view(np.uint32)
        assert np.array_equal(a, o.ancestors()), y
        fewest = min(fewest, len(np.unique(a)))
    assert fewest < 10  # some cycle had tiles of many windows
    assert np.array_equal(g.particles()["x"].cpu().numpy(), o.state_raw()["x"])
    g.close()


@pytest.mark.parametrize("scheme", ["systematic", "stratified"])
@pytest.mark.parametrize("n", [4097, 8193, 12_289, 28_607, 28_608, 28_609, 28_656, 28_657, 28_672, 28_673, 32_769])
def test_binary64_windows_of_one_tile(pf, orc, n, scheme):
    """All slots in one tile: its own CTA stores seven windows, other CTAs the rest."""
    g = pf.Filter(n, seed=n, scheme=scheme, precision="fp64", **KW)
    o = orc.Filter(orc.make_config(n, seed=n, scheme=pf.SCHEMES[scheme], precision=1, **KW))
    tiles = []
    for y in (60.0, -60.0, 60.0):
        g.step(y)
        o.step(y)
        a = g.ancestors().cpu().numpy().view(np.uint32)
        assert np.array_equal(a, o.ancestors()), y
        tiles.append(len(np.unique(a // 2048)))
    assert min(tiles) == 1
    g.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", [None, (512, 152, 1, 0), (256, 152, 8, 16384), (512, 152, 8, 16384)])
def test_batch_with_heavy_particles(pf, prec, shape):
    ns = [131_072, 40_003, 9000, 4096, 65_535]
    specs = [dict(n=n, seed=50 + i, filter_id=i, **KW) for i, n in enumerate(ns)]
    b = pf.Batch(specs, scheme="systematic", precision=prec)
    if shape:
        try:
            b.set_shape(*shape)
        except pf.PfError:
            pytest.skip("shape not resident on this part")
    fs = [pf.Filter(scheme="systematic", precision=prec, **s) for s in specs]
    for y in YS:
        b.step(np.full(len(ns), y))
        for i, f in enumerate(fs):
            f.step(y)
            assert np.array_equal(b.ancestors(i).cpu().numpy(), f.ancestors().cpu().numpy()), (y, ns[i])
    for i, f in enumerate(fs):
        p, r = b.particles(i), f.particles()
        assert all(np.array_equal(p[k].cpu().numpy(), r[k].cpu().numpy()) for k in r)
        f.close()
    b.close()
