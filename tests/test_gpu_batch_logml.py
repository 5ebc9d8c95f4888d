"""A batched filter of several scan tiles: its log marginal likelihood equals a
standalone filter's bit for bit after many cycles (a tile's partial sums are
read by one thread while the other warps already form the next tile's)."""
import numpy as np
import pytest

from paper_1212_1639_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_batch_logml_of_several_tiles(pf, prec):
    T, count = 40, 160
    ns = [4097 + 97 * i for i in range(count)]
    ys = np.stack([synth.local_level_series(7, T, filter_id=i)[1] for i in range(count)], axis=1)
    specs = [dict(n=n, seed=100 + i, filter_id=i) for i, n in enumerate(ns)]
    b = pf.Batch(specs, scheme="systematic", precision=prec)
    for y in ys:
        b.step(y)
    e = b.estimates()
    for i in range(0, count, 8):
        f = pf.Filter(scheme="systematic", precision=prec, **specs[i])
        f.run(np.ascontiguousarray(ys[:, i]))
        assert f.estimate() == e[i], i
        f.close()
