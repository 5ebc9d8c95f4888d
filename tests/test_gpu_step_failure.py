"""A numeric failure of any particle reaches the call that publishes its cycle's
summaries, whichever CTA holds the particle.

The particle is made to fail through a checkpoint: its x is replaced by a NaN,
whose log-likelihood is left out of the maximum and fails the cycle.  A small
filter's cycle runs in one cluster of eight CTAs, and the first of them
publishes the error word with the summaries."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LAST = {"fp32": [2, 33, 4096, 4097, 8192, 8193], "fp64": [2, 33, 4096, 4097]}


def _with_nan(f, i):
    """f's checkpoint with a NaN for particle i's x (the arrays end the checkpoint, x first)."""
    rs = 4 if f.precision == 0 else 8
    blob = f.checkpoint().copy()
    lam = rs if f._cfg.ess_frac > 0 else 0
    at = blob.size - f.n * (3 * rs + 16 + lam)
    x = blob[at:at + f.n * rs].view(np.float32 if rs == 4 else np.float64)
    assert np.isfinite(x).all()
    x[i] = np.nan
    return blob


@pytest.mark.parametrize("kw", [{}, {"ess_frac": 0.5}])
@pytest.mark.parametrize("scheme", ["systematic", "multinomial"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_step_estimate_reports_a_failure_of_the_last_particle(pf, prec, scheme, kw):
    for n in LAST[prec]:
        f = pf.Filter(n, seed=n, scheme=scheme, precision=prec, **kw)
        f.run([0.2, -0.1])
        good = f.checkpoint()
        bad = _with_nan(f, n - 1)
        for _ in range(20):
            g = pf.Filter.restore(bad)
            with pytest.raises(pf.PfError) as e:
                g.step_estimate(0.3)
            assert e.value.status == pf.PF_ERR_NUMERIC, n
            with pytest.raises(pf.PfError):  # and stays failed
                g.step(0.1)
            g.close()
        g = pf.Filter.restore(good)
        assert g.step_estimate(0.3)["t"] == 3
        g.close()
        f.close()
