"""Binary32 propagation around the sizes where the launch changes form.

The learning forms hand their slots out by ticket from a number of 64-slot units
per warp on, the fused and the known-variance forms never do.  A slot's
arithmetic does not depend on the warp that computes it, so every particle
equals the oracle's exactly on both sides of each line.
"""
import numpy as np
import pytest
import torch

from paper_1212_1639_gb300 import synth

pytestmark = pytest.mark.gpu

UNITS_PER_WARP = {"plain": 68, "adaptive": 44}  # where tickets begin


def _edge(form):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 64 * UNITS_PER_WARP[form] * sms * 3 * 8  # 3 CTAs of 8 warps per SM


@pytest.mark.parametrize("form,offset", [("plain", -64), ("plain", -63), ("plain", 1),
                                         ("adaptive", -64), ("adaptive", -63), ("adaptive", 1)])
def test_ticket_edge(pf, orc, form, offset):
    n = _edge(form) + offset
    kw = {"ess_frac": 0.5} if form == "adaptive" else {}
    g = pf.Filter(n, seed=7, scheme="systematic", precision="fp32", **kw)
    o = orc.Filter(orc.make_config(n, seed=7, scheme=1, precision=0, **kw))
    _, y = synth.local_level_series(1212, 3)
    for v in y:
        g.step(float(v))
        o.step(float(v))
    p, r = g.particles(), o.state_raw()
    for k in ("x", "sigma2", "tau2", "b_sigma", "b_tau"):
        got = p[k].cpu().numpy()
        assert np.array_equal(got.view(r[k].dtype), r[k]), k
    g.close()


@pytest.mark.parametrize("kw,ahead", [({}, True), ({"known_variances": True}, False),
                                      ({"known_variances": True, "ess_frac": 0.5}, False)])
def test_fixed_forms_large(pf, orc, kw, ahead):
    n = (1 << 22) + 1
    g = pf.Filter(n, seed=8, scheme="systematic", precision="fp32", **kw)
    o = orc.Filter(orc.make_config(n, seed=8, scheme=1, precision=0, **kw))
    _, y = synth.local_level_series(1212, 4)
    for t in range(3):
        if ahead:
            g.step_ahead(float(y[t]), float(y[t + 1]))
        else:
            g.step(float(y[t]))
        o.step(float(y[t]))
    p, r = g.particles(), o.state_raw()
    for k in ("x", "sigma2", "tau2"):
        assert np.array_equal(p[k].cpu().numpy(), r[k]), k
    g.close()
