"""Handles on device memory that starts at 16 bytes past a multiple of 32, as a
caller's allocator may give it: the same results as on the default allocator's
memory, and the blocks freed as they came."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1212_1639_gb300 import synth

pytestmark = pytest.mark.gpu


class Shifted:
    """Torch's caching allocator, every block 16 bytes further on."""

    def __init__(self, pf):
        self.live = {}
        dev = torch.cuda.current_device()

        def _alloc(nbytes, stream, ctx):
            base = torch.cuda.caching_allocator_alloc(int(nbytes) + 16, dev, stream)
            self.live[base + 16] = base
            return base + 16

        def _free(p, stream, ctx):
            torch.cuda.caching_allocator_delete(self.live.pop(p))

        self.alloc, self.free = pf.ALLOC_FN(_alloc), pf.FREE_FN(_free)


@pytest.fixture
def shifted(pf):
    """A shifted allocator, once the host code is seen to align its blocks: no
    kernel is launched on a block that it would misread."""
    a = Shifted(pf)
    raw, start = C.c_void_p(), C.c_void_p()
    for nbytes in (1, 256, 4096, 100_000):
        assert pf._lib.pf_diag_block(a.alloc, a.free, None, nbytes, C.byref(raw), C.byref(start)) == pf.PF_OK
        assert raw.value % 32 == 16 and start.value == raw.value + 16
        a.free(raw.value, None, None)
    assert not a.live
    return a


@pytest.mark.parametrize("scheme,prec,n,kw", [
    ("systematic", "fp32", 1000, {}),
    ("systematic", "fp32", 70_001, {}),
    ("stratified", "fp32", 70_001, {}),
    ("multinomial", "fp32", 70_001, {}),
    ("multinomial_cutpoint", "fp32", 9000, {}),
    ("systematic", "fp32", 70_001, {"ess_frac": 0.5}),
    ("systematic", "fp64", 20_001, {}),
    ("multinomial", "fp64", 20_001, {"ess_frac": 0.5}),
    ("stratified", "fp64", 2001, {"known_variances": True, "algorithm": "bootstrap"}),
])
def test_filter_on_shifted_memory(pf, shifted, scheme, prec, n, kw):
    _, y = synth.local_level_series(17, 6)
    f = pf.Filter(n, seed=3, scheme=scheme, precision=prec, torch_alloc=shifted, **kw)
    g = pf.Filter(n, seed=3, scheme=scheme, precision=prec, **kw)
    assert shifted.live
    for h in (f, g):
        h.run(y[:4])
        h.step_ahead(y[4], y[5])
        h.step(y[5])
    p, r = f.particles(), g.particles()
    assert all(torch.equal(p[k], r[k]) for k in r)
    assert torch.equal(f.ancestors(), g.ancestors())
    assert f.step_estimate(0.25) == g.step_estimate(0.25)
    f.close()
    assert not shifted.live


@pytest.mark.parametrize("scheme,prec,adaptive", [("systematic", "fp32", False), ("systematic", "fp32", True),
                                                  ("multinomial", "fp32", False), ("systematic", "fp64", False)])
def test_batch_on_shifted_memory(pf, shifted, scheme, prec, adaptive):
    specs = [dict(n=n, seed=n, filter_id=i, ess_frac=0.5 if adaptive and i % 2 else 0.0)
             for i, n in enumerate([1, 300, 4099, 20_001, 4096, 7])]
    _, y = synth.local_level_series(19, 5)
    b = pf.Batch(specs, scheme=scheme, precision=prec, adaptive=adaptive, torch_alloc=shifted)
    c = pf.Batch(specs, scheme=scheme, precision=prec, adaptive=adaptive)
    for h in (b, c):
        for v in y:
            h.step(np.full(len(specs), v))
    assert b.estimates() == c.estimates()
    b.close()
    assert not shifted.live
