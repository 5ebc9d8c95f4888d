"""pf_resample in one cluster launch: a thread of the eight CTAs has one to eight
slots, and searches for as many.  Ancestors equal the oracle's on both sides of
every step and at the limits."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [1, 255, 2048] + [2048 * k + d for k in range(1, 8) for d in (1, 2048)] + [16385]


@pytest.mark.parametrize("scheme", ["systematic", "stratified", "multinomial", "systematic_cutpoint"])
def test_every_number_of_slots_per_thread(pf, orc, scheme):
    for n in SIZES:
        rng = np.random.default_rng(n)
        one = np.zeros(n, np.float32)
        one[n // 3] = 0.5
        for w in (np.exp(rng.standard_normal(n)).astype(np.float32), one):
            ref = orc.resample_weights(w, pf.SCHEMES[scheme], 41, 1, 3)
            got = pf.resample(torch.from_numpy(w).cuda(), seed=41, filter_id=1, t=3, scheme=scheme)
            assert np.array_equal(got.cpu().numpy().view(np.uint32), ref), n
