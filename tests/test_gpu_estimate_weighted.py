"""Summaries of an adaptive filter over many blocks: seven threads of a block
store its sums and one of them announces the block, so the last block must find
all seven.  The fold's order is fixed: every reading of an unchanged state is
the same to the last bit."""
import pytest

from paper_1212_1639_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [4097, 8192, 300_001, 1 << 21])
def test_weighted_summaries_do_not_vary(pf, orc, n, prec):
    _, y = synth.local_level_series(31, 3)
    f = pf.Filter(n, seed=31, precision=prec, ess_frac=1e-9)  # never resamples: the weights stay uneven
    for v in y:
        f.step(v)
    first = f.estimate()
    for _ in range(200):
        assert f.estimate() == first
    if n <= 300_001:
        o = orc.Filter(orc.make_config(n, seed=31, scheme=1, precision=int(prec == "fp64"), ess_frac=1e-9))
        for v in y:
            o.step(v)
        e = o.estimate()
        for k in ("x_mean", "sigma2_mean", "tau2_mean", "log_marglik"):
            # binary64 sums of binary32 terms (a rounding of 2^-24 each) or of binary64 terms
            assert abs(first[k] - e[k]) <= (1e-5 if prec == "fp32" else 1e-12) * max(1.0, abs(e[k])), k
    f.close()
