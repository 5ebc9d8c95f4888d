"""The kernels' own reciprocals, quotients and square roots against IEEE division
and square root (numpy), bit for bit: every significand where one operand
decides, quotients beside the midpoints of two neighbours, the guards between
the paired forms and the compiler's operations, and for binary64 (integer
residuals) the whole range with zeros, subnormal numbers, infinities and NaN."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

RCP2, DIV2, SQRT2, SQRT1, QUOT2, IG2, IG2_WIDE, SCALE_R, SCALE_S, DIV64, SQRT64 = 0, 1, 2, 3, 4, 5, 6, 7, 8, 16, 17
N = 1 << 22


def _run(pf, op, a, b=None):
    b = np.ones_like(a) if b is None else b
    return pf.diag_arith(op, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()


def _same(got, ref, *operands):
    bits = np.uint32 if ref.dtype == np.float32 else np.uint64
    bad = (got.view(bits) != ref.view(bits)) & ~(np.isnan(got) & np.isnan(ref))
    i = np.flatnonzero(bad)[:4]
    assert not bad.any(), (int(bad.sum()), [o[i] for o in operands], got[i], ref[i])


def _f32(sig, exp):
    """(1 + sig 2^-23) 2^exp, the float32 of a 23-bit fraction and an exponent."""
    return ((np.asarray(exp) + 127).astype(np.uint32) << 23 | np.asarray(sig, np.uint32)).view(np.float32)


def _f64(sig, exp):
    return ((np.asarray(exp) + 1023).astype(np.uint64) << np.uint64(52) | np.asarray(sig, np.uint64)).view(np.float64)


def _pairs32(rng, n, lo, hi):
    """Random (a, b) with exponents in [lo, hi), half of them with a / b beside the midpoint of two
    neighbouring floats: a is b (q + half a unit) rounded."""
    b = _f32(rng.integers(0, 1 << 23, n), rng.integers(lo, hi, n))
    a = _f32(rng.integers(0, 1 << 23, n), rng.integers(lo, hi, n))
    q = 1.0 + (rng.integers(0, 1 << 23, n) + 0.5) * 2.0 ** -23
    mid = (b.astype(np.float64) * q).astype(np.float32)
    return np.where(np.arange(n) % 4 < 2, a, mid), b


def test_reciprocal_of_every_significand(pf):
    s = np.arange(1 << 23, dtype=np.uint32)
    for e in (0, -39, 41, -81):
        b = _f32(s, e)
        _same(_run(pf, RCP2, b), np.float32(1) / b, b)


@pytest.mark.parametrize("op", [SQRT2, SQRT1])
def test_root_of_every_significand(pf, op):
    s = np.arange(1 << 23, dtype=np.uint32)
    for e in (0, 1, -24, 5, -80, -81, 40):
        x = _f32(s, e)
        _same(_run(pf, op, x), np.sqrt(x), x)


def test_quotient_of_safe_operands(pf):
    for seed in range(6):
        a, b = _pairs32(np.random.default_rng(seed), N, -40, 40)
        _same(_run(pf, DIV2, a, b), a / b, a, b)


def test_quotient_of_the_weights_at_any_operands(pf):
    """Operands on both sides of 2^-40 and 2^40, zeros, subnormal, infinite, NaN."""
    rng = np.random.default_rng(9)
    a, b = _pairs32(rng, N, -44, 44)
    edge = np.array([2.0 ** -40, 2.0 ** 40], np.float32)
    edge = np.concatenate([edge, np.nextafter(edge, np.float32(0)), np.nextafter(edge, np.float32(np.inf))])
    odd = np.array([0.0, 1e-45, 1e-39, 1.1754944e-38, 3.4028235e38, np.inf, np.nan, 1e-30, 1e30], np.float32)
    pool = np.concatenate([edge, odd])
    for x in (a, b):
        at = rng.integers(0, N, N // 8)
        x[at] = rng.choice(pool, at.size)
    with np.errstate(all="ignore"):
        _same(_run(pf, QUOT2, a, b), a / b, a, b)


def test_quotient_of_the_gamma_draws(pf):
    """b: 0 or a multiple of 2^-32 below 2^32; G = d v^3, v in (0.04, 4), d from 1 to 2^60, and wider."""
    rng = np.random.default_rng(10)
    for op, lo, hi in ((IG2, -14, 66), (IG2_WIDE, -126, 127)):
        a, G = _pairs32(rng, N, -32, 32)
        a[rng.integers(0, N, N // 16)] = 0.0
        G = _f32(rng.integers(0, 1 << 23, N), rng.integers(lo, hi, N))
        with np.errstate(all="ignore"):
            _same(_run(pf, op, a, G), a / G, a, G)


def test_scale_of_the_state_draw(pf):
    """Variances on both sides of 2^-40 and 2^40."""
    rng = np.random.default_rng(11)
    for lo, hi in ((-44, -36), (-8, 8), (36, 44), (-62, 62)):
        a = _f32(rng.integers(0, 1 << 23, N), rng.integers(lo, hi, N))
        b = _f32(rng.integers(0, 1 << 23, N), rng.integers(lo, hi, N))
        for x in (a, b):
            x[rng.integers(0, N, N // 64)] = np.float32(2.0 ** -40)
            x[rng.integers(0, N, N // 64)] = np.float32(2.0 ** 40)
        r = np.float32(1) / (a + b)
        _same(_run(pf, SCALE_R, a, b), r, a, b)
        _same(_run(pf, SCALE_S, a, b), np.sqrt((a * b) * r), a, b)


def _odd64(rng, n):
    tiny, big = 2.2250738585072014e-308, 1.7976931348623157e308
    return rng.choice(np.array([0.0, -0.0, 5e-324, -5e-324, 1e-310, tiny, np.nextafter(tiny, 0), big, np.inf, -np.inf,
                                np.nan, 1.0, -1.0, 2.0 ** -1022, 2.0 ** 1023]), n)


def test_binary64_quotient(pf):
    for seed, (lo, hi) in enumerate([(-4, 4), (-1022, 1024), (-512, 512), (-1022, -960), (960, 1024)]):
        rng = np.random.default_rng(seed)
        sb = rng.integers(0, 1 << 52, N)
        b = _f64(sb, rng.integers(lo, hi, N))
        a = _f64(rng.integers(0, 1 << 52, N), rng.integers(lo, hi, N))
        # beside a midpoint: a = b (q + half a unit), its leading 53 bits
        q = (rng.integers(0, 1 << 26, N).astype(np.uint64) << np.uint64(27)) | np.uint64(1)  # q, 54 bits, odd
        hi64 = (sb.astype(np.uint64) | np.uint64(1 << 52)) >> np.uint64(26)
        near = _f64((hi64 * (q >> np.uint64(27))) & np.uint64((1 << 52) - 1), rng.integers(-3, 4, N))
        a = np.where(np.arange(N) % 3 == 0, near, a)
        a = np.where(rng.random(N) < 0.5, -a, a)
        at = rng.integers(0, N, N // 16)
        a[at] = _odd64(rng, at.size)
        at = rng.integers(0, N, N // 16)
        b[at] = _odd64(rng, at.size)
        with np.errstate(all="ignore"):
            _same(_run(pf, DIV64, a, b), a / b, a, b)
    # exact quotients and their neighbours
    rng = np.random.default_rng(20)
    b = _f64(rng.integers(0, 1 << 26, N) << 26, rng.integers(-3, 4, N))
    a = b * (1.0 + rng.integers(0, 1 << 25, N) * 2.0 ** -25)
    for d in (-np.inf, None, np.inf):
        x = a if d is None else np.nextafter(a, d)
        _same(_run(pf, DIV64, x, b), x / b, x, b)


def test_binary64_root(pf):
    for seed, (lo, hi) in enumerate([(-2, 2), (-1022, 1024), (-1022, -1000)]):
        rng = np.random.default_rng(seed)
        x = _f64(rng.integers(0, 1 << 52, N), rng.integers(lo, hi, N))
        at = rng.integers(0, N, N // 16)
        x[at] = _odd64(rng, at.size)
        with np.errstate(all="ignore"):
            _same(_run(pf, SQRT64, x), np.sqrt(x), x)
    # squares of 26-bit numbers and their neighbours; roots beside a midpoint
    rng = np.random.default_rng(21)
    r = rng.integers(1 << 25, 1 << 26, N).astype(np.float64)
    mid = (r + 0.5) * (1 + 2.0 ** -26)
    for x in (r * r, np.nextafter(r * r, 0), np.nextafter(r * r, np.inf), mid * mid):
        _same(_run(pf, SQRT64, x), np.sqrt(x), x)
