"""The values of reduce_by_index * over FP32: hs itself, from the adjoint call and
from the forward operator, against exact products rounded once (subnormal and
overflowing ones too), with signs, zeros and empty bins, in the bins of every
tier; the block's shared words wrap both ways."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

M = 9000
TIERS = {"hot": 0, "block": 70, "global": 8300}


def _round(x):
    """x (a Fraction) to FP32, to nearest."""
    if x == 0:
        return np.float32(0)
    s, x = (-1 if x < 0 else 1), abs(x)
    e = x.numerator.bit_length() - x.denominator.bit_length()
    if Fraction(2) ** e > x:
        e -= 1
    ulp = Fraction(2) ** (max(e, -126) - 23)
    r = round(x / ulp) * ulp
    return np.float32(s * np.inf) if r >= Fraction(2) ** 128 else np.float32(s * float(r))


def _run(bins):
    """hs of {bin: [factors]} by both entry points, the elements in a random order."""
    from paper_2202_10297_gb300 import adpar as A
    inds = np.concatenate([np.full(len(f), b) for b, f in bins.items()]).astype(np.int32)
    vals = np.concatenate([np.asarray(f, np.float32) for f in bins.values()])
    p = np.random.default_rng(len(vals)).permutation(len(vals))
    i, v = torch.from_numpy(inds[p]).cuda(), torch.from_numpy(vals[p]).cuda()
    hs, _ = A.adpar_hist("mul", v, i, M)
    out = A.adpar_vjp_hist("mul", i, M, torch.ones(M, device="cuda"), vals=v, want_hs=True, want_aux=True)
    assert torch.equal(hs, out["hs"])
    assert hs[M - 1].item() == 1.0  # empty
    return hs.cpu().numpy(), out["aux"]


def _check(bins):
    hs, aux = _run(bins)
    for b, f in bins.items():
        exact = Fraction(1)
        for x in f:
            exact *= Fraction(float(np.float32(x)))
        want = _round(exact)
        # a product within 2^-50 of a tie may go either way
        near = {want, _round(exact * (1 + Fraction(1, 2 ** 50))), _round(exact * (1 - Fraction(1, 2 ** 50)))}
        assert hs[b] in near, (b, hs[b], want)
        assert aux["sign"][b] == np.prod(np.sign([x for x in f if x != 0]))


@pytest.mark.parametrize("base", TIERS.values(), ids=TIERS)
def test_products(base):
    g = np.random.default_rng(base)
    bins = {}
    for k in range(40):
        f = np.exp(g.normal(0, 1 + k % 5, g.integers(1, 30))).astype(np.float32) 
        f *= g.choice([-1, 1], len(f)).astype(np.float32)
        if k % 10 == 9:
            f[g.integers(0, len(f))] = 0
        bins[base + k] = f
    _check(bins)


@pytest.mark.parametrize("base", TIERS.values(), ids=TIERS)
def test_subnormal_and_overflowing_products_round_once(base):
    up, dn = 1 + 2.0 ** -23, 1 - 2.0 ** -24
    tiny = [up, dn, dn, 3 * 2.0 ** -75, 2.0 ** -75]  # 1.5 * 2^-149, less a little: one unit, not two
    bins = {base: tiny, base + 1: tiny[:3] + [-7 * 2.0 ** -70, 2.0 ** -80], base + 2: [2.0 ** -75, 2.0 ** -75],
            base + 3: [2.0 ** -75, up, 2.0 ** -75], base + 4: [2.0 ** -74, 2.0 ** -77], base + 5: [2.0 ** 64, 2.0 ** 64],
            base + 6: [2.0 ** 64, -dn * 2.0 ** 64], base + 7: [2.0 ** -126, dn], base + 8: [-(2.0 ** -149)],
            base + 9: [float(np.finfo(np.float32).max)], base + 10: [2.0 ** -126, 1 - 2.0 ** -23]}
    _check(bins)


# whole parts far from 0 in a crowded bin: w2 (and the carries from the fraction
# words) run up and down, with an odd and an even number of negative factors
@pytest.mark.parametrize("base", TIERS.values(), ids=TIERS)
@pytest.mark.parametrize("kind", ["up", "down", "both"])
def test_whole_parts(base, kind):
    g = np.random.default_rng(base)
    bins = {}
    for k in range(4):
        hi = (1.9999999 * 2.0 ** g.integers(120, 128, 400)).astype(np.float32)
        lo = (1.0000001 * 2.0 ** -g.integers(120, 127, 400).astype(np.float64)).astype(np.float32)
        sub = np.exp2(-g.integers(140, 150, 400).astype(np.float64)).astype(np.float32)
        f = {"up": hi, "down": np.concatenate([lo, sub]), "both": np.concatenate([hi, sub, lo])}[kind]
        s = g.choice([-1.0, 1.0], len(f)).astype(np.float32)
        if (np.count_nonzero(s < 0) + k) % 2:
            s[0] = -s[0]
        bins[base + k] = f * s
    _, aux = _run(bins)
    for k in range(4):
        f = bins[base + k]
        assert aux["sign"][base + k] == (1 if k % 2 == 0 else -1)
        exact = Fraction(1)
        for x in f:
            exact *= abs(Fraction(float(x)))
        got = Fraction(abs(float(aux["mant"][base + k]))) * Fraction(2) ** int(aux["exp2"][base + k])
        assert abs(got / exact - 1) <= len(f) * Fraction(1, 2 ** 62) + Fraction(1, 2 ** 53)
