"""The integer arithmetic of the * rule (top-aligned 64-bit products, the map's
reciprocal quotients) where it can go wrong: mantissas of all ones and of none,
subnormal factors and results, sizes around a vector, a block and a whole wave
of blocks."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(a, ybar, **kw):
    from paper_2202_10297_gb300 import adpar as A
    t = torch.from_numpy(a).cuda()
    out = A.adpar_vjp_reduce("mul", t, float(ybar), want_y=True, **kw)
    return out["abar"].cpu().numpy(), out["y"].cpu().numpy()[0]


def _product(a):
    """The product of a in [1/2, 2)^n to about 2^-100: a tree of two-term products."""
    hi, lo = a.astype(np.float64), np.zeros(len(a))
    while len(hi) > 1:
        if len(hi) % 2:
            hi, lo = np.append(hi, 1.0), np.append(lo, 0.0)
        x, y = hi[::2], hi[1::2]
        c = 134217729.0  # Dekker's split
        xh = c * x - (c * x - x)
        yh = c * y - (c * y - y)
        p = x * y
        e = ((xh * yh - p) + xh * (y - yh) + (x - xh) * yh) + (x - xh) * (y - yh)
        e += x * lo[1::2] + y * lo[::2]
        hi, lo = p + e, e - ((p + e) - p)
    return hi[0], lo[0]


# FP64: each of n factors below 2^-62, the quotient within 2^-50 of K / m, the
# numerator's two roundings 2^-52: 2^-49 in all for these n.  FP32: the
# numerator's rounding and one of the quotient, and one more of a subnormal.
@pytest.mark.parametrize("dt,rel,tiny", [(np.float64, 2.0 ** -49, 2.0 ** -1074), (np.float32, 2.0 ** -22, 2.0 ** -149)])
@pytest.mark.parametrize("ybar", [1.0, -1.9999998807907104, 2.0 ** -120])
def test_mantissa_edges_and_subnormals(dt, rel, tiny, ybar):
    eps = float(np.finfo(dt).eps)
    lo = float(np.finfo(dt).smallest_subnormal)
    big = 2.0 ** (1000 if dt == np.float64 else 120)
    vals = [1.0, 2.0 - eps, 1.0 + eps, -1.5, 2.0 - 2 * eps, 0.5 + eps / 2, -(1.0 - eps / 2), 4.0 / 3.0, 2.0 ** -30]
    a = np.array(vals + [lo * 5, 1 / big, big, big / 8, -3.0 * lo, big, big / 4], dtype=dt)
    prod = Fraction(1)
    for v in a:
        prod *= Fraction(float(v))
    got, y = _run(a, ybar)
    for v, g in zip(a, got):
        ref = prod / Fraction(float(v)) * Fraction(ybar)
        if abs(ref) >= Fraction(float(np.finfo(dt).max)):
            assert np.isinf(g) and (g > 0) == (ref > 0)
        else:
            assert abs(Fraction(float(g)) - ref) <= abs(ref) * Fraction(rel) + Fraction(tiny), (v, g, float(ref))
    assert abs(Fraction(float(y)) - prod) <= abs(prod) * Fraction(rel) + Fraction(tiny)


@pytest.mark.parametrize("dt,rel", [(np.float64, 2.0 ** -48), (np.float32, 2.0 ** -22)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 511, 513, 1027, 608 * 512 - 1, 608 * 512 + 1, 608 * 2048 + 5, 4 * 608 * 1024 + 7])
@pytest.mark.parametrize("accumulate", [False, True])
def test_sizes(dt, rel, n, accumulate):
    r = np.random.default_rng(n)
    # each factor adds at most 2^-62 to the product; the quotient is within 2^-50
    a = np.exp(r.uniform(-2.0 ** -10, 2.0 ** -10, n)).astype(dt)
    a[r.integers(0, n, max(1, n // 3))] *= -1
    ref = 1.25 * _product(a)[0] / a.astype(np.float64)
    init = np.full(n, 0.5, dtype=dt) if accumulate else None
    kw = {"accumulate": True, "abar": torch.from_numpy(init.copy()).cuda()} if accumulate else {}
    got, _ = _run(a, 1.25, **kw)
    if accumulate:
        assert np.all(np.abs(got - (0.5 + ref)) <= (np.abs(ref) + 1.0) * 2 * rel)
    else:
        assert np.all(np.abs(got - ref) <= np.abs(ref) * rel * (1 + n * 2.0 ** -14 * (dt == np.float64)))


# one cluster of 8 x 1024 threads up to 1 MB, three launches beyond
@pytest.mark.parametrize("dt", [np.float64, np.float32])
@pytest.mark.parametrize("over", [-1, 0, 1])
@pytest.mark.parametrize("zeros", [0, 1, 2])
def test_one_cluster_boundary(dt, over, zeros):
    from paper_2202_10297_gb300 import adpar as A
    n = (1 << 20) // np.dtype(dt).itemsize + over
    g = np.random.default_rng(n + zeros)
    a = np.exp(g.uniform(-2.0 ** -10, 2.0 ** -10, n)).astype(dt)
    pos = np.sort(g.choice(n, zeros, replace=False))
    nz = np.delete(a, pos)
    a[pos] = 0
    p = _product(nz)[0]
    out = A.adpar_vjp_reduce("mul", torch.from_numpy(a).cuda(), 1.25, want_y=True, want_aux=True)
    assert out["aux"].nzero == zeros and out["aux"].first_zero == (pos[0] if zeros else -1)
    rel = 2.0 ** -47 if dt == np.float64 else 2.0 ** -22
    got = out["abar"].cpu().numpy().astype(np.float64)
    ref = 1.25 * p / a.astype(np.float64) if zeros == 0 else np.zeros(n)
    if zeros == 1:
        ref[pos[0]] = 1.25 * p
    assert np.all(np.abs(got - ref) <= rel * np.abs(ref))
    assert A.adpar_workspace_status(out["work"]) == A.OK
    lg = A.adpar_vjp_reduce("mul", torch.from_numpy(a).cuda(), 1.25, logdomain=True)["abar"].cpu().numpy()
    assert np.array_equal(np.isfinite(lg), ref != 0)
