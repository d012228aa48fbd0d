"""reduce_by_index * over FP32 values as sums of logarithms: bins on both sides
of the tier boundaries (64 bins with a copy per lane, 8256 in shared memory, the
rest in global memory), lengths around a vector, a block and a wave of blocks,
powers of two, subnormals, zeros and bins that hold every element."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(oracle, vals, inds, m, hsbar, accumulate=False):
    from paper_2202_10297_gb300 import adpar as A
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    ref = oracle.hist_prod_vjp(vals, inds, m, hsbar)
    kw = {}
    if accumulate:
        kw = {"accumulate": True, "valsbar": torch.full((len(vals),), 0.5, device="cuda")}
    out = A.adpar_vjp_hist("mul", dev(inds), m, dev(hsbar), vals=dev(vals), want_hs=True, want_aux=True, **kw)
    aux = out["aux"]
    np.testing.assert_array_equal(aux["nzero"], ref["nzero"])
    np.testing.assert_array_equal(aux["first_zero"], ref["first_zero"])
    np.testing.assert_array_equal(aux["sign"], ref["signnz"])
    # each logarithm within 2^-54.4 (the sum below n 2^-54) and its FP64 form; ln 2 < 1
    err = np.abs(aux["log_abs_nz"] - ref["lognz"])
    assert np.all(err <= len(vals) * 2.0 ** -54 + 2.0 ** -51 * np.maximum(1, np.abs(ref["lognz"])))
    # the factor's rounding, the quotient's, and 2^-25 for what the sums leave
    got = out["valsbar"].cpu().numpy().astype(np.float64)
    r = ref["valsbar"]
    fin = np.abs(r) < float(np.finfo(np.float32).max)
    base = 0.5 if accumulate else 0.0
    slack = 2.0 ** -22 * np.abs(r) + 2.0 ** -149 + (2.0 ** -24 * (np.abs(r) + 0.5) if accumulate else 0.0)
    assert np.all(np.abs(got - (base + r))[fin] <= slack[fin])
    assert np.all(np.isinf(got[~fin]))


@pytest.mark.parametrize("m", [1, 2, 63, 64, 65, 8255, 8256, 8257, 20000])
@pytest.mark.parametrize("n", [1, 5, 4095, 4097, 30011])
@pytest.mark.parametrize("itype", [np.int32, np.int64])
def test_tiers_and_sizes(oracle, n, m, itype):
    g = np.random.default_rng(n * 31 + m)
    vals = np.exp(g.normal(0, 0.01, n)).astype(np.float32) * g.choice([-1, 1], n).astype(np.float32)
    vals[g.integers(0, n, 2)] = 0
    inds = g.integers(-1, m + 1, n)
    inds[g.random(n) < 0.3] = g.integers(max(0, m - 3), m)  # and a crowded bin near the end
    hsbar = g.normal(size=m).astype(np.float32)
    hsbar[g.integers(0, m)] = 0
    _check(oracle, vals, inds.astype(itype), m, hsbar)


@pytest.mark.parametrize("n,m", [(152 * 4096 + 3, 100), (2 * 152 * 4096 + 4093, 70000)])
def test_waves_and_accumulate(oracle, n, m):
    g = np.random.default_rng(m)
    vals = np.exp(g.normal(0, 0.002, n)).astype(np.float32)
    inds = (m * g.random(n) ** 6).astype(np.int32)  # skewed to the low bins
    _check(oracle, vals, inds, m, g.normal(size=m).astype(np.float32), accumulate=True)


def test_exact_factors(oracle):
    """Powers of two (exact logarithms) over the whole exponent range, subnormals
    among them: the product of each bin is exactly representable."""
    g = np.random.default_rng(3)
    n, m = 4000, 9000
    vals = np.exp2(g.integers(-149, 128, n).astype(np.float64)).astype(np.float32)
    vals[::3] = np.float32(1.5) * np.exp2(g.integers(-140, 120, len(vals[::3])).astype(np.float64)).astype(np.float32)
    inds = np.repeat(np.arange(n // 2), 2).astype(np.int32) * 4
    _check(oracle, vals, inds, m, np.ones(m, np.float32))
