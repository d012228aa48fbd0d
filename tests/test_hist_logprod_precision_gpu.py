"""The products of reduce_by_index * over FP32 values are held as closely as by
63-bit mantissas, whose every factor cost at most 2^-62: bins of many equal
factors (whose errors all have one sign), of random ones, and arrays of more
than one chunk of 2^27 elements.  The record's FP64 mantissa adds its rounding,
2^-53."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
getcontext().prec = 60
LN2 = Decimal(2).ln()


def _rel(aux, counts):
    """The relative error of a bin's record against the product of v^k over counts = {v: k}."""
    exact = sum(Decimal(k) * abs(Decimal(float(v))).ln() for v, k in counts.items())
    got = abs(Decimal(float(aux["mant"]))).ln() + int(aux["exp2"]) * LN2
    return abs(float(got - exact))


# bins of each tier: a copy per lane, one per block, words in global memory
@pytest.mark.parametrize("bins", [[0, 63], [64, 8255], [8256, 20000]])
@pytest.mark.parametrize("bits", [0x3f83ffaa, 0x3f824077, 0x3f816f15, 0x3f333333, 0x7f000001, 0x00000003])
def test_equal_factors(bins, bits):
    from paper_2202_10297_gb300 import adpar as A
    v = np.array([bits], np.uint32).view(np.float32)[0]
    n, m = 1 << 21, 20001
    inds = torch.tensor(bins, dtype=torch.int32, device="cuda").repeat(n // 2)
    vals = torch.full((n,), float(v), device="cuda")
    aux = A.adpar_vjp_hist("mul", inds, m, torch.ones(m, device="cuda"), vals=vals, want_aux=True)["aux"]
    for b in bins:
        assert _rel(aux[b], {v: n // 2}) <= n // 2 * 2.0 ** -62 + 2.0 ** -53


@pytest.mark.parametrize("m", [40, 300, 9000])
def test_random_factors(m):
    from paper_2202_10297_gb300 import adpar as A
    g = np.random.default_rng(m)
    n = 64 * m
    vals = (np.exp(g.normal(0, 0.5, n)) * g.choice([-1.0, 1.0], n)).astype(np.float32)
    inds = g.permutation(np.arange(n) % m).astype(np.int64)
    dev = lambda x: torch.from_numpy(x).cuda()
    aux = A.adpar_vjp_hist("mul", dev(inds), m, torch.ones(m, device="cuda"), vals=dev(vals), want_aux=True)["aux"]
    for b in range(0, m, max(1, m // 40)):
        x = vals[inds == b]
        exact = sum(abs(Decimal(float(v))).ln() for v in x)
        got = abs(Decimal(float(aux["mant"][b]))).ln() + int(aux["exp2"][b]) * LN2
        assert abs(float(got - exact)) <= 64 * 2.0 ** -62 + 2.0 ** -53
        assert aux["sign"][b] == np.prod(np.sign(x))


@pytest.mark.parametrize("n", [(1 << 27) - 1, (1 << 27) + 1, (1 << 28) + 4099])
def test_chunks(n):
    """Bin i % 5 of element i, value by i % 7; bin 8191 + i % 5 beyond the shared tiers' first bins."""
    from paper_2202_10297_gb300 import adpar as A
    tbl = np.array([1.4, -0.7, 1.0312088, 3.0, -1.0000001, 0.33333334, 1e-30], np.float32)
    m = 9000
    i = torch.arange(n, device="cuda")
    base = torch.where(i % 70 < 35, 0, 8254)  # both sides of the shared tiers' end
    inds = (base + i % 5).to(torch.int32)
    vals = torch.from_numpy(tbl).cuda()[i % 7]
    del base
    zero = [n - 7, n - 7 - 70] if n > 1 << 27 else [3]
    for z in zero:
        vals[z] = 0
    out = A.adpar_vjp_hist("mul", inds, m, torch.ones(m, device="cuda"), vals=vals, want_aux=True, want_hs=True)
    aux = out["aux"]
    counts = {}
    for r in range(70):
        c = (n - r + 69) // 70
        b = (0 if r < 35 else 8254) + r % 5
        v = tbl[r % 7]
        c -= sum(1 for z in zero if z % 70 == r)
        counts.setdefault(b, {})
        counts[b][v] = counts[b].get(v, 0) + c
    for b, cn in counts.items():
        k = sum(cn.values())
        zs = [z for z in zero if (0 if z % 70 < 35 else 8254) + z % 5 == b]
        assert _rel(aux[b], cn) <= k * 2.0 ** -62 + 2.0 ** -53
        assert aux["sign"][b] == (-1) ** (sum(c for v, c in cn.items() if v < 0) % 2)
        assert aux["nzero"][b] == len(zs) and aux["first_zero"][b] == (min(zs) if zs else -1)
    assert aux["mant"][8000] == 0.5 and aux["exp2"][8000] == 1 and out["hs"][8000].item() == 1.0


def test_workspace_depends_on_the_bins_alone():
    from paper_2202_10297_gb300 import adpar as A
    sizes = {A.adpar_workspace_size(A.RULE_HIST, A.OP_MUL, A.F32, n, 1000) for n in (0, 1, 1 << 27, 1 << 33)}
    assert len(sizes) == 1
