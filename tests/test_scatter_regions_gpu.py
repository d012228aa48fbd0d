"""Scatter over a target larger than L2: taken in regions for random indices, in
one for local ones; the results are moves of values, so they are exact."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _indices(n, m, kind, itype):
    g = torch.Generator(device="cuda").manual_seed(n + m)
    is_ = torch.randperm(n, generator=g, device="cuda")[:m]
    if kind == "sorted":
        is_ = torch.sort(is_).values
    is_[::1001] = -1 - is_[::1001] // 7  # out of range, half below and half above
    is_[500::1001] = n + is_[500::1001] // 7
    is_[7] = n
    return is_.to(itype)


# 2^25 FP32 (2^24 FP64) elements are the first size in regions; 8 regions the most
@pytest.mark.parametrize("n", [1, 31, (1 << 25) - 1, (1 << 25) + 5, (1 << 26) + 33, (1 << 27) + 1])
@pytest.mark.parametrize("kind", ["random", "sorted"])
@pytest.mark.parametrize("dtype,itype", [(torch.float32, torch.int32), (torch.float64, torch.int64)])
def test_exact(n, kind, dtype, itype):
    from paper_2202_10297_gb300 import adpar as A
    if dtype == torch.float64:
        n = (n + 1) // 2
    m = max(1, min(n, n // 7 + 13))
    is_ = _indices(n, m, kind, itype) if n > 1000 else torch.arange(m, device="cuda").to(itype)
    ok = (is_ >= 0) & (is_ < n)
    k = is_[ok].long()
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda c: torch.randn(c, generator=g, device="cuda", dtype=dtype)
    xs, vs, ybar = rnd(n), rnd(m), rnd(n)
    ref = xs.clone()
    ref[k] = vs[ok]
    ys, saved = xs.clone(), torch.full((m,), 9.0, device="cuda", dtype=dtype)
    A.adpar_scatter(is_, vs, ys, xs_saved=saved)
    assert torch.equal(ys, ref)
    assert torch.equal(saved[ok], xs[k]) and not saved[~ok].any()
    y2 = xs.clone()
    A.adpar_scatter(is_, vs, y2)
    assert torch.equal(y2, ref)
    xref = ybar.clone()
    xref[k] = 0
    for acc in (False, True):
        yb = ybar.clone()
        vb = torch.full((m,), 3.0, device="cuda", dtype=dtype)
        y3 = ref.clone()
        kw = {"ys": y3, "xs_saved": saved} if acc else {}
        A.adpar_vjp_scatter(is_, yb, vsbar=vb, accumulate=acc, **kw)
        assert torch.equal(yb, xref)
        want = torch.full((m,), 3.0 if acc else 0.0, device="cuda", dtype=dtype)
        want[ok] += ybar[k]
        assert torch.equal(vb, want)
        if acc:
            assert torch.equal(y3, xs)
