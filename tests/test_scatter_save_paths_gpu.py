"""scatter that keeps the overwritten values: by regions, by exchanges in one
region, by a load and a store per index (targets of 96 to 224 MB with few indices
per line; neighbouring indices), with indices out of range, against torch."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mb,frac", [(95, 8), (97, 2), (97, 4), (97, 8), (97, 16), (223, 4), (223, 16), (225, 4), (225, 16),
                                     (340, 2), (1, 2), (1, 300)])
@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("order", ["random", "sorted", "run"])
@pytest.mark.parametrize("itype", [torch.int32, torch.int64])
def test_paths(mb, frac, dt, order, itype):
    from paper_2202_10297_gb300 import adpar as A
    n = (mb << 20) // torch.empty(0, dtype=dt).element_size() + 5
    m = n // frac + 3
    g = torch.Generator(device="cuda").manual_seed(n)
    is_ = torch.randperm(n, generator=g, device="cuda")[:m] if order != "run" else torch.arange(7, 7 + m, device="cuda")
    if order == "sorted":
        is_ = is_.sort().values
    is_[m // 3] = -1
    is_[m // 2] = n
    ys, vs = torch.randn(n, generator=g, device="cuda", dtype=dt), torch.randn(m, generator=g, device="cuda", dtype=dt)
    ok = (is_ >= 0) & (is_ < n)
    want_saved = torch.where(ok, ys[is_.clamp(0, n - 1)], torch.zeros((), dtype=dt, device="cuda"))
    want = ys.clone()
    want[is_[ok]] = vs[ok]
    saved = torch.full_like(vs, 3.0)
    A.adpar_scatter(is_.to(itype), vs, ys, xs_saved=saved)
    assert torch.equal(ys, want) and torch.equal(saved, want_saved)
    ys2 = ys.clone()
    A.adpar_scatter(is_.to(itype), 2 * vs, ys2)
    want[is_[ok]] = 2 * vs[ok]
    assert torch.equal(ys2, want)
