"""The general reduce_by_index rule around its tile sizes and on both sides of the
large-tile rule (2^21 elements), and the forward operator on its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _close(x, ref, tol):
    x = x.cpu().numpy()
    tiny = float(np.finfo(x.dtype).tiny)  # long products leave the type's range
    return np.linalg.norm(x.astype(np.float64) - ref) <= tol * np.linalg.norm(ref) + tiny * len(ref)


def _case(n, m, dt, it, seed):
    g = np.random.default_rng(seed)
    inds = (m * g.random(n) ** 3).astype(it)  # skewed to the low bins
    bad = g.random(n) < 0.01
    inds[bad] = g.integers(0, 2, int(bad.sum())) * (m + 1) - 1  # -1 or m
    a = g.uniform(0.9, 1.0, n).astype(dt)
    return (a, g.normal(size=n).astype(dt), inds, g.normal(size=m).astype(dt), g.normal(size=m).astype(dt))


@pytest.mark.parametrize("op", ["linrec", "max"])
@pytest.mark.parametrize("dt,it,tol", [(np.float32, np.int32, 1e-5), (np.float64, np.int64, 1e-13)])
@pytest.mark.parametrize("n,m", [(1, 1), (2047, 5), (2048, 257), (2049, 70000), ((1 << 21) - 1, 300),
                                 (1 << 21, 65536), ((1 << 21) + 5119, 1 << 17), (304 * 5120 * 2 + 3, 65537)])
def test_vjp_and_forward(oracle, op, dt, it, tol, n, m):
    from paper_2202_10297_gb300 import adpar as A
    a, b, inds, ha, hb = _case(n, m, dt, it, n + m)
    # unaligned caller arrays: no alignment is required of them
    dev = lambda x: torch.from_numpy(np.concatenate([x[:1], x])).cuda()[1:]
    w2 = op == "linrec"
    kw = {"b": dev(b), "hsbar_b": dev(hb)} if w2 else {}
    ab, bb, hs_a, hs_b = A.adpar_vjp_hist_general(op, dev(a), dev(inds), m, dev(ha), want_hs=True, **kw)
    okw = {"b": b, "hsbar_b": hb} if w2 else {}
    rab, rbb, rha, rhb = oracle.hist_general_vjp(op, a, inds, m, ha, **okw)
    fa, fb = A.adpar_hist_general(op, dev(a), dev(inds), m, b=dev(b) if w2 else None)
    if not w2:
        assert torch.equal(ab.cpu(), torch.from_numpy(rab.astype(dt)))
        assert torch.equal(hs_a.cpu(), torch.from_numpy(rha.astype(dt))) and torch.equal(fa, hs_a) and fb is None
        return
    for got, ref in ((ab, rab), (bb, rbb), (hs_a, rha), (hs_b, rhb), (fa, rha), (fb, rhb)):
        assert _close(got, ref, tol)


def test_forward_arguments():
    from paper_2202_10297_gb300 import adpar as A
    e = torch.empty(0, device="cuda")
    ha, hb = A.adpar_hist_general("linrec", e, torch.empty(0, dtype=torch.int32, device="cuda"), 3, b=e)
    assert ha.tolist() == [1.0] * 3 and hb.tolist() == [0.0] * 3
    ha, hb = A.adpar_hist_general("linrec", torch.ones(9, device="cuda"), torch.full((9,), 5, device="cuda"), 0,
                                  b=torch.ones(9, device="cuda"))
    assert ha.numel() == 0 and hb.numel() == 0
    with pytest.raises(A.AdparError):
        A.adpar_hist_general("linrec", torch.ones(9, device="cuda"), torch.zeros(9, dtype=torch.int32, device="cuda"),
                             2)  # b is missing
