"""The vectorised scan around its chunk (32 rows), its batches of rows, its groups
of chunks and its blocks of columns, against the column-by-column definition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["add", "mul", "min", "max", "linrec"])
@pytest.mark.parametrize("dt,tol", [(np.float32, 1e-5), (np.float64, 1e-13)])
@pytest.mark.parametrize("n,d", [(1, 1), (3, 65), (31, 33), (32, 32), (33, 31), (37, 64), (32 * 32 * 8 + 5, 3),
                                 (32 * 32 + 1, 257)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_edges(oracle, op, dt, tol, n, d, accumulate):
    from paper_2202_10297_gb300 import adpar as A
    g = np.random.default_rng(n * 7 + d)
    a = (g.uniform(0.9, 1.0, (n, d)) if op in ("linrec", "mul") else g.normal(size=(n, d))).astype(dt)
    b, ya, yb = (g.normal(size=(n, d)).astype(dt) for _ in range(3))
    dev = lambda x: torch.from_numpy(x).cuda()
    w2 = op == "linrec"
    kw = {"b": dev(b), "ybar_b": dev(yb)} if w2 else {}
    if accumulate:
        kw.update(accumulate=True, abar=torch.ones((n, d), dtype=dev(a).dtype, device="cuda"))
        if w2:
            kw["bbar"] = torch.ones((n, d), dtype=dev(a).dtype, device="cuda")
    ab, bb, _ = A.adpar_vjp_scan_vec(op, dev(a), dev(ya), **kw)
    c = lambda x, j: np.ascontiguousarray(x[:, j], dtype=np.float64)
    ra, rb = np.zeros((n, d)), np.zeros((n, d))
    for j in range(d):
        r = oracle.scan_vjp(op, c(a, j), c(ya, j), c(b, j) if w2 else None, c(yb, j) if w2 else None)
        ra[:, j] = r[0]
        if w2:
            rb[:, j] = r[1]
    one = 1.0 if accumulate else 0.0
    for got, ref in ((ab, ra), (bb, rb))[:2 if w2 else 1]:
        x = got.cpu().numpy().astype(np.float64) - one
        assert np.linalg.norm(x - ref) <= tol * (np.linalg.norm(ref) + one * np.sqrt(ref.size))
