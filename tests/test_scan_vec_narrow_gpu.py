"""The vectorised scan where threads run over (chunk, column) pairs (fewer than
1024 columns and more blocks of them than SMs: 152 on a GB300) and where a column
block's chunks form 1, 2, 8, 9 or 32 groups, against the column-by-column definition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["add", "mul", "max", "linrec"])
@pytest.mark.parametrize("dt,tol", [(np.float32, 1e-5), (np.float64, 1e-13)])
@pytest.mark.parametrize("n,d", [(152 * 32, 1), (152 * 32 + 1, 1), (153 * 32 + 5, 7), (8 * 32, 33), (8 * 32 + 1, 33),
                                 (63 * 32 + 31, 64), (64 * 32 + 1, 40), (39 * 32 - 7, 1023), (39 * 32 - 7, 1024),
                                 (260 * 32, 255), (1100 * 32 + 3, 2)])
def test_narrow(oracle, op, dt, tol, n, d):
    from paper_2202_10297_gb300 import adpar as A
    g = np.random.default_rng(n * 7 + d)
    a = (g.uniform(0.9, 1.0, (n, d)) if op in ("linrec", "mul") else g.normal(size=(n, d))).astype(dt)
    b, ya, yb = (g.normal(size=(n, d)).astype(dt) for _ in range(3))
    dev = lambda x: torch.from_numpy(x).cuda()
    w2 = op == "linrec"
    kw = {"b": dev(b), "ybar_b": dev(yb)} if w2 else {}
    ab, bb, _ = A.adpar_vjp_scan_vec(op, dev(a), dev(ya), **kw)
    ab, bb = ab.cpu().numpy(), bb.cpu().numpy() if w2 else None
    c = lambda x, j: np.ascontiguousarray(x[:, j], dtype=np.float64)
    for j in range(0, d, max(1, d // 16)):
        r = oracle.scan_vjp(op, c(a, j), c(ya, j), c(b, j) if w2 else None, c(yb, j) if w2 else None)
        for got, ref in ((ab, r[0]), (bb, r[1]))[:2 if w2 else 1]:
            x = got[:, j].astype(np.float64)
            assert np.linalg.norm(x - ref) <= tol * np.linalg.norm(ref)
