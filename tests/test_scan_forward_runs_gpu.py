"""The forward linear-recurrence scan on per-thread runs: lengths around a tile
(128 runs), the L2 prefetch distance (152 tiles) and in place."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt,tile,tol", [(np.float32, 4096, 1e-5), (np.float64, 2048, 1e-13)])
@pytest.mark.parametrize("tiles,rest", [(0, 1), (0, 33), (1, -1), (1, 0), (1, 1), (2, 17), (33, 5), (153, 0), (154, 3)])
@pytest.mark.parametrize("in_place", [False, True])
def test_forward(oracle, dt, tile, tol, tiles, rest, in_place):
    from paper_2202_10297_gb300 import adpar as A
    n = tiles * tile + rest
    g = np.random.default_rng(n)
    a, b = g.uniform(0.9, 1.0, n).astype(dt), g.normal(size=n).astype(dt)
    z = np.zeros(n)
    _, _, ra, rb = oracle.scan_vjp("linrec", a, z, b, z)
    ta, tb = torch.from_numpy(a.copy()).cuda(), torch.from_numpy(b.copy()).cuda()
    kw = {"ys_a": ta, "ys_b": tb} if in_place else {}
    ya, yb, work = A.adpar_scan("linrec", ta, b=tb, **kw)
    assert A.adpar_workspace_status(work) == A.OK
    tiny = float(np.finfo(dt).tiny)
    for got, ref in ((ya, ra), (yb, rb)):
        x = got.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(x - ref) <= tol * np.linalg.norm(ref) + tiny * n
