"""k-means with points that have no finite distance: they belong to no centroid and
leave the gradient of the others as it is (the 256th row is the last of the
block's sums), and the loss is not finite."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [32, 256])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("N", [1, 300, 5000])
def test_points_without_a_centroid(oracle, k, bad, N):
    from paper_2202_10297_gb300 import adpar as A
    g = np.random.default_rng(N + k)
    X = g.normal(size=(N, 32)).astype(np.float32)
    C = g.normal(size=(k, 32)).astype(np.float32)
    rows = np.unique(g.integers(0, N, 3))
    X[rows, g.integers(0, 32, len(rows))] = bad
    out = A.adpar_kmeans_vjp(torch.from_numpy(X).cuda(), torch.from_numpy(C).cuda(), 1.0, want_argmin=True)
    keep = np.delete(np.arange(N), rows)
    got = out["Cbar"].cpu().numpy()
    if len(keep):
        _, arg, _, cbar = oracle.kmeans(X[keep].astype(np.float64), C.astype(np.float64))
        assert np.linalg.norm(got - cbar) <= 1e-5 * np.linalg.norm(cbar)
        np.testing.assert_array_equal(out["argmin"].cpu().numpy()[keep], arg)
    else:
        assert np.all(got == 0)
    assert not np.isfinite(out["loss"].item())
