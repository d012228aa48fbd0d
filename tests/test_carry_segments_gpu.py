"""The tile carries of the linear recurrence in segments of 512 tiles: numbers of
tiles on both sides of a segment, and of 32 segments (a lane's share of the fold).
Coefficients of +-1 and small integers: every value is exact in FP64, so the
carries of all tiles count and the results are equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [511, 512, 513, 1024, 1025, 512 * 33 + 1])
def test_vjp_across_segments(oracle, tiles):
    from paper_2202_10297_gb300 import adpar as A
    n = tiles * 2048 - 5  # FP64 tiles of 128 runs of 16
    g = np.random.default_rng(tiles)
    a = g.choice([-1.0, 1.0], n, p=[0.001, 0.999])
    b, ya, yb = (g.integers(-2, 3, n).astype(np.float64) for _ in range(3))
    dev = lambda x: torch.from_numpy(x).cuda()
    ab, bb, _ = A.adpar_vjp_scan("linrec", dev(a), dev(ya), b=dev(b), ybar_b=dev(yb))
    ra, rb, _, _ = oracle.scan_vjp("linrec", a, ya, b, yb)
    assert max(np.abs(ra).max(), np.abs(rb).max()) < 2.0 ** 52
    np.testing.assert_array_equal(ab.cpu().numpy(), ra)
    np.testing.assert_array_equal(bb.cpu().numpy(), rb)


@pytest.mark.parametrize("tiles", [512, 513, 1025, 4096, 4097])
def test_fp32_across_segments(oracle, tiles):
    from paper_2202_10297_gb300 import adpar as A
    n = tiles * 4096 - 5  # FP32 tiles of 128 runs of 32
    g = np.random.default_rng(tiles)
    a = g.choice([-1.0, 1.0], n, p=[0.4, 0.6])  # sums stay below 2^24: exact in FP32
    b, ya, yb = (g.integers(-1, 2, n).astype(np.float64) for _ in range(3))
    f = lambda x: torch.from_numpy(x.astype(np.float32)).cuda()
    ab, bb, _ = A.adpar_vjp_scan("linrec", f(a), f(ya), b=f(b), ybar_b=f(yb))
    ra, rb, _, _ = oracle.scan_vjp("linrec", a, ya, b, yb)
    # bbar is a signed sum of integers; abar adds a product of two such sums, rounded
    np.testing.assert_array_equal(bb.cpu().numpy(), rb)
    assert np.all(np.abs(ab.cpu().numpy() - ra) <= 2.0 ** -22 * (np.abs(ra) + 2.0 ** 24))
