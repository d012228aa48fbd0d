"""* over factors whose products are exact: the result is that product, bit for
bit, however many threads hold the neutral element and however the blocks'
states are combined (one cluster, a grid, a batch)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# one cluster up to 1 MB (131072 FP64 values), then a grid of up to 608 blocks
@pytest.mark.parametrize("n", [1, 2, 3, 33, 8193, 65536, 131072, 131073, 1000003, 1 << 23])
@pytest.mark.parametrize("dt", [np.float64, np.float32])
def test_reduce_of_exact_products(n, dt):
    from paper_2202_10297_gb300 import adpar as A
    g = np.random.default_rng(n)
    e = np.zeros(n, dtype=np.int64)  # powers of two that cancel over the whole array
    e[:n // 2] = g.integers(-120, 121, n // 2)
    e[n // 2:n // 2 * 2] = -e[:n // 2]
    g.shuffle(e)
    a = np.ldexp(1.0, e) * g.choice([-1.0, 1.0], n)
    k = min(n, 5)
    a[g.choice(n, k, replace=False)] *= 1.5
    want = np.prod(np.sign(a)) * 1.5 ** k
    a = a.astype(dt)
    out = A.adpar_vjp_reduce("mul", torch.from_numpy(a).cuda(), 1.0, want_y=True, want_aux=True)
    assert out["y"].item() == want
    m, x = np.frexp(want)
    assert out["aux"].mant == m and out["aux"].exp2 == x
    y, _ = A.adpar_reduce("mul", torch.from_numpy(a).cuda())
    assert y.item() == want


@pytest.mark.parametrize("n", [1, 257, 8192, 16385, 300001])
def test_batch_of_exact_products(n):
    from paper_2202_10297_gb300.batch import Batch
    dev = lambda x: torch.from_numpy(x).cuda()
    x = np.ones(n)
    x[n // 2] = -1.5
    z = np.zeros(n)
    B = Batch([{"x": dev(x), "a": dev(z), "b": dev(z), "ybar_a": dev(z), "ybar_b": dev(z), "aux": True}])
    B.run()
    r = B.aux_records()[0]
    assert (r["mant"], r["exp2"], r["sign"]) == (-0.75, 1, -1)


# the only zero's adjoint 1 + 2^-14 + 2^-30 is not an FP32 value: it is added to
# the accumulated -(1 + 2^-14) before the sum is rounded
@pytest.mark.parametrize("n", [3, 4, 7, 4096, 300001])
@pytest.mark.parametrize("at", [0, -1])
def test_zero_adjoint_joins_the_accumulated_value(n, at):
    from paper_2202_10297_gb300 import adpar as A
    a = np.ones(n, np.float32)
    a[1] = 1 + 2.0 ** -15
    a[at] = 0
    rest = 1 + 2.0 ** -15
    init = torch.full((n,), 3.0, device="cuda")
    init[at] = -(1 + 2.0 ** -14)
    ybar = torch.tensor([1 + 2.0 ** -15], device="cuda")
    out = A.adpar_vjp_reduce("mul", torch.from_numpy(a).cuda(), ybar, abar=init, accumulate=True)["abar"].cpu()
    assert out[at].item() == rest * rest - (1 + 2.0 ** -14) == 2.0 ** -30
    keep = torch.ones(n, dtype=torch.bool)
    keep[at] = False
    assert torch.all(out[keep] == 3.0)
