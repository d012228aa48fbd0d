"""FP32 min/max reduce_by_index where a thread takes four elements per step instead
of one (6 M elements) and where global words are read before their atomics (256
elements a bin), with ties and indices out of range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N = 6 << 20


@pytest.mark.parametrize("op", ["max", "min"])
@pytest.mark.parametrize("n,m", [(N - 1, 100), (N, 100), (N + 3, N // 256), (N + 2, N // 256 + 1), (N - 1, N // 256),
                                 (N + 1, 1 << 20)])
@pytest.mark.parametrize("itype", [np.int32, np.int64])
def test_long(oracle, op, n, m, itype):
    from paper_2202_10297_gb300 import adpar as A
    g = np.random.default_rng(n + m)
    vals = (np.round(g.normal(size=n) * 64) / 64).astype(np.float32)
    inds = g.integers(-1, m + 1, n).astype(itype)
    hsbar = g.normal(size=m).astype(np.float32)
    dev = lambda x: torch.from_numpy(x).cuda()
    vb, hs, arg = oracle.hist_vjp(op, vals, inds, m, hsbar)
    out = A.adpar_vjp_hist(op, dev(inds), m, dev(hsbar), vals=dev(vals), want_hs=True, want_argidx=True)
    np.testing.assert_array_equal(out["argidx"].cpu().numpy(), arg)
    np.testing.assert_array_equal(out["valsbar"].cpu().numpy(), vb)
    np.testing.assert_array_equal(out["hs"].cpu().numpy()[arg >= 0], hs[arg >= 0])
    acc = torch.full((n,), 2.0, device="cuda")
    A.adpar_vjp_hist(op, dev(inds), m, dev(hsbar), vals=dev(vals), valsbar=acc, accumulate=True)
    np.testing.assert_array_equal(acc.cpu().numpy(), (2.0 + vb).astype(np.float32))
