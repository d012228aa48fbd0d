"""FP32 min/max reduce_by_index on both sides of the rule that reads a global word
before its atomic (64 elements per bin), with bins in shared and global memory,
ties, and lengths around a vector and a block."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["max", "min"])
@pytest.mark.parametrize("n,m", [(1, 3), (3, 1), (5, 9000), (2047, 31), (2049, 8193), (64 * 12000, 12000),
                                 (64 * 12000 - 1, 12000), (64 * 20011 + 3, 20011)])
@pytest.mark.parametrize("itype", [np.int32, np.int64])
def test_paths(oracle, op, n, m, itype):
    from paper_2202_10297_gb300 import adpar as A
    g = np.random.default_rng(n + m)
    vals = (np.round(g.normal(size=n) * 8) / 8).astype(np.float32)  # ties; -0.0 and 0.0 among them
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
