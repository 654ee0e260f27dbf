"""The ILU sweeps of scalar rows (b = 1) kept in the tail, against the oracle.

Rows of a few to a few hundred entries: at most 32 (a warp sums), more (every
warp takes part).  1e-11 in FP64 and 1e-4 in FP32, as for the other applications.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("n,groups,reach", [(300, 2, 3), (300, 2, 29), (300, 2, 31), (300, 3, 22), (300, 3, 300),
                                            (700, 5, 700)])
def test_application(oracle, n, groups, reach):
    """Every two rows of different groups at most reach apart are coupled: rows of
    up to about 2 reach (1 - 1 / groups) + 1 entries."""
    from paper_1812_03952_gb300 import trs
    rng = np.random.default_rng(reach)
    i, j = (v.ravel() for v in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
    ok = (i == j) | ((abs(i - j) <= reach) & (i % groups != j % groups))
    i, j = i[ok], j[ok].astype(np.int32)
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, i + 1, 1)
    rp = np.cumsum(rp)
    val = np.where(i == j, 1.5 * np.diff(rp)[i], -rng.random(i.size))
    A = trs.Matrix.from_bsr(rp, j, val, 1, None)
    Ao = oracle.BSR(n, 1, rp, j, val.reshape(-1, 1, 1))
    v = rng.standard_normal(n)
    want = oracle.CPR(Ao).apply(v)
    for precision, tol in (("fp64", 1e-11), ("fp32", 1e-4)):
        got = trs.CPR(A, precision=precision).apply(torch.from_numpy(v).cuda()).cpu().numpy()
        assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
