"""The V-cycle where many rows of the finest level are kept in the tail.

A 7-point matrix given without grid dimensions, or with those of its lowest
layer only, has the entries of the same matrix with its grid in the same order,
so the levels are the same and each row's ordered sum is too: 1e-13, and 1e-5 in
FP32, leave room for the zero terms of absent slots only.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)


def _bsr(nx, ny, nz):
    rng = np.random.default_rng(nx * ny * nz)
    n = nx * ny * nz
    idx = np.arange(n).reshape(nz, ny, nx)
    ij = [(idx.ravel(), idx.ravel())]
    for axis in range(3):
        lo, up = idx.take(range(idx.shape[axis] - 1), axis).ravel(), idx.take(range(1, idx.shape[axis]), axis).ravel()
        ij += [(lo, up), (up, lo)]
    i, j = (np.concatenate(v) for v in zip(*ij))
    order = np.lexsort((j, i))
    i, j = i[order], j[order]
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, i + 1, 1)
    v = np.where(i == j, 7.5, -0.5 - rng.random(i.size))
    return np.cumsum(rp), j.astype(np.int32), v


def _cpr(shape, grid, precision):
    from paper_1812_03952_gb300 import trs
    rp, col, val = _bsr(*shape)
    A = trs.Matrix.from_bsr(rp, col, val, 1, grid)
    return A, trs.CPR(A, precision=precision)


# 1872 rows (13,104 entries at most): a warp each; 18,000 rows: a thread each
@pytest.mark.parametrize("shape", [(13, 12, 12), (30, 30, 20)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("fp32", 1e-5)])
def test_same_as_with_grid(shape, precision, tol):
    r = torch.from_numpy(np.random.default_rng(1).standard_normal(int(np.prod(shape)))).cuda()
    ref = None
    for grid in (shape, None, (shape[0], shape[1], 1)):
        e = _cpr(shape, grid, precision)[1].vcycle(r)
        ref = e if ref is None else ref
        assert float((e - ref).norm()) <= tol * float(ref.norm())


def test_time():
    """Not more than 1.4 times the V-cycle with the grid (1.9 with a warp per row)."""
    r = torch.rand(18000, device="cuda", dtype=torch.float64)

    def best(grid):
        A, M = _cpr((30, 30, 20), grid, "fp64")
        times = []
        for _ in range(30):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(20):
                M.vcycle(r)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        return min(times)

    assert best(None) <= 1.4 * best((30, 30, 20))
