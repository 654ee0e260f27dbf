"""The outer product by runs of entries, at the edges of the run lengths.

Runs are of 4 * 256 / b^2 to 256 entries, by the number of entries over 1216.
Each value is one product: exact.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)


def _matrix(nx, ny, nz, b):
    from paper_1812_03952_gb300 import trs
    return trs.Matrix.synthetic_pattern(nx, ny, nz, b, 0, [], [])


@pytest.mark.parametrize("shape,b", [((1, 1, 1), 5), ((3, 3, 2), 4), ((16, 16, 8), 5), ((40, 40, 20), 5),
                                     ((40, 40, 21), 3), ((47, 40, 25), 2), ((47, 40, 25), 1), ((26, 40, 50), 4)])
def test_values(shape, b):
    from paper_1812_03952_gb300 import trs
    A = _matrix(*shape, b)
    rng = np.random.default_rng(4)
    lam, x = rng.standard_normal((2, A.n, b))
    rp, col = A.pattern()
    row = np.repeat(np.arange(A.n), np.diff(rp))
    dA = trs.outer_product(A, *(torch.from_numpy(v.reshape(-1)).cuda() for v in (lam, x)))
    ref = -(lam[row][:, :, None] * x[col][:, None, :])
    assert np.array_equal(dA.cpu().numpy().reshape(ref.shape), ref)


def test_time_of_a_small_matrix():
    """16x16x8, b = 5: a call on an idle GPU takes at most 2.7 us more than one on a
    single cell (4 with 256 entries for every block, 1 now); the best of five
    attempts, as it is the host that is timed."""
    import time
    from paper_1812_03952_gb300 import trs
    calls = []
    for shape in ((1, 1, 1), (16, 16, 8)):
        A = _matrix(*shape, 5)
        calls.append((A, torch.rand(A.N, device="cuda", dtype=torch.float64)))

    def attempt():
        times = [[], []]
        for k in range(600):
            A, v = calls[k % 2]
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            trs.outer_product(A, v, v)
            torch.cuda.synchronize()
            times[k % 2].append(1e6 * (time.perf_counter() - t0))
        one, small = (sorted(t)[75] for t in times)
        return small - one

    assert min(attempt() for _ in range(5)) <= 2.7
