"""The residual's split of the rows over a fixed grid of 1216 blocks of 256.

Sizes at the edges of its ranges: a quarter of a round (77,824 rows), two and
eight rounds (622,592 and 2,490,368).  A row's sum runs in the product's order,
so r is b - A x but for its own rounding: 8 * 2^-53 of its size and of the
product's.  The norm adds squares in a fixed order over at most a few hundred
terms per thread and a tree: 1e-12.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)


def _system(nx, ny, nz, b):
    from paper_1812_03952_gb300 import trs
    n = nx * ny * nz
    g = torch.Generator(device="cuda").manual_seed(n + b)
    draw = lambda *s: torch.rand(s, generator=g, device="cuda", dtype=torch.float64)   # noqa: E731
    A = trs.Matrix.synthetic_pattern(nx, ny, nz, b, 0, [], [])
    none = draw(1)
    A.assemble(0.5 + draw(n), draw(n * 6 * b * b), draw(n * b * b), none, none, 0.7, 1.0)
    return A, draw(n * b) - 0.5, draw(n * b)


@pytest.mark.parametrize("n,b", [(31, 1), (77824, 1), (77825, 1), (311297, 1), (622592, 1), (622593, 1), (2490368, 1),
                                 (2490369, 1), (33, 5), (77825, 5), (622593, 5), (5000, 3)])
def test_values(n, b):
    from paper_1812_03952_gb300 import trs
    A, x, rhs = _system(n, 1, 1, b)
    r = torch.full_like(x, float("nan"))
    nrm = trs.residual_norm_noalloc(A, x, rhs, r)
    y = A.spmv(x)
    assert bool(((r - (rhs - y)).abs() <= 8 * 2.0**-53 * (rhs.abs() + y.abs())).all())
    ref = float(torch.linalg.vector_norm(r))
    assert abs(nrm - ref) <= 1e-12 * ref


@pytest.mark.parametrize("shape", [(80, 80, 20), (104, 100, 32)])
def test_time(shape):
    """A call takes the product's time, the host's wait (30 to 40 us here) and the
    reduction; with rows dealt out by the warp it took 83 and 118 us more than it."""
    from paper_1812_03952_gb300 import trs
    A, x, rhs = _system(*shape, 5)
    r, y = torch.empty_like(x), torch.empty_like(x)

    def best(f, many):
        times = []
        for _ in range(30):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(many):
                f()
            t1.record()
            torch.cuda.synchronize()
            times.append(1e3 * t0.elapsed_time(t1) / many)
        return min(times)

    product = best(lambda: A.spmv(x, y), 10)
    assert best(lambda: trs.residual_norm_noalloc(A, x, rhs, r), 1) <= 1.15 * product + 60.0
