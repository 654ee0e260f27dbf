"""The gradient chain on grids of one or a few cells in some direction.

Tiles take the shape of such grids.  Values as for the boxes; and a pass over a
section or a column may take no more than twice the time of a box of as many
cells (it has fewer faces; with one tile shape for all it took 3 to 13 times).
"""
import pytest
import test_gpu_chain_faces as faces

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(300, 1, 1), (1, 300, 1), (1, 1, 300), (40, 1, 20), (1, 40, 20), (33, 18, 1),
                                   (5, 2, 40), (2, 2, 100), (257, 2, 1), (2, 3, 1)])
@pytest.mark.parametrize("b", [1, 3])
def test_values(shape, b):
    faces.test_chain_faces_not_stored(shape, b, 0.2)


def test_time_by_shape():
    from paper_1812_03952_gb300 import trs
    b, n = 3, 64 * 64 * 64
    g = torch.Generator(device="cuda").manual_seed(1)
    k, lam, x, M = (torch.rand(m, generator=g, device="cuda", dtype=torch.float64) for m in
                    (n, n * b, n * b, n * 6 * b * b))

    def best(shape):
        A = trs.Matrix.synthetic_pattern(*shape, b, 0, [], [])
        times = []
        for _ in range(12):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            for _ in range(4):
                trs.chain_theta(A, k, M, lam, x, 0.3, 1.0)
            t1.record()
            torch.cuda.synchronize()
            times.append(t0.elapsed_time(t1))
        return min(times)

    box = best((64, 64, 64))
    for shape in ((n, 1, 1), (1, n, 1), (1, 1, n), (512, 512, 1), (512, 1, 512), (1, 512, 512)):
        assert best(shape) <= 2.0 * box, shape
