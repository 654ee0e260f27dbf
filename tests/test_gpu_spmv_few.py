"""y = alpha A x + beta y around the line between the form with a thread per cell
and block row (few rows) and the form with a thread per cell, against the oracle.

A row sums at most 7 b terms (b (perforations + 1) for a well), each product and
addition within 2^-53, so 2 (terms + 4) 2^-53 of the sum of the absolute values
bounds the difference of two orders of it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

# two warps per quarter of an SM: 1216 warps of 32 cells, b of them per cell, and b per well
LINE = {2: (38, 32, 16), 3: (30, 27, 16), 4: (38, 32, 8), 5: (25, 31, 10)}


@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-1.0, 1.0), (0.5, -2.0)])
@pytest.mark.parametrize("b,shape,pairs", [(2, (1, 1, 1), 0), (5, (9, 7, 5), 2), (3, (40, 5, 3), 1)] + [
    (b, (nx + d, ny, nz), 1) for b, (nx, ny, nz) in LINE.items() for d in (-1, 0, 1)])
def test_spmv_few_rows(oracle, synth, b, shape, pairs, alpha, beta):
    from paper_1812_03952_gb300 import trs
    s = synth.small_system(nx=shape[0], ny=shape[1], nz=shape[2], b=b, seed=7, n_pairs=pairs)
    ds = trs.DeviceSystem(s)
    ds.assemble()
    Ao = oracle.assemble(s)
    rng = np.random.default_rng(8)
    x, y0 = rng.standard_normal((2, s.n_unknowns))
    y = torch.from_numpy(y0.copy()).cuda()
    ds.A.spmv(torch.from_numpy(x).cuda(), y, alpha=alpha, beta=beta)
    ref = alpha * oracle.spmv(Ao, x) + beta * y0
    rp = np.asarray(Ao.rp)
    mag = abs(alpha) * oracle.spmv(oracle.BSR(len(rp) - 1, b, rp, Ao.col, np.abs(Ao.val)), np.abs(x)) + abs(beta * y0)
    terms = np.repeat(np.diff(rp) * b, b)
    assert np.all(np.abs(y.cpu().numpy() - ref) <= 2 * (terms + 4) * 2.0**-53 * mag)
