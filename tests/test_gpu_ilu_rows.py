"""Block ILU(0) on the rows that leave the plain 7-point form, against the oracle.

The factorisation takes cell rows without tail entries directly, cell rows
with tail entries a warp each (one with more than 32 entries here), and falls
back to the general elimination when some cells are coupled outside the star;
the sweeps take a thread, b lanes by rows or b lanes by columns per row by
block size and precision.  Tolerances of the other CPR applications: 1e-11 in
FP64 (the same operations in another order), 1e-4 in FP32.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)


def _check(oracle, A, Ao, opts):
    from paper_1812_03952_gb300 import trs
    v = np.random.default_rng(5).standard_normal(Ao.n * Ao.b)
    ref = oracle.CPR(Ao, **opts).apply(v)
    vt = torch.from_numpy(v).cuda()
    for precision, tol in (("fp64", 1e-11), ("fp32", 1e-4)):
        M = trs.CPR(A, precision=precision, **opts)
        for _ in range(2):   # factors made at the setup, and by a refresh
            z = M.apply(vt).cpu().numpy()
            assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref), precision
            M.update(A, reuse_amg=True)


@pytest.mark.parametrize("b", [1, 2, 3, 4, 5])
def test_perforated_rows(oracle, synth, b):
    """40 wells through one cell (a row of more than 32 entries), wells crossing others, b = 1 .. 5."""
    from paper_1812_03952_gb300 import trs
    nx, ny, nz = 7, 6, 5
    hub = 3 + nx * (2 + ny * 2)
    wells = [[hub]] * 40 + [[x + nx * (2 + ny * 2) for x in range(1, 6)], [3 + nx * (y + ny * 2) for y in range(6)]]
    k = synth.lognormal_perm(np.random.default_rng(3), nx * ny * nz, 500.0, 1.0)
    s = synth.build_system(nx, ny, nz, b, k, wells, 17)
    ds = trs.DeviceSystem(s)
    _check(oracle, ds.assemble(), oracle.assemble(s), {})


@pytest.mark.parametrize("b", [1, 3, 4, 5])
@pytest.mark.parametrize("decoupling", ["abf", "none"])
def test_cells_coupled_outside_the_star(oracle, synth, b, decoupling):
    """Extra couplings between cells two apart (each closes a triangle with the cell between them)."""
    from paper_1812_03952_gb300 import trs
    s = synth.small_system(8, 7, 4, b, seed=9, n_pairs=1)
    Ao = oracle.assemble(s)
    extra = [(i, i + 2) for i in range(10, 40, 3)] + [(5, 60), (61, 5)]
    rows = [dict(zip(Ao.col[Ao.rp[i]:Ao.rp[i + 1]].tolist(), Ao.val[Ao.rp[i]:Ao.rp[i + 1]])) for i in range(Ao.n)]
    rng = np.random.default_rng(4)
    for i, j in extra:
        for a, c in ((i, j), (j, i)):
            if c not in rows[a]:
                rows[a][c] = -0.05 * abs(rows[a][a]).max() * rng.uniform(0.5, 1.0, (b, b))
    rp = np.zeros(Ao.n + 1, np.int64)
    rp[1:] = np.cumsum([len(r) for r in rows])
    col = np.array([c for r in rows for c in sorted(r)], np.int32)
    val = np.array([r[c] for r in rows for c in sorted(r)])
    A = trs.Matrix.from_bsr(rp, col, val, b, (s.nx, s.ny, s.nz))
    _check(oracle, A, oracle.BSR(Ao.n, b, rp, col, val), dict(decoupling=decoupling))
