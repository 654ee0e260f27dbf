"""The coarsest levels of the V-cycle: which of them one block runs together.

Each case says by its level sizes which branch it takes: levels whose entries
fill the block's shared memory in FP64 but not in FP32, a coarsest level of one
row below others, one whose inverse is multiplied by the block (65 to 160 rows
below a level that it runs too), by a kernel of its own (above, or alone).
Against the oracle; 1e-11 in FP64, 1e-4 in FP32, as for the other V-cycles.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

SMEM = 200 * 1024


def _bytes(rows, nnz, l, size):
    """Shared memory of level l of at most 1024 rows, and of those below it."""
    total = 8 * rows[-1] ** 2 if rows[-1] <= 64 else 0
    for m in range(l, len(rows) - 1):
        total += (nnz[m] + 6 * rows[m]) * size + (rows[m] + rows[m + 1] + 2) * 4 + (nnz[m] + 2 * rows[m]) * 2
    return total + 2 * rows[-1] * size


def _fits_fp32_only(rows, nnz):
    return rows[2] <= 1024 and _bytes(rows, nnz, 2, 4) < SMEM < _bytes(rows, nnz, 2, 8)


CASES = [
    ((64, 48, 40), {}, _fits_fp32_only),
    ((12, 12, 6), dict(coarse_max=1), lambda rows, nnz: rows[-1] == 1 and len(rows) > 3 and rows[-3] <= 1024),
    ((1, 1, 20000), dict(coarse_max=200), lambda rows, nnz: 64 < rows[-1] <= 160 < rows[-2] <= 1024),
    ((1, 1, 8000), dict(coarse_max=200), lambda rows, nnz: 160 < rows[-1] and rows[-2] <= 1024),
    ((2, 2, 6000), dict(coarse_max=900), lambda rows, nnz: 160 < rows[-1] <= 1024 < rows[-2]),
    ((30, 30, 30), dict(coarse_max=300), lambda rows, nnz: 160 < rows[-1] <= 300),
    ((5, 4, 3), {}, lambda rows, nnz: len(rows) == 1),
]


@pytest.mark.parametrize("shape,opts,branch", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else "")
def test_values(oracle, synth, shape, opts, branch):
    from paper_1812_03952_gb300 import trs
    s = synth.small_system(*shape, 1, seed=5, n_pairs=0)
    ds = trs.DeviceSystem(s)
    ds.assemble()
    ref = oracle.CPR(oracle.assemble(s), **opts)
    r = np.random.default_rng(2).standard_normal(s.n_rows)
    want = ref.amg.vcycle(r)
    for precision, tol in (("fp64", 1e-11), ("fp32", 1e-4)):
        M = trs.CPR(ds.A, precision=precision, **opts)
        info = M.info()
        assert branch(info["level_rows"], info["level_nnz"])
        e = M.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
        assert np.linalg.norm(e - want) <= tol * np.linalg.norm(want)


def test_time(synth):
    """A coarsest level of hundreds of rows costs no more than the levels below it
    would (1.5 times leaves room; one block took 1.9 at 400 rows, 8 at 800)."""
    from paper_1812_03952_gb300 import trs
    s = synth.small_system(2, 2, 6000, 1, seed=5, n_pairs=0)
    ds = trs.DeviceSystem(s)
    ds.assemble()
    r = torch.rand(s.n_rows, device="cuda", dtype=torch.float64)

    def best(**opts):
        M = trs.CPR(ds.A, **opts)
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

    assert best(coarse_max=900) <= 1.5 * best()
