"""The V-cycle's kernels at the edges of their ranges, against the oracle.

Level 0 takes a thread per cell row and a warp per well row (with more than
32 * 4 perforations in one case), CSR levels kCsrLanes lanes per row (rows of
more than 32 entries on the coarse levels), the coarsest levels one block out
of shared memory (a single row, a coarsest level above and below the 64 rows
whose inverse is staged, levels that do not fit), with Chebyshev degrees 2
and 3.  Tolerance 1e-11 as for the other FP64 applications: the same
operations in another summation order over at most a few hundred terms a row
and five levels, a few thousand units of 2^-53 at worst.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

CASES = [
    (dict(nx=3, ny=1, nz=2, b=1, seed=3, n_pairs=0), {}),
    (dict(nx=200, ny=6, nz=4, b=2, seed=4, n_pairs=1), {}),                      # wells of 198 perforations
    (dict(nx=40, ny=36, nz=20, b=1, seed=5, n_pairs=2, sigma=1.5, kvkh=0.1), {}),
    (dict(nx=40, ny=36, nz=20, b=1, seed=5, n_pairs=2), dict(coarse_max=900)),   # coarsest level not staged
    (dict(nx=40, ny=36, nz=20, b=1, seed=6, n_pairs=2), dict(max_levels=2)),     # coarsest level above 1024 rows
    (dict(nx=33, ny=17, nz=9, b=3, seed=7, n_pairs=3), dict(cheb_degree=3)),
    (dict(nx=64, ny=48, nz=16, b=1, seed=8, n_pairs=2, shale_frac=0.1), dict(cheb_degree=3)),
]


@pytest.mark.parametrize("case,opts", CASES, ids=lambda v: "-".join(f"{k}{x}" for k, x in v.items()) or "default")
def test_vcycle_levels(oracle, synth, case, opts):
    from paper_1812_03952_gb300 import trs
    s = synth.small_system(**case)
    ds = trs.DeviceSystem(s)
    ds.assemble()
    Mo = oracle.CPR(oracle.assemble(s), **opts)
    r = np.random.default_rng(11).standard_normal(s.n_rows)
    ref = Mo.amg.vcycle(r)
    rt = torch.from_numpy(r).cuda()
    e = trs.CPR(ds.A, **opts).vcycle(rt).cpu().numpy()
    assert np.linalg.norm(e - ref) <= 1e-11 * np.linalg.norm(ref)
    # the FP32 form of the same kernels, 1e-4 as for the other FP32 applications
    e32 = trs.CPR(ds.A, precision="fp32", **opts).vcycle(rt).cpu().numpy()
    assert np.linalg.norm(e32 - ref) <= 1e-4 * np.linalg.norm(ref)
