"""The AMG setup's kernels at the edges of their ranges, against the oracle.

Every level's operator, aggregates and eigenvalue bound equal the oracle's bit
for bit: wells whose aggregates hold more than 32 and more than 256 members
and whose rows are longer than a warp, levels of at most 8 entries a row and
of more (1 and 8 lanes per row), a diagonal of ones and others (no
decoupling), and the V-cycle through the coarsest inverse at 1, 63, 64 and 65
rows (1e-11 as for the other FP64 applications).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

CASES = [
    (dict(nx=400, ny=5, nz=3, b=2, seed=3, n_pairs=1), {}),
    (dict(nx=31, ny=9, nz=7, b=3, seed=4, n_pairs=2, kvkh=0.1, sigma=1.5), dict(decoupling="none")),
    (dict(nx=24, ny=20, nz=16, b=1, seed=5, n_pairs=3), {}),
    (dict(nx=1, ny=1, nz=1, b=2, seed=6, n_pairs=0), {}),
    (dict(nx=9, ny=7, nz=1, b=1, seed=7, n_pairs=0), dict(max_levels=1, coarse_max=64)),
    (dict(nx=8, ny=8, nz=1, b=1, seed=8, n_pairs=0), dict(max_levels=1, coarse_max=64)),
    (dict(nx=13, ny=5, nz=1, b=1, seed=9, n_pairs=0), dict(max_levels=1, coarse_max=64)),
]


@pytest.mark.parametrize("case,opts", CASES, ids=lambda v: "-".join(f"{k}{x}" for k, x in v.items()) or "default")
def test_setup_edges(oracle, synth, case, opts):
    from paper_1812_03952_gb300 import trs
    s = synth.small_system(**case)
    ds = trs.DeviceSystem(s)
    ds.assemble()
    M = trs.CPR(ds.A, **opts)
    Mo = oracle.CPR(oracle.assemble(s), **opts)
    amg = Mo.amg
    info = M.info()
    assert info["level_rows"] == amg.sizes()
    for l in range(amg.n_levels):
        for got, ref in zip(M.level(l), amg.level(l)):
            np.testing.assert_array_equal(got, ref)
        np.testing.assert_array_equal(M.aggregates(l), amg.agg(l))
        assert info["level_lambda"][l] == amg.lam(l)
    r = np.random.default_rng(12).standard_normal(s.n_rows)
    ref = amg.vcycle(r)
    e = M.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    assert np.linalg.norm(e - ref) <= 1e-11 * np.linalg.norm(ref)
