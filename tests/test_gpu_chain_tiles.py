"""The gradient chain over tiles of 8 x 8 x 4 cells, and the outer product over
runs of 256 entries, at the edges of tiles and runs.

The reference is the same contraction in extended precision; a cell's value is
a sum of at most 6 faces of 2 (B^2 + B) products, each within a few units of
2^-53, so 64 * 2^-53 of the sum of the terms' absolute values is the bound.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("is_log", [False, True])
@pytest.mark.parametrize("shape,b", [((1, 1, 1), 2), ((8, 8, 4), 1), ((9, 1, 5), 3), ((1, 17, 3), 4), ((7, 9, 9), 5),
                                     ((17, 8, 5), 3), ((16, 16, 8), 2)])
def test_chain_tiles(synth, shape, b, is_log):
    from paper_1812_03952_gb300 import trs
    s = synth.small_system(nx=shape[0], ny=shape[1], nz=shape[2], b=b, seed=5, n_pairs=0, kvkh=0.3)
    k = s.k.reshape(shape[::-1]).copy()
    k[0, 0, 0] = 0.0 if not is_log else k[0, 0, 0]
    if k.size > 1 and not is_log:
        k.reshape(-1)[1] = 0.0     # a face between two zero permeabilities, where x has an extent
    ds = trs.DeviceSystem(s)
    ds.assemble()
    rng = np.random.default_rng(6)
    lam, x = rng.standard_normal((2, s.n_unknowns))
    perm = np.log(k) if is_log else k
    dev = [torch.from_numpy(np.ascontiguousarray(v).reshape(-1)).cuda() for v in (perm, lam, x)]
    got = trs.chain_theta(ds.A, dev[0], ds.M, dev[1], dev[2], s.kvkh, s.c_t, perm_is_log=is_log).cpu().numpy()
    dA = trs.outer_product(ds.A, dev[1], dev[2]).cpu().numpy().reshape(-1, b, b)
    rp, col = ds.A.pattern()
    row = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    np.testing.assert_array_equal(dA, -(lam.reshape(-1, b)[row][:, :, None] * x.reshape(-1, b)[col][:, None, :]))

    kl = (np.exp(perm.astype(np.longdouble)) if is_log else k.astype(np.longdouble))
    nz, ny, nx = kl.shape
    M = s.M.reshape(nz, ny, nx, 6, b, b).astype(np.longdouble)
    L = lam[:s.n_cells * b].reshape(nz, ny, nx, b).astype(np.longdouble)
    X = x[:s.n_cells * b].reshape(nz, ny, nx, b).astype(np.longdouble)
    ref, mag = np.zeros((2,) + kl.shape, np.longdouble)
    for a, axis in ((0, 2), (1, 1), (2, 0)):
        lo = tuple(slice(None, -1) if d == axis else slice(None) for d in range(3))
        up = tuple(slice(1, None) if d == axis else slice(None) for d in range(3))
        dx = X[up] - X[lo]
        t = [np.einsum("...r,...rc,...c->...", L[lo], M[lo][..., 3 + a, :, :], dx),
             -np.einsum("...r,...rc,...c->...", L[up], M[up][..., 2 - a, :, :], dx)]
        mt = sum(np.einsum("...r,...rc,...c->...", abs(l), abs(m), abs(X[up]) + abs(X[lo]))
                 for l, m in ((L[lo], M[lo][..., 3 + a, :, :]), (L[up], M[up][..., 2 - a, :, :])))
        den = kl[lo] + kl[up]
        den[den == 0] = 1
        c = s.c_t * (s.kvkh if a == 2 else 1.0)
        T = c * 2 * kl[lo] * kl[up] / den
        for side, other in ((lo, up), (up, lo)):
            ref[side] += (t[0] + t[1]) * T * kl[other] / den
            mag[side] += mt * T * kl[other] / den
    assert np.all(np.abs(got.reshape(ref.shape) - ref) <= 64 * 2.0**-53 * mag)
