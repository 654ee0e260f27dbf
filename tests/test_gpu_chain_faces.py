"""The gradient chain on matrices that do not store every face of their grid.

A face whose blocks are left out of the pattern (a sealed fault, an inactive
cell) has no transmissibility: it adds nothing, and its M is not used (NaN
here).  The reference is the contraction over the stored faces in extended
precision, with the tolerance of the complete grids: 64 * 2^-53 of the sum of
the terms' absolute values (6 faces of 2 (B^2 + B) products each).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("left_out", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("shape,b", [((9, 7, 6), 3), ((8, 8, 4), 1), ((17, 3, 5), 4), ((1, 9, 10), 2)])
def test_chain_faces_not_stored(shape, b, left_out):
    from paper_1812_03952_gb300 import trs
    nx, ny, nz = shape
    n = nx * ny * nz
    rng = np.random.default_rng(8)
    idx = np.arange(n).reshape(nz, ny, nx)
    k = rng.lognormal(size=n)
    M = rng.standard_normal((n, 6, b, b))
    lam, x = rng.standard_normal((2, n, b))
    kvkh, c_t = 0.3, 1.7
    pairs = [(i, i) for i in range(n)]
    ref, mag = np.zeros((2, n), np.longdouble)
    for a, axis in ((0, 2), (1, 1), (2, 0)):
        lo = idx.take(range(idx.shape[axis] - 1), axis).ravel()
        up = idx.take(range(1, idx.shape[axis]), axis).ravel()
        keep = rng.random(lo.size) >= left_out
        M[lo[~keep], 3 + a] = np.nan
        M[up[~keep], 2 - a] = np.nan
        lo, up = lo[keep], up[keep]
        pairs += list(zip(lo, up)) + list(zip(up, lo))
        L, X, Ml = lam.astype(np.longdouble), x.astype(np.longdouble), M.astype(np.longdouble)
        kl = k.astype(np.longdouble)
        t = (np.einsum("nr,nrc,nc->n", L[lo], Ml[lo, 3 + a], X[up] - X[lo])
             - np.einsum("nr,nrc,nc->n", L[up], Ml[up, 2 - a], X[up] - X[lo]))
        mt = (np.einsum("nr,nrc,nc->n", abs(L[lo]), abs(Ml[lo, 3 + a]), abs(X[up]) + abs(X[lo]))
              + np.einsum("nr,nrc,nc->n", abs(L[up]), abs(Ml[up, 2 - a]), abs(X[up]) + abs(X[lo])))
        den = kl[lo] + kl[up]
        T = c_t * (kvkh if a == 2 else 1.0) * 2 * kl[lo] * kl[up] / den
        for side, other in ((lo, up), (up, lo)):
            np.add.at(ref, side, t * T * kl[other] / den)
            np.add.at(mag, side, mt * T * kl[other] / den)
    pairs = np.array(sorted(pairs))
    rp = np.zeros(n + 1, np.int64)
    np.add.at(rp, pairs[:, 0] + 1, 1)
    A = trs.Matrix.from_bsr(np.cumsum(rp), pairs[:, 1], None, b, shape)
    d = [torch.from_numpy(np.ascontiguousarray(v)).reshape(-1).cuda() for v in (k, M, lam, x)]
    got = trs.chain_theta(A, d[0], d[1], d[2], d[3], kvkh, c_t).cpu().numpy()
    assert np.all(np.abs(got - ref) <= 64 * 2.0**-53 * mag)
