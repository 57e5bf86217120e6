"""Host check of the low-rank levels' factorization (no GPU): a plaquette tensor's own matricization on
either sublattice is X Yt^T of the stated factors, and the core of their QR factors has its singular values."""
import numpy as np
import pytest


@pytest.mark.parametrize("d,D,parity", [(2, 3, 0), (2, 3, 1), (3, 4, 0), (3, 4, 1), (4, 5, 1), (4, 12, 0), (4, 12, 1)])
def test_factors_and_core(d, D, parity):
    rng = np.random.default_rng(100 * d + 10 * D + parity)
    F3, F4 = rng.standard_normal((D, d, d)), rng.standard_normal((D, d, d))       # [al,i,j], [be,k,i]
    F2, F1 = rng.standard_normal((d, d, D)), rng.standard_normal((d, d, D))       # [j,m,ga], [m,k,de]
    T = np.einsum("aij,bki,jmg,mkd->abdg", F3, F4, F2, F1)                         # legs (l,u,r,d) = (al,be,de,ga)
    if parity == 0:
        M = T.reshape(D * D, D * D)
        X = np.einsum("aij,bki->abjk", F3, F4).reshape(D * D, d * d)
        Y = np.einsum("jmg,mkd->dgjk", F2, F1).reshape(D * D, d * d)
    else:
        M = T.transpose(1, 2, 3, 0).reshape(D * D, D * D)                          # (u,r),(d,l)
        X = np.einsum("bki,mkd->bdim", F4, F1).reshape(D * D, d * d)
        Y = np.einsum("aij,jmg->gaim", F3, F2).reshape(D * D, d * d)
    np.testing.assert_allclose(X @ Y.T, M, rtol=0, atol=1e-12 * np.abs(M).max())
    (Qx, Rx), (Qy, Ry) = np.linalg.qr(X), np.linalg.qr(Y)
    U, s, Vt = np.linalg.svd(Rx @ Ry.T)
    full = np.linalg.svd(M, compute_uv=False)
    # backward stable: a few eps |X| |Y| (absolute), K = d^2 nonzero values
    bound = 50 * np.finfo(float).eps * np.linalg.norm(X) * np.linalg.norm(Y)
    assert np.abs(s - full[:d * d]).max() <= bound and full[d * d:].max() <= bound
    np.testing.assert_allclose((Qx @ U * s) @ (Vt @ Qy.T), M, rtol=0, atol=bound)
