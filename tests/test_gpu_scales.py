"""Matrices of extreme scale through the Jacobi SVD: scaled by a power of two, everything but the rotation tests'
own products scales exactly, so the vectors stay as orthogonal as at scale 1."""
import numpy as np
import pytest

from paper_1710_03757_gb300 import build, mctrg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    build.build()
    mctrg.lib()
    return pytest.importorskip("torch")


def _svd(torch, A):
    M = torch.tensor(A, device="cuda")
    batch, n = A.shape[0], A.shape[1]
    sig = torch.zeros((batch, n), dtype=torch.float64, device="cuda")
    vt = torch.zeros((batch, n, n), dtype=torch.float64, device="cuda")
    assert mctrg.mctrg_svd_batched(M, sig, vt) == mctrg.MCTRG_OK
    return sig.cpu().numpy(), vt.cpu().numpy()


@pytest.mark.parametrize("n", [8, 16, 32, 64, 96])
@pytest.mark.parametrize("k", [-270, -262, -256, -252, -248, -244, -240, -232, -215, -200, 230, 250])
def test_vectors_at_extreme_scales(torch, n, k):
    # squared row norms are about 2^2k n: their products pass 2^-926 and 2^-1000 at k = -233 and -252, 2^1000 at 248.
    # Rows are rotated while |g| > n 2^-53 sqrt(al be), g summed over n terms (n 2^-53 more) and rotations leave a few
    # eps: 8 n eps in all.  Values are within a few n eps s_1 of those at scale 1
    A = np.random.default_rng(1000 + n).standard_normal((12, n, n))
    s0, _ = _svd(torch, A)
    s, vt = _svd(torch, np.ldexp(A, k))
    eps = np.finfo(float).eps
    dots = np.einsum("bij,bkj->bik", vt, vt) - np.eye(n)
    assert np.abs(dots).max() <= 8 * n * eps
    assert np.abs(np.ldexp(s, -k) - s0).max() <= 8 * n * eps * s0.max()
