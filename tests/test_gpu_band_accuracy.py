"""Rounding of the two-stage SVD route, against matrices whose singular values are known exactly: M = S1 P1 H D H P2 S2
with H the Hadamard matrix of order n (H H = n I), D a diagonal of integers, permutations P and signs S, so that M is
exact in FP64 and its singular values are n |D_i|."""
import numpy as np
import pytest

from paper_1710_03757_gb300 import build, mctrg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    build.build()
    mctrg.lib()
    return pytest.importorskip("torch")


def _hadamard(n):
    H = np.ones((1, 1))
    while H.shape[0] < n:
        H = np.block([[H, H], [H, -H]])
    return H


def _known(n, batch, seed):
    """Matrices with a flat spectrum (ratio 3 from largest to smallest) and their singular values, descending."""
    rng = np.random.default_rng(seed)
    H = _hadamard(n)
    mats, vals = [], []
    for _ in range(batch):
        D = rng.integers(1 << 19, 3 << 19, n).astype(np.float64)
        M = (H * D) @ H                                    # integers below 2^30: exact
        M = M[rng.permutation(n)][:, rng.permutation(n)]
        mats.append(M * rng.choice([-1.0, 1.0], (n, 1)) * rng.choice([-1.0, 1.0], n))
        vals.append(np.sort(D)[::-1] * n)
    return np.stack(mats), np.stack(vals)


def _svd(torch, A, n_vec):
    batch, n = A.shape[0], A.shape[1]
    sig = torch.zeros((batch, n), dtype=torch.float64, device="cuda")
    vt = torch.zeros((batch, n_vec, n), dtype=torch.float64, device="cuda")
    assert mctrg.mctrg_svd_band_batched(torch.tensor(np.ascontiguousarray(A), device="cuda"), sig, vt) == mctrg.MCTRG_OK
    return sig.cpu().numpy(), vt.cpu().numpy()


@pytest.mark.parametrize("n", [128, 256])
def test_rms_error_on_a_flat_spectrum(torch, n):
    # |M|_F is 0.7 sqrt(n) s_1, so the fixed point has few bits to spare: the digit products keep 2^-65 |M|_F, below
    # 1e-17 s_1 a panel, and the FP64 panels and the bulge chase remain, 1.3e-16 s_1 rms on other matrices of these
    # sides.  Half as much again is allowed; eight digit groups instead of nine gave 2.65e-16 at n = 256
    A, ref = _known(n, 24, 5 + n)
    sig, _ = _svd(torch, A, 1)
    rms = np.sqrt((((sig - ref) / ref[:, :1]) ** 2).mean())
    print("n %d: rms error %.2e s_1" % (n, rms))
    assert rms <= 2.0e-16


@pytest.mark.parametrize("n,n_vec,batch", [(64, 3, 5), (200, 16, 5), (256, 16, 5), (256, 16, 200)])
def test_vectors_have_unit_length(torch, n, n_vec, batch):
    # the squared length is summed over n / 32 terms and five steps of a tree, at most 13 roundings, its root and the
    # scaling take three more and each entry's rounding one: |v|^2 = 1 within 2 (13 / 2 + 4) 2^-53 at worst, and within
    # half of that as roundings average (without the scaling 1.3e-15 to 3e-15)
    rng = np.random.default_rng(n + batch)
    A = rng.standard_normal((batch, n, n)) * np.logspace(0, -8, n) @ rng.standard_normal((n, n))
    _, vt = _svd(torch, A, n_vec)
    lengths = (vt.astype(np.longdouble) ** 2).sum(2)
    assert float(np.abs(lengths - 1).max()) <= 10.5 * 2.0 ** -53
