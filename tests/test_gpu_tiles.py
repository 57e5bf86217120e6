"""The sizes at which work is divided differently: the FP64 product's tile
against exact integer products at sides around its tiles, and runs of few
trajectories (items and ranks shared by several blocks) against the same
trajectories in a run of many, bit by bit."""
import numpy as np
import pytest

from paper_1710_03757_gb300 import build, mctrg

from test_gpu_parity import gpu_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    build.build()
    mctrg.lib()
    return pytest.importorskip("torch")


@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 6, 7, 10, 12, 13])
def test_fp64_products_of_integers(torch, D):
    rng = np.random.default_rng(D)
    n, K = D * D, D * D + 3
    X = rng.integers(-(1 << 20), 1 << 20, size=(3, n, K)).astype(np.float64)
    Y = rng.integers(-(1 << 20), 1 << 20, size=(3, n, K)).astype(np.float64)
    M = torch.full((3, n, n), float("nan"), dtype=torch.float64, device="cuda")
    st = mctrg.mctrg_contract_batched(torch.tensor(X, device="cuda"), torch.tensor(Y, device="cuda"), M,
                                      precision=mctrg.MCTRG_FP64)
    assert st == mctrg.MCTRG_OK
    np.testing.assert_array_equal(M.cpu().numpy(), np.einsum('bik,bjk->bij', X, Y))


@pytest.mark.parametrize("chi,svd", [(8, mctrg.SVD_BIDIAG), (9, mctrg.SVD_AUTO), (12, mctrg.SVD_AUTO),
                                     (16, mctrg.SVD_AUTO)])
def test_few_trajectories_equal_the_same_of_many(torch, chi, svd):
    few = gpu_run(8, chi, 3, 5, beta=0.44, h=0.02, svd=svd)
    many = gpu_run(8, chi, 330, 5, beta=0.44, h=0.02, svd=svd)
    for i in (1, 2, 3):
        np.testing.assert_array_equal(few[i], many[i][:3])
