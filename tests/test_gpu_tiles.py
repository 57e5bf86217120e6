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


@pytest.mark.parametrize("K", [64, 320])
def test_tensor_core_products_at_the_edges(torch, K):
    # rows at the ends of the exponent range, values that round up to the row's power of two, zeros, and inputs
    # off a 16-byte boundary.  With one nonzero per row and column each product is exact up to the 55 bits kept
    # of either factor: within 2^-54 of it relative to |row max| |column max|, rounded once (2^-53)
    n, batch = 49, 2
    rng = np.random.default_rng(K)
    X, Y = np.zeros((batch, n, K)), np.zeros((batch, n, K))
    k = rng.integers(0, K, size=(batch, n))
    for b in range(batch):
        for r in range(n):
            X[b, r, k[b, r]] = rng.choice([-1.0, 1.0]) * 2.0 ** rng.integers(-500, 500) * rng.uniform(1, 2)
            Y[b, r, k[b, r]] = rng.choice([-1.0, 1.0]) * 2.0 ** rng.integers(-500, 500) * rng.uniform(1, 2)
    X[0, 0] = 0.0
    X[0, 1, k[0, 1]], Y[0, 1, k[0, 1]] = 1.0 - 2.0 ** -53, -(1.0 - 2.0 ** -53)
    X[0, 2, k[0, 2]], Y[0, 2, k[0, 2]] = 5e-324 * 12345, 2.0 ** 1000      # a row of subnormal numbers
    X[0, 3, k[0, 3]], Y[0, 3, k[0, 3]] = 2.0 ** -1000, 2.0 ** -60         # a subnormal product
    ref = np.einsum('bik,bjk->bij', X, Y)
    pad = torch.zeros(2 * batch * n * K + 3, dtype=torch.float64, device="cuda")
    Xd = pad[1:1 + batch * n * K].view(batch, n, K)
    Yd = pad[2 + batch * n * K:2 + 2 * batch * n * K].view(batch, n, K)
    Xd.copy_(torch.tensor(X))
    Yd.copy_(torch.tensor(Y))
    M = torch.full((batch, n, n), float("nan"), dtype=torch.float64, device="cuda")
    assert mctrg.mctrg_contract_batched(Xd, Yd, M, precision=mctrg.MCTRG_FP64TC) == mctrg.MCTRG_OK
    scale = np.abs(X).max(2)[:, :, None] * np.abs(Y).max(2)[:, None, :]
    assert (np.abs(M.cpu().numpy() - ref) <= 2.0 ** -51 * scale + 5e-324).all()
    assert (M.cpu().numpy()[ref == 0] == 0).all()


@pytest.mark.parametrize("over", ["X", "Yt"])
def test_tensor_core_product_over_an_operand(torch, over):
    # D = 16, K = 256: the result has the operands' shape and may be written over one of them
    rng = np.random.default_rng(3)
    X, Y = (torch.tensor(rng.standard_normal((40, 256, 256)), device="cuda") for _ in range(2))
    ref = torch.empty_like(X)
    assert mctrg.mctrg_contract_batched(X, Y, ref, precision=mctrg.MCTRG_FP64TC) == mctrg.MCTRG_OK
    out = X if over == "X" else Y
    assert mctrg.mctrg_contract_batched(X, Y, out, precision=mctrg.MCTRG_FP64TC) == mctrg.MCTRG_OK
    assert torch.equal(out, ref)


@pytest.mark.parametrize("chi,svd", [(8, mctrg.SVD_BIDIAG), (9, mctrg.SVD_AUTO), (12, mctrg.SVD_AUTO),
                                     (16, mctrg.SVD_AUTO)])
def test_few_trajectories_equal_the_same_of_many(torch, chi, svd):
    few = gpu_run(8, chi, 3, 5, beta=0.44, h=0.02, svd=svd)
    many = gpu_run(8, chi, 330, 5, beta=0.44, h=0.02, svd=svd)
    for i in (1, 2, 3):
        np.testing.assert_array_equal(few[i], many[i][:3])
