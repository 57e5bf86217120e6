"""The low-rank levels' split (the core of the QR factors) on the device, per trajectory against the oracle
(1e-10, tests/parity.py) and against the same level split as a whole matrix (route BIDIAG).

Sides and inner dimensions at the edges of the kernel's layouts: K = 16 in half-warps (n = 25, 49, 64, 144), a K that
is no power of two (a D = 3 site tensor: K = 9; D = 5: K = 25), K = 256 in shared and global memory (n = 289, 576)."""
import numpy as np
import pytest

from oracle import ising
from oracle.trg import Problem, run_many
from paper_1710_03757_gb300 import build, mctrg
from paper_1710_03757_gb300.workloads import generic_tensor

from parity import compare
from test_gpu_parity import gpu_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


@pytest.mark.parametrize("L,chi,n,h", [(8, 5, 40, 0.0), (16, 7, 10, 0.05), (16, 8, 12, 0.0), (16, 12, 6, 0.05)])
@pytest.mark.parametrize("precision", [mctrg.MCTRG_FP64, mctrg.MCTRG_FP64TC])
def test_ising_against_oracle(L, chi, n, h, precision):
    gpu = gpu_run(L, chi, n, 31 + chi, beta=0.44, h=h, precision=precision)
    orc = run_many(Problem(ising.site_tensor(0.44, h), L, chi), 31 + chi, 0, n, workers=4)
    compare(gpu, orc, min_ok=0.9, label="low rank L%d chi%d" % (L, chi))


@pytest.mark.parametrize("D,L,chi,n", [(3, 4, 4, 40), (3, 8, 6, 10), (5, 4, 7, 10)])
def test_generic_against_oracle(D, L, chi, n):
    T0 = generic_tensor(D, seed=50 + D)
    gpu = gpu_run(L, chi, n, 77, T0=T0)
    orc = run_many(Problem(T0, L, chi), 77, 0, n, workers=4)
    compare(gpu, orc, min_ok=0.9, label="low rank generic D%d chi%d" % (D, chi))


@pytest.mark.parametrize("chi,svd", [(17, mctrg.SVD_AUTO), (24, mctrg.SVD_AUTO), (24, mctrg.SVD_BAND)])
def test_large_core_against_whole_matrices(chi, svd):
    a = gpu_run(16, chi, 3, 9, beta=0.44, svd=svd)
    b = gpu_run(16, chi, 3, 9, beta=0.44, svd=mctrg.SVD_BIDIAG)
    ok = (a[3] == 0) & (b[3] == 0)
    assert ok.sum() >= 2 and np.array_equal(a[2][ok], b[2][ok])
    assert (np.abs(a[1] - b[1])[ok] <= 1e-10 * np.abs(b[1][ok])).all()
