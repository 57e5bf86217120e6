"""The launch geometry of batches that mix SVD routes: which shapes are timed and kept in the cache file."""

import numpy as np
import pytest

from paper_1710_03757_gb300 import build, mctrg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()
    mctrg.lib()


# (beta, h, L, chi, n, seed, first): chi = 12 has n = 144 on the one-stage route, chi = 16 n = 256 on the two-stage one
MIXED = [(0.44, 0.0, 8, 12, 64, 1, 0), (0.44, 0.0, 16, 16, 1, 2, 0)]


def _run(cache, jobs=MIXED, svd=mctrg.SVD_AUTO):
    total = sum(j[4] for j in jobs)
    ln = np.zeros(total)
    st, _ = mctrg.mctrg_batch_run(jobs, mctrg.make_options(svd=svd, autotune_cache=str(cache)), ln)
    assert st == mctrg.MCTRG_OK
    return ln


def _shapes(cache):
    rows = [tuple(int(x) for x in line.split()) for line in cache.read_text().splitlines()]
    return {(n, kc): items for n, kc, items, _ in rows}


def test_only_timed_shapes_are_kept(tmp_path):
    cache = tmp_path / "geometry.txt"
    _run(cache)
    first = _shapes(cache)
    assert (144, 12) in first and (256, 16) not in first
    # the same lattices on the one-stage route throughout: its own shape is timed then (1 to 16 matrices per SM)
    _run(cache, svd=mctrg.SVD_BIDIAG)
    assert 0 < _shapes(cache)[256, 16] < 1 << 14


def test_an_untimed_line_is_timed_when_needed(tmp_path):
    cache = tmp_path / "geometry.txt"
    cache.write_text("256 16 65536 1216\n")
    _run(cache, jobs=MIXED[1:], svd=mctrg.SVD_BIDIAG)
    assert 0 < _shapes(cache)[256, 16] < 1 << 14
