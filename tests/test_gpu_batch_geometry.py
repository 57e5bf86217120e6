"""The launch geometry of batches that mix SVD routes: which shapes are timed and kept in the cache file, and that the
kept value of a one-stage shape is the one its launches take."""
import time

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
    t = time.perf_counter()
    st, _ = mctrg.mctrg_batch_run(jobs, mctrg.make_options(svd=svd, autotune_cache=str(cache)), ln)
    assert st == mctrg.MCTRG_OK
    return ln, time.perf_counter() - t


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


def test_mixed_batches_take_the_one_stage_shape(tmp_path):
    # 128 matrices of n = 144, one per launch (one of 152 SMs at a time) or all in one: at least three times apart in
    # whole calls; the values do not depend on it
    slow, fast = tmp_path / "slow.txt", tmp_path / "fast.txt"
    slow.write_text("144 12 1 1216\n")
    fast.write_text("144 12 2432 1216\n")
    _run(fast)                                          # loads the kernels
    a, t_slow = _run(slow)
    b, t_fast = min((_run(fast) for _ in range(3)), key=lambda r: r[1])
    print("one matrix a launch %.1f ms, 2432 %.1f ms" % (1e3 * t_slow, 1e3 * t_fast))
    np.testing.assert_array_equal(a, b)
    assert t_slow > 3 * t_fast
