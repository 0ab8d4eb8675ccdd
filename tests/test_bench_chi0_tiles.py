"""bench.py's executed-to-algorithmic MMA work of the chi0 kernels counts the tiles that the pair kernel launches: strips of eight
128-column blocks, in a strip row level by row level, every tile 256 rows from any 128-row block."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _pair_tile(t, n, strip=8):
    """(first row block, column block) of tile t of n blocks."""
    c0 = 0
    while True:
        left = n - c0
        w = min(strip, left)
        for level in range((left + 1) // 2):
            full = level < left // 2
            cnt = min(w, 2 * level + 2) if full else min(w - 1, 2 * level) // 2 + 1
            if t < cnt:
                j = t if full else 2 * t
                return c0 + j + 2 * (level - j // 2), c0 + j
            t -= cnt
        c0 += strip


@pytest.mark.parametrize("kernel", ["pair", "single"])
def test_executed_work_counts_the_launched_tiles(kernel, monkeypatch):
    sys.path.insert(0, ROOT)
    import bench

    monkeypatch.setenv("GWC_CHI0_KERNEL", "single") if kernel == "single" else monkeypatch.delenv("GWC_CHI0_KERNEL", raising=False)
    for n_aux, n_ov in ((1, 64), (200, 416), (300, 640), (1100, 5859), (1190, 6099), (4500, 100), (10112, 7)):
        n = -(-n_aux // 128)
        if kernel == "pair":
            tiles = sum((n - q + 1) // 2 for q in range(n))
            cover = np.zeros((n + 1, n), dtype=np.int32)
            for t in range(tiles):
                p, q = _pair_tile(t, n)
                cover[p:p + 2, q] += 1
            assert np.all(cover[:n][np.tril(np.ones((n, n), dtype=bool))] == 1)
            assert not np.any(cover[:n][np.triu(np.ones((n, n), dtype=bool), 1)])
            blocks = 2 * tiles
        else:
            blocks = n * (n + 1) // 2
        executed = blocks * 128 * 128 * (-(-n_ov // 64) * 64)
        assert abs(bench.chi0_executed_ratio(n_aux, n_ov) - executed / (n_aux * (n_aux + 1) / 2 * n_ov)) < 1e-9
