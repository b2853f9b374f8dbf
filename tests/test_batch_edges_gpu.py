"""Batched scans at the edges of their kernel: zone windows (32 blocks a load, whole
tiles of it) entered, left and crossed with survivors in every pattern, tiles wider
than a window, runs of tiles with nothing to read, empty predicates between others,
columns shorter than a tile, and launches of several width groups whose warps move
from one to the next.  Against the oracle: COUNT, SUM and blocks read, exactly."""
import numpy as np
import pytest

import oracle
import synth
from paper_2606_22423_gb300 import gbscan

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    import __graft_entry__

    __graft_entry__.build()
    torch.cuda.init()
    gbscan.load()
    gbscan.autotune_reset()
    yield
    gbscan.autotune_reset()


def patterned(b, blocks, rem, keep, seed):
    """A column whose block k holds values of the upper half of the domain where keep(k), of
    the lower half elsewhere."""
    n = blocks * 1024 + rem
    half = 1 << (b - 1)
    rng = np.random.default_rng(seed)
    v = rng.integers(0, max(half, 1), size=n, dtype=np.uint32)
    k = np.arange(n) // 1024
    v[keep(k)] += np.uint32(half)
    return v


PATTERNS = [lambda k: k % 2 == 0, lambda k: k % 33 == 32, lambda k: (k % 64) < 2, lambda k: k < 0,
            lambda k: k >= 0, lambda k: (k == 0) | (k == 95), lambda k: k % 5 == 3]


@pytest.mark.parametrize("widths", [(1, 2, 3, 4), (5, 8, 9, 12), (13, 16, 17, 20), (24, 28, 29, 32)])
@pytest.mark.parametrize("tile_blocks", [None, 64])
def test_zone_windows_and_groups_match_the_oracle(widths, tile_blocks):
    gbscan.autotune_reset()
    cols, strategies, preds, want = [], [], [], []
    for b in widths:
        if tile_blocks and 4 * 2 * (tile_blocks * 128 * b + 24) <= 226 * 1024:
            for branchy in (False, True):
                gbscan.batch_shape_set(b, branchy, dict(warps=4, stages=2, tile_blocks=tile_blocks))
        for i, keep in enumerate(PATTERNS):
            blocks, rem = [(96, 0), (33, 1), (31, 1023), (200, 17), (1, 0), (96, 5), (0, 700)][i]
            v = patterned(b, blocks, rem, keep, 100 * b + i)
            col = gbscan.Column.from_host(v, b)
            col.zonemap_build()
            top = 1 << b
            for strategy, (lo, hi) in (("zone_bf", (top // 2, top)), ("zone_br", (top // 2, top)),
                                       ("branchfree", (0, 0)), ("branchfree", (top // 2, top)), ("zone_bf", (top, top + 9)),
                                       ("branchy", (0, top))):
                words = oracle.pack(v, b, 0)
                zmin, zmax = oracle.zonemap(words, v.size, b, 0)
                pair = oracle.scan_values(v, lo, hi)
                if lo >= hi or lo >= top:
                    touched = 0
                elif strategy.startswith("zone"):
                    touched = oracle.scan_zoneskip(words, zmin, zmax, v.size, b, 0, lo, hi)[2]
                else:
                    touched = (v.size + 1023) // 1024
                cols.append(col)
                strategies.append(strategy)
                preds.append((lo, hi))
                want.append((*pair, touched))
    for pop in (0, 1, 3):
        bt = gbscan.Batch(cols, strategies, tiles_per_pop=pop)
        for _ in range(2):
            got = [(r.count, r.sum, r.blocks_scanned) for r in bt.run(preds)]
            assert got == want, (widths, tile_blocks, pop)
        bt.close()
    for c in set(cols):
        c.close()
