"""The bit-sliced scans against the oracle at their edges: every width they serve
and the first ones they do not, odd block counts (a tile's last block runs alone),
ragged tails, columns of one value, and bounds at both ends of the domain and at
bit patterns that take every branch of the carry chains.  Integers: exact."""
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


def bounds(b):
    top = 1 << b
    ones, zeros = int("01" * 16, 2) % top, int("10" * 16, 2) % top
    cuts = sorted({0, 1, top // 2, top - 1, ones, zeros})
    return [(lo, hi) for lo in cuts for hi in cuts + [top] if lo < hi]


@pytest.mark.parametrize("b", range(1, 18))
def test_sliced_scans_match_the_oracle_at_their_edges(b):
    base = 5 if b < 32 else 0
    layouts = ["lanes", "rowmajor"] + (["bytes"] if b in (8, 16) else [])
    for n in (1024, 3 * 1024, 37 * 1024 + 1, 2433 * 1024 + 1023):
        v = synth.uniform_values(synth.seed_for(95, b, n), n, b, base)
        for const in (None, 0, (1 << b) - 1):
            if const is not None:
                if n != 3 * 1024:
                    continue
                v = np.full(n, base + const, dtype=np.uint32)
            want = [oracle.scan_values(v, base + lo, base + hi) for lo, hi in bounds(b)]
            for layout in layouts:
                col = gbscan.Column.from_host(v, b, base, layout=layout)
                for strategy in ("branchfree", "branchy"):
                    for (lo, hi), w in zip(bounds(b), want):
                        r = col.run(base + lo, base + hi, strategy)
                        assert r.pair() == w, (b, n, const, layout, strategy, lo, hi)
                        assert r.blocks_scanned == (n + 1023) // 1024
                col.close()
