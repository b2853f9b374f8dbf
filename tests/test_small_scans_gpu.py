"""Small columns against the oracle at the sizes where the launch changes: one CTA
with a warp per tile, the step to several CTAs, to all SMs, and to more than one tile
per warp; with and without a ragged tail, both layouts and flavours.  Integers: exact."""
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


@pytest.mark.parametrize("b", [1, 5, 12, 13, 16, 17, 24, 32])
def test_small_scans_match_the_oracle_at_launch_changes(b):
    sms = gbscan.scan_launch_shape(b)["sms"]
    edges = sorted({1, 2, 4, 7, 8, 9, 15, 16, 17, 31, 33, 8 * sms - 1, 8 * sms + 1, 16 * sms, 16 * sms + 1})
    base = min(9, (1 << 32) - (1 << b))
    v = synth.uniform_values(synth.seed_for(96, b), (edges[-1] + 1) * 1024, b, base)
    preds = [synth.pick_range(synth.seed_for(96, b, i), b, s, base) for i, s in enumerate((0.001, 0.5, 1.0))]
    for blocks in [0] + edges:
        for rem in (0, 1, 1023):
            n = blocks * 1024 + rem
            if n == 0:
                continue
            part = v[:n]
            want = [oracle.scan_values(part, lo, hi) for lo, hi in preds]
            for layout in ("lanes", "rowmajor"):
                col = gbscan.Column.from_host(part, b, base, layout=layout)
                for strategy in ("branchfree", "branchy"):
                    for (lo, hi), w in zip(preds, want):
                        r = col.run(lo, hi, strategy)
                        assert r.pair() == w, (b, n, layout, strategy)
                        assert r.blocks_scanned == (n + 1023) // 1024
                col.close()
