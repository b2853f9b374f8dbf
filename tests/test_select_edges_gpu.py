"""The select's write pass where it changes form, against the oracle's position lists:
matches around 1024 per 8-block iteration (the stage's size), rows around 20 matches
(the sparse form's most), blocks without a match between others, an odd number of
blocks, ragged tails, widths of both count passes, and truncated capacities."""
import numpy as np
import pytest

import oracle
from paper_2606_22423_gb300 import gbscan

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    import __graft_entry__

    __graft_entry__.build()
    torch.cuda.init()
    gbscan.load()


def column(kind, n, b, rng):
    """Values whose lower half-domain matches: where `hit` is set."""
    i = np.arange(n)
    row, blk = i // 32, i // 1024
    if kind == "near_stage":                 # 127-129 matches per block, evenly spread
        hit = (i % 8 == 0) | ((i % 1024 == 5) & (blk % 3 == 0))
    elif kind == "full_rows":                # rows of 19, 20 and 21 matches among empty ones
        hit = (i % 32 < np.choose(row % 16 % 3, [19, 20, 21])) & (row % 16 < 3)
    elif kind == "one_full_row":             # a row of 32 in an otherwise empty iteration
        hit = (row % 512 == 100)
    elif kind == "some_blocks":
        hit = (blk % 3 == 1) & (rng.random(n) < 0.1)
    elif kind == "sparse":
        hit = rng.random(n) < 0.02
    else:                                    # dense
        hit = rng.random(n) < 0.7
    half = max(1, (1 << b) // 2)
    u = rng.integers(0, half, size=n, dtype=np.uint32)
    return u + np.where(hit, 0, half).astype(np.uint32), half


@pytest.mark.parametrize("b", [1, 2, 5, 8, 9, 12, 13, 16, 24, 32])
@pytest.mark.parametrize("kind", ["near_stage", "full_rows", "one_full_row", "some_blocks", "sparse", "dense"])
def test_positions_match_the_oracle_where_the_write_changes_form(b, kind):
    rng = np.random.default_rng(1000 * b + len(kind))
    for n in (7 * 1024 + 31, 3 * 152 * 1024 + 1):
        v, half = column(kind, n, b, rng)
        col = gbscan.Column.from_host(v, b)
        want, k = oracle.select_packed(oracle.pack(v, b, 0), n, b, 0, 0, half)
        for strategy in ("branchfree", "branchy"):
            for cap in (k + 5, k // 2):
                pos = torch.full((k + 8,), -7, dtype=torch.int32, device="cuda")
                assert col.select(0, half, pos, strategy, capacity=cap) == k
                got = pos.cpu().numpy().view(np.uint32)
                m = min(k, cap)
                assert np.array_equal(got[:m], want[:m]), (b, kind, n, strategy, cap)
                assert (got[m:] == np.uint32(0xFFFFFFF9)).all()        # nothing past the capacity
        col.close()
