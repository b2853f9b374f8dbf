"""How a batch's work is cut into pops, on CPU (the runtime's calls replaced): the number
of pops is read off the size of the table that the plan uploads."""
import pytest

from tests.test_failed_calls import child  # noqa: F401


@pytest.mark.parametrize("b", [2, 8, 12, 16, 20, 32])
def test_pops_of_one_width_keep_within_their_counter(child, b):  # noqa: F811
    """A group's pops go through one counter, some 1.75 ns each: with all warps of the GPU
    on one group they have to take less than half of the group's own time (bytes at 6.7 TB/s
    or values at 10 T/s bit-sliced and 4.3 T/s direct), and, where a zone map leaves out most
    of the blocks, no more than the whole of it.  Equal pops of at least four tiles always did."""
    child(f"""
        b = {b}
        rate = 10e6 if b <= 12 else 4.3e6
        for ncols in (1, 4, 16):
            for n in (1 << 22, 3 << 22, 1 << 24, 5 << 25):
                cols = [column(n=n, b=b) for _ in range(ncols)]
                for c in cols:
                    c.zonemap_build()
                us = ncols * n * max(b / 8 / 6.7e6, 1 / rate)
                for strategy, share in (("branchfree", 0.5), ("branchy", 0.5), ("zone_bf", 1.0)):
                    bt = gbscan.Batch(cols, [strategy] * ncols)
                    pops = rt.fake_copy_bytes() // 8 - 1
                    warps = 152 * 2 * 8
                    # (the pops before the least one is reached: some ln(tiles / warps) per warp and half)
                    assert pops * 1.75e-3 <= share * us + 1.0 or pops <= 2 * warps, (ncols, n, strategy, pops, us)
                    bt.close()
    """)


def test_pops_of_a_given_size_stay_within_a_warps_work(child):  # noqa: F811
    child("""
        b, n = 8, 60_000 * 1024
        tiles = -(-60_000 // gbscan.batch_shape_get(b)["tile_blocks"])
        for per_pop in (1, 7, 1000, 1024, 1025, 1 << 20, (1 << 32) - 1):
            bt = gbscan.Batch([column(n=n, b=b)], tiles_per_pop=per_pop)
            assert rt.fake_copy_bytes() // 8 - 1 == -(-tiles // min(per_pop, 1024)), per_pop
            bt.close()
    """)
