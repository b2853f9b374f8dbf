"""Launches as the host makes them, on CPU (the runtime's calls replaced, kernels do nothing).
The autotuner: several candidate shapes run the same kernel in the same way at the
bit-sliced widths, and each launch is timed once, the rule's only as the rule.  Small
columns: cut into tiles of one step of the decode, on one CTA while that holds them."""
import pytest

from tests.test_failed_calls import child  # noqa: F401


@pytest.mark.parametrize("kind", ["branchfree", "branchy", "zone_bf", "zone_br"])
def test_every_launch_is_timed_once(child, kind):  # noqa: F811
    child(f"""
        kind = {kind!r}

        def launch(b, s):
            '''What shape s runs, by the header's words.'''
            branchy = kind in ("branchy", "zone_br")
            sliced = b <= (16 if branchy else 12)
            w = s["warps"]
            fills = sliced or (kind == "branchy" and (b <= 25 or b >= 28) and s["vote_rows"] == 0)
            if fills and w <= 8:
                fit = 226 * 1024 // (s["stages"] * (s["tile_blocks"] * 128 * b + 12))
                w = max(w, 2 * w if fit >= 2 * w else fit // 4 * 4)
            form = () if sliced else (s["vote_rows"], s["vec_lanes"])
            return (w, s["stages"], s["tile_blocks"]) + form

        for b in (1, 5, 8, 10, 12, 13, 16, 17, 21, 24, 27, 32):
            gbscan.autotune_reset()
            c = column(n=5000, b=b)
            c.zonemap_build()
            rule = gbscan.shape_get(b, kind)
            timed = {{launch(b, s) for s in gbscan.shape_candidates(b, kind)}} - {{launch(b, rule)}}
            before = rt.fake_launches()
            r = c.autotune(0, 1, kind, reps=2)
            # a warm-up and two scans of each, then three rounds of the rule and the three fastest
            scans = 3 * len(timed) + 3 * (1 + min(3, len(timed))) * 5
            assert rt.fake_launches() - before == scans * (2 if kind.startswith("zone") else 1), b
            assert r["best"] == rule and r["best_us"] == r["rule_us"], b     # all take the same time here
            assert r["candidates"] == len(gbscan.shape_candidates(b, kind))
    """)


def test_small_columns_are_cut_into_steps_of_their_decode(child):  # noqa: F811
    child("""
        def launched(n, b, layout, strategy):
            c = gbscan.Column.from_packed(x, n, b, layout=layout)
            c.run_async(0, 1, x, strategy)
            return rt.fake_grid(), rt.fake_block_size() // 32

        for strategy in ("branchfree", "branchy"):
            for b, layout in ((8, "lanes"), (16, "lanes"), (20, "lanes"), (5, "rowmajor"), (16, "rowmajor"),
                              (16, "bytes"), (20, "rowmajor")):
                # blocks per step: four lanes a thread, two above 16 bits, one where a lane is a thread's
                sliced = b <= (16 if strategy == "branchy" else 12 if layout == "lanes" else 8 if b in (8, 16) else 15)
                step = 1 if sliced or (layout == "rowmajor" and b & (b - 1)) else 4 if b <= 16 else 2
                for blocks in (1, 3, 4, 7):
                    tiles = -(-blocks // step)
                    assert launched(1024 * blocks, b, layout, strategy) == (1, tiles), (b, layout, strategy, blocks)
                    if tiles < 8:                      # the tail takes a warp of its own
                        assert launched(1024 * blocks + 5, b, layout, strategy) == (1, tiles + 1), (b, layout, strategy)
    """)
