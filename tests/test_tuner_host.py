"""What the autotuner times, on CPU (the runtime's calls replaced, kernels do nothing):
several candidate shapes run the same kernel in the same way at the bit-sliced widths, and
each launch is timed once, the rule's only as the rule."""
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
