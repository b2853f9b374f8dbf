"""Calls that are in flight together: device encodes on many threads and streams, each
with its own verdict, and scans enqueued one behind the other without a wait between
(zone filters and scans, conjunctive passes: each starts while the kernel before it ends)."""
import threading

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
    return gbscan.load()


def test_concurrent_encodes_each_report_their_own_values():
    """96 calls at a time, more than the encoder has error words, every third with one value
    out of range: each reports its own, and the others' words equal the host encoder's."""
    b, base, calls = 11, 500, 96
    n = [1024 * (1 + i % 7) + i for i in range(calls)]
    vals = [synth.uniform_values(synth.seed_for(61, i), n[i], b, base) for i in range(calls)]
    want = [oracle.pack(v, b, base) for v in vals]
    dev, out = [], []
    for i, v in enumerate(vals):
        t = torch.from_numpy(v.view(np.int32).copy())
        if i % 3 == 0:
            t[(17 * i) % n[i]] = base + (1 << b) if i % 2 else base - 1
        dev.append(t.cuda())
        out.append(torch.empty(gbscan.scan_packed_words(n[i], b), dtype=torch.int32, device="cuda"))
    streams = [torch.cuda.Stream() for _ in range(calls)]
    torch.cuda.synchronize()
    start, problems = threading.Barrier(calls), []

    def work(i):
        start.wait()
        for _ in range(20):
            try:
                gbscan.scan_encode_device(dev[i], n[i], b, base, out[i], streams[i])
                status = gbscan.SCAN_OK
            except gbscan.ScanError as e:
                status = e.status
            if status != (gbscan.SCAN_EINVAL if i % 3 == 0 else gbscan.SCAN_OK):
                problems.append((i, status))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(calls)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not problems
    for i in range(calls):
        if i % 3:
            assert np.array_equal(out[i].cpu().numpy().view(np.uint32), want[i]), i


def test_scans_enqueued_without_a_wait_are_exact():
    n = 700 * 1024 + 333
    widths = (6, 12, 20)
    vals = [synth.clustered_values(synth.seed_for(62, b), n, b, 0.01) for b in widths]
    cols = [gbscan.Column.from_host(v, b) for v, b in zip(vals, widths)]
    for c in cols:
        c.zonemap_build()
    preds = [[synth.pick_range(synth.seed_for(62, b, i), b, s) for b in widths] for i, s in enumerate((0.3, 0.02, 0.9))]
    jobs, want = [], []
    for k in range(30):                       # on one column after the other, on one stream
        pr = preds[k % 3]
        for st in ("zone_bf", "zone_agg_br", "branchfree"):
            c = (k + len(jobs)) % 3
            jobs.append(lambda o, c=c, p=pr[c], st=st: cols[c].run_async(*p, o, st))
            want.append(oracle.scan_values(vals[c], *pr[c]))
        sel = np.ones(n, bool)
        for v, (lo, hi) in zip(vals, pr):
            sel &= (v >= lo) & (v < hi)
        jobs.append(lambda o, q=gbscan.Conj(cols, pr, cols[2]): q.run_async(o))
        want.append((int(sel.sum()), int(vals[2][sel].astype(np.int64).sum())))
    out = torch.zeros((len(jobs), 4), dtype=torch.int64, device="cuda")
    for job, o in zip(jobs, out):
        job(o)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    for i, w in enumerate(want):
        assert (int(got[i, 0]), int(got[i, 1])) == tuple(w), i
    for c in cols:
        c.status()
        c.close()


@pytest.mark.parametrize("ncols", [3, 340, 342, 700])
@pytest.mark.parametrize("spread", [4, 9])
def test_batch_replays_with_new_predicates_are_exact(ncols, spread):
    """One launch and several, small and large descriptor tables (copied before the reset
    of the results, or beside it): replays without a wait between, each with predicates of
    its own."""
    widths = [5 + i % spread for i in range(ncols)]
    vals = [synth.uniform_values(synth.seed_for(63, i), 900 + 37 * (i % 50), b) for i, b in enumerate(widths)]
    cols = [gbscan.Column.from_host(v, b) for v, b in zip(vals, widths)]
    bt = gbscan.Batch(cols)
    out = torch.zeros((4, ncols, 4), dtype=torch.int64, device="cuda")
    preds = [[synth.pick_range(synth.seed_for(63, i, k), b, 0.2 * (k + 1)) for i, b in enumerate(widths)] for k in range(4)]
    for k in range(4):
        bt.run(preds[k], dev_out=out[k], host=False)
    got = out.cpu().numpy()
    for k in range(4):
        for i, v in enumerate(vals):
            assert (int(got[k, i, 0]), int(got[k, i, 1])) == tuple(oracle.scan_values(v, *preds[k][i])), (k, i)
    bt.close()
    for c in cols:
        c.close()
