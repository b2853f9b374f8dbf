"""The device encoder at its edges, byte for byte against the oracle's packing: every
width and layout, block counts around a CTA's eight blocks and around one grid of
CTAs, ragged tails, values at both ends of the domain, and the error for a value
outside it wherever it stands in the column."""
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


def packed(layout, v, b, base):
    return oracle.pack(v, b, base) if layout == "lanes" else oracle.pack_rowmajor(v, b, base)


@pytest.mark.parametrize("b", range(1, 33))
def test_device_encoder_matches_the_oracle(b):
    base = min(1234, (1 << 32) - (1 << b))
    top = base + (1 << b) - 1
    for n in (1, 33, 1023, 1024, 7 * 1024 + 1, 8 * 1024, 17 * 1024 + 1000):
        v = synth.uniform_values(synth.seed_for(97, b, n), n, b, base)
        v[0], v[-1] = base, top
        dev = torch.from_numpy(v.view(np.int32)).cuda()
        for layout in ["lanes", "rowmajor"] + (["bytes"] if b in (8, 16, 32) else []):
            col = gbscan.Column.from_device(dev, n, b, base, layout=layout)
            words = gbscan.scan_packed_words(n, b)
            got = torch.empty(words, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            src = torch.as_tensor(_View(col.dev_packed, words), device="cuda")
            got.copy_(src)
            assert np.array_equal(got.cpu().numpy().view(np.uint32), packed(layout, v, b, base)), (b, n, layout)
            del src
            col.close()
    if b < 32:
        n = 9 * 1024 + 5
        for where in (0, 1024, n - 1):
            for bad in ([base - 1] if base else []) + ([top + 1] if top < 0xFFFFFFFF else []):
                v = synth.uniform_values(synth.seed_for(97, b), n, b, base)
                v[where] = bad
                dev = torch.from_numpy(v.view(np.int32)).cuda()
                for layout in ("lanes", "rowmajor"):
                    with pytest.raises(gbscan.ScanError) as e:
                        gbscan.Column.from_device(dev, n, b, base, layout=layout)
                    assert e.value.status == gbscan.SCAN_EINVAL


def test_device_encoder_past_one_grid():
    """More blocks than one grid holds (its CTAs take several)."""
    b, base = 3, 7
    sms = gbscan.scan_launch_shape(b)["sms"]
    n = (16 * sms * 8 + 9) * 1024 + 77
    v = synth.uniform_values(synth.seed_for(98, b), n, b, base)
    dev = torch.from_numpy(v.view(np.int32)).cuda()
    for layout in ("lanes", "rowmajor"):
        col = gbscan.Column.from_device(dev, n, b, base, layout=layout)
        words = gbscan.scan_packed_words(n, b)
        got = torch.as_tensor(_View(col.dev_packed, words), device="cuda").cpu().numpy().view(np.uint32)
        assert np.array_equal(got, packed(layout, v, b, base)), layout
        col.close()


class _View:
    def __init__(self, ptr, words):
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (words,), "typestr": "<i4", "version": 2}
