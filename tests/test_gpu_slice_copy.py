"""The bytes a seek and a cached seek hand out, for every alignment of the
range against the place it is written to, and every short length: exactly the
range, and nothing beside it."""
import numpy as np
import pytest

import synth
import __graft_entry__

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2606_24531_gb300 import ace  # noqa: E402
from paper_2606_24531_gb300.archive import DeviceArchive  # noqa: E402
from paper_2606_24531_gb300.serve import SeekCache  # noqa: E402

B = 4096


@pytest.fixture(scope="module")
def resident():
    __graft_entry__.build()
    torch.cuda.set_device(0)
    data = synth.generate("mixed", 40 * B + 77, 12)
    da = DeviceArchive(ace.ace_encode(data, 12, 4), max_seek_blocks=64)
    yield data, da
    da.close()


def _ranges(n):
    for r in range(17):
        for length in (1, 2, 15, 16, 17, 31, 33, 2048 + r, B - r, B, B + 1, 3 * B + 5):
            yield 5 * B - 20 + r, length
    yield 0, n
    yield n - 1, 1


@pytest.mark.parametrize("shift", [0, 1, 7, 15])
def test_seek_writes_exactly_the_range(resident, shift):
    data, da = resident
    buf = torch.empty(data.size + 64, dtype=torch.uint8, device="cuda")
    for coord, length in _ranges(data.size):
        buf.fill_(0xA5)
        da.seek(coord, length, buf[16 + shift:16 + shift + length])
        assert da.sync() == ace.ACE_OK
        got = buf.cpu().numpy()
        assert np.array_equal(got[16 + shift:16 + shift + length], data[coord:coord + length]), (coord, length)
        assert (got[:16 + shift] == 0xA5).all() and (got[16 + shift + length:] == 0xA5).all(), (coord, length)


@pytest.mark.parametrize("requests", [1, 3, 40, 204])
def test_cached_seeks_write_exactly_their_ranges(resident, requests):
    """Batches of few and of many requests (their CTAs per request differ),
    results packed without gaps at any alignment."""
    data, da = resident
    ranges = list(_ranges(data.size))
    cache = SeekCache([da], 64, 256, 1 << 20)
    for k in range(0, len(ranges), max(requests, len(ranges) // 6 + 1)):
        part = ranges[k:k + requests]
        r = np.zeros(len(part), ace.SEEK_REQ)
        r["coord"], r["len"] = zip(*part)
        r["out_off"][1:] = np.cumsum(r["len"])[:-1]
        r["out_off"] += 3
        cache.pool.fill_(0xA5)
        torch.cuda.synchronize()
        cache.run_batch(r)
        got = cache.pool.cpu().numpy()
        want = np.concatenate([data[c:c + n] for c, n in part])
        assert np.array_equal(got[3:3 + want.size], want)
        assert (got[:3] == 0xA5).all() and (got[3 + want.size:] == 0xA5).all()
    cache.close()
