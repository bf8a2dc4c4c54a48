"""Placement of literals by the literal pass: runs that start, end and cross at
rounds of 32 literals and at the steps the pass takes (two runs and up to 32
literals per token of the window), runs of none, blocks of only literals; the original bytes are
the one correct answer."""
import numpy as np
import pytest

import oracle
import __graft_entry__

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2606_24531_gb300 import ace  # noqa: E402
from paper_2606_24531_gb300.archive import DeviceArchive  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _runs(lengths, total, seed):
    """Random literal runs of the given lengths, each followed by a copy of
    earlier bytes (several copies in a row for a run of none)."""
    rng = np.random.default_rng(seed)
    out, k = [rng.integers(0, 256, 64).astype(np.uint8)], 0
    size = 64
    while size < total:
        n = lengths[k % len(lengths)]
        run = rng.integers(0, 256, n).astype(np.uint8)
        out.append(run)
        size += n
        flat = np.concatenate(out[-40:])
        m = int(rng.integers(8, 40))
        at = int(rng.integers(0, max(1, flat.size - m)))
        out.append(flat[at:at + m].copy())
        size += out[-1].size
        k += 1
    return np.concatenate(out)[:total]


@pytest.mark.parametrize("window", [32, 128, 256])
@pytest.mark.parametrize("log2b", [8, 13, 16])
@pytest.mark.parametrize("lengths", [(0, 1, 2), (31, 32, 33), (127, 128, 129), (511, 512, 513), (1023, 1024, 1025, 0, 1),
                                     (4095, 4096, 4097), (9000,)], ids=str)
def test_runs_at_rounds_and_steps(lengths, log2b, window):
    data = _runs(lengths, 70_003, log2b * 1000 + lengths[0])
    arc = ace.ace_encode(data, log2b, 6)
    da = DeviceArchive(arc, max_seek_blocks=400)
    out = da.decode_all(tune=ace.make_tune(chunk_tokens=window))
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy(), data)
    ace.ace_index_set_tune(da.idx, ace.make_tune(chunk_tokens=window))
    s = da.seek(30_001, 20_000)
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(s.cpu().numpy(), oracle.seek(arc, 30_001, 20_000))
    da.close()
