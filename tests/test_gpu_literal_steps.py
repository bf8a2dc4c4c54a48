"""Placement of literals by the literal pass: runs that start, end and cross at
rounds of 32 literals and at the steps the pass takes (two runs and up to 32
literals per token of the window), runs of none, blocks of only literals; the
original bytes are the one correct answer."""
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
    # these few blocks go a warp per stream above; the literal pass itself: the
    # passes as separate calls, and the fused schedule's decodes and seeks
    out.zero_()
    for p in range(3):
        ace.ace_decode_pass(da.idx, p, out, da.total, da.d_scratch, da.scratch_bytes,
                            ace.make_tune(chunk_tokens=window), da.stream)
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy(), data)
    fused = ace.make_tune(chunk_tokens=window, schedule=ace.ACE_SCHEDULE_FUSED)
    out.zero_()
    da.decode_all(out, tune=fused)
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy(), data)
    ace.ace_index_set_tune(da.idx, fused)
    for coord, n in ((30_001, 20_000), (7, 69_000)):
        s = da.seek(coord, n)
        assert da.sync() == ace.ACE_OK
        assert np.array_equal(s.cpu().numpy(), data[coord:coord + n])
    da.close()


@pytest.mark.parametrize("lengths", [(31, 32, 33), (1023, 1024, 1025, 0, 1), (9000,)], ids=str)
def test_blocks_of_several_steps(lengths):
    """The tests' blocks do hold more literals than a step takes, so that runs and
    their shifts pass from step to step."""
    data = _runs(lengths, 70_003, 13 * 1000 + lengths[0])
    arc = ace.ace_encode(data, 13, 6)
    hdr = arc[:64].view(np.uint64)
    entries = arc[int(hdr[4]):int(hdr[4]) + 64 * int(hdr[3])].reshape(-1, 64)
    literals = entries[:, 36:40].copy().view(np.uint32)[:, 0]
    assert (literals > 2 * 32 * 32).any()
