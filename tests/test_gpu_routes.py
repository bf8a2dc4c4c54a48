"""Calls on both sides of every size at which another way through the passes
begins: the blocks a seek covers, a cached batch's blocks and requests, the
blocks of a whole decode.  The original bytes are the one correct answer."""
import numpy as np
import pytest

import oracle
import synth
import __graft_entry__

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2606_24531_gb300 import ace  # noqa: E402
from paper_2606_24531_gb300.archive import DeviceArchive  # noqa: E402
from paper_2606_24531_gb300.batch import DeviceBatch, autotune  # noqa: E402
from paper_2606_24531_gb300.serve import SeekCache  # noqa: E402

MM = {"fastq": 16, "genome": 20, "text": 4, "mixed": 4}


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _blocks(size, log2b):
    return (size + (1 << log2b) - 1) >> log2b


def _archive(profile, n, log2b, seed=3, **kw):
    data = synth.generate(profile, n, seed)
    arc = ace.ace_encode_gpu(torch.from_numpy(data).cuda(), log2b, MM[profile]).cpu().numpy()
    return data, DeviceArchive(arc, **kw)


@pytest.mark.parametrize("profile", sorted(MM))
@pytest.mark.parametrize("log2b, blocks", [(8, (1, 32, 33, 1024, 1025, 3000)), (12, (1, 32, 33, 48, 49, 1024, 1025)),
                                           (14, (1, 32, 33, 48, 49)), (15, (1, 5, 33)), (16, (1, 3, 33))])
def test_seeks_of_every_length(profile, log2b, blocks):
    B = 1 << log2b
    data, da = _archive(profile, (max(blocks) + 40) * B + 77, log2b, max_seek_blocks=max(blocks) + 300)
    for n in blocks:
        for coord, length in ((17 * B, n * B), (11 * B + 5, n * B - 5), (30 * B + 3, (n - 1) * B + 1)):  # n blocks each
            for _ in range(2):
                out = da.seek(coord, length)
                assert da.sync() == ace.ACE_OK
                assert np.array_equal(out.cpu().numpy(), data[coord:coord + length]), (n, coord)
    da.close()


@pytest.mark.parametrize("profile, log2b, size", [("text", 8, 120_000), ("fastq", 10, 700_000), ("fastq", 12, 600_000),
                                                  ("fastq", 13, 500_000), ("text", 12, 300_000), ("fastq", 16, 700_000)])
def test_seeks_in_many_levels(profile, log2b, size):
    data = synth.generate(profile, size, 17 * log2b)
    arc = oracle.encode(data, log2b, MM[profile], 16)
    nb = (size + (1 << log2b) - 1) >> log2b
    da = DeviceArchive(arc, max_seek_blocks=nb)
    for coord, length in ((size - 9000, 9000), (size // 2, 1), (size // 3, 50_001), (0, size)):
        out = da.seek(coord, length)
        assert da.sync() == ace.ACE_OK
        assert np.array_equal(out.cpu().numpy(), data[coord:coord + length])
    da.close()


@pytest.mark.parametrize("log2b, nb", [(8, 6000), (13, 2500)])  # by warps, by CTAs
def test_long_seek_in_a_chain_of_blocks(log2b, nb):
    """Each block reads the one before it, over more blocks than are resident at
    once: blocks are handed out before those that wait for them."""
    B = 1 << log2b
    rng = np.random.default_rng(8)
    data = np.empty(nb * B, np.uint8)
    data[:B] = rng.integers(0, 256, B)
    for k in range(1, nb):
        data[k * B:(k + 1) * B] = data[(k - 1) * B:k * B]
        data[k * B + int(rng.integers(0, B))] ^= 1 + int(rng.integers(0, 255))
    arc = oracle.encode(data, log2b, 8, 16)
    da = DeviceArchive(arc, max_seek_blocks=nb)
    assert da.info["n_levels"] > 2000
    out = da.seek(data.size - 700, 700)
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy(), data[-700:])
    out = da.decode_all()
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy(), data)
    da.close()


@pytest.mark.parametrize("blocks", [3071, 3072, 3073, 5000])
def test_cached_batches_by_blocks(blocks):
    B = 256
    pairs = [_archive(p, 900_000, 8, seed=k) for k, p in enumerate(("text", "genome"))]
    cache = SeekCache([da for _, da in pairs], 9000, 320, 4 << 20)
    n = 50
    lens = np.full(n, (blocks // n - 1) * B + 100, np.uint64)  # counted as len / B + 1
    lens[:blocks - n * (blocks // n)] += B
    assert int((lens // B + 1).sum()) == blocks
    arcs = np.arange(n, dtype=np.uint32) % 2
    coords = (np.arange(n, dtype=np.uint64) * 15_013) % np.uint64(900_000 - int(lens.max()))
    for _ in range(2):
        r = cache.plan_arrays(arcs, coords, lens)
        cache.run_batch(r)
        for k in range(n):
            c, ln = int(coords[k]), int(lens[k])
            assert np.array_equal(cache.result(r, k).cpu().numpy(), pairs[int(arcs[k])][0][c:c + ln])
        cache.reset()
    cache.close()


@pytest.mark.parametrize("n", [1, 64, 65, 200])
def test_cached_batches_of_device_requests(n):
    pairs = [_archive(p, 1_500_000, 12, seed=k) for k, p in enumerate(("mixed", "fastq", "genome"))]
    cache = SeekCache([da for _, da in pairs], 2000, max(n, 64), 4 << 20)
    rng = np.random.default_rng(n)
    lens = rng.integers(1, 20_000, n).astype(np.uint64)
    coords = (rng.random(n) * (1_500_000 - 20_000)).astype(np.uint64)
    arcs = rng.integers(0, 3, n).astype(np.uint32)
    r = cache.plan_arrays(arcs, coords, lens)
    d = torch.from_numpy(r.view(np.uint8).copy()).cuda()
    torch.cuda.synchronize()
    for _ in range(2):
        ace.ace_seek_batch(cache.cache, d, n, cache.pool, cache.pool_bytes, cache.stream)
        assert cache.sync() == ace.ACE_OK
        for k in range(n):
            c, ln = int(coords[k]), int(lens[k])
            assert np.array_equal(cache.result(r, k).cpu().numpy(), pairs[int(arcs[k])][0][c:c + ln])
    cache.close()


@pytest.mark.parametrize("profile, log2b, per_sm", [("fastq", 12, 1), ("fastq", 14, 1), ("text", 9, 8), ("genome", 12, 8),
                                                    ("mixed", 12, 8), ("text", 16, 1)])
def test_whole_decodes_by_blocks(profile, log2b, per_sm):
    limit = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    for nb in (limit - 1, limit, limit + 1):
        data, da = _archive(profile, nb << log2b, log2b, seed=nb)
        out = da.decode_all()
        assert da.sync() == ace.ACE_OK
        assert np.array_equal(out.cpu().numpy(), data)
        da.close()


@pytest.mark.parametrize("copy_width", [8, 16])
def test_copy_widths_of_many_blocks(copy_width):
    """Where a warp resolves a block's matches: levels of more than four blocks
    per SM by rounds and by rows, fused seeks, batches of few matches."""
    tune = ace.make_tune(copy_width=copy_width)
    for profile in ("genome", "fastq"):
        data, da = _archive(profile, 6_000_001, 12, seed=9, max_seek_blocks=600)
        out = da.decode_all(tune=tune)
        assert da.sync() == ace.ACE_OK
        assert np.array_equal(out.cpu().numpy(), data)
        ace.ace_index_set_tune(da.idx, ace.make_tune(schedule=ace.ACE_SCHEDULE_FUSED, copy_width=copy_width))
        s = da.seek(5_000_003, 700_001)
        assert da.sync() == ace.ACE_OK
        assert np.array_equal(s.cpu().numpy(), data[5_000_003:5_700_004])
        db = DeviceBatch([da.d_arc.cpu().numpy()] * 2, tune=tune)
        db.decode()
        assert db.sync() == ace.ACE_OK
        assert np.array_equal(db.output(1).cpu().numpy(), data)
        db.close()
        da.close()


@pytest.mark.parametrize("profile, log2b, size", [("text", 8, 340_000), ("text", 12, 6_000_000), ("fastq", 12, 4_000_000),
                                                  ("genome", 12, 6_000_000)])
def test_corrupt_payloads_in_the_passes(profile, log2b, size):
    """A flipped payload bit, in decodes, seeks and batches that take the token,
    literal and match passes: reported, or the bytes the oracle decodes from the
    same archive."""
    data = synth.generate(profile, size, 13)
    arc = ace.ace_encode(data, log2b, MM[profile])
    payload_off = int(arc[48:56].view(np.uint64)[0])
    rng = np.random.default_rng(log2b)
    seen = set()
    for trial in range(8):
        bad = arc.copy()
        bad[int(rng.integers(payload_off, bad.size))] ^= np.uint8(1 << int(rng.integers(0, 8)))
        ref = None
        da = DeviceArchive(bad, max_seek_blocks=_blocks(size, log2b))
        ace.ace_index_set_tune(da.idx, ace.make_tune(wait_timeout_ns=50_000_000))
        db = DeviceBatch([bad, arc], tune=ace.make_tune(wait_timeout_ns=50_000_000))
        db.decode()
        got = [(lambda o: (da.sync(), o))(da.decode_all()), (lambda o: (da.sync(), o))(da.seek(0, size)),
               (db.sync(), db.output(0))]
        for st, out in got:
            assert st in (ace.ACE_OK, ace.ACE_E_CORRUPT), ace.ace_status_str(st)
            seen.add(st)
            if st == ace.ACE_OK:
                ref = oracle.decode(bad) if ref is None else ref
                assert np.array_equal(out.cpu().numpy()[:size], ref)
        db.close()
        da.close()
    assert ace.ACE_E_CORRUPT in seen


def test_autotune_times_each_launch_once():
    """A batch decoded a stream per warp has one launch under the pass schedule,
    and reports it; one of many blocks has the candidates' own."""
    for size, one in ((60_000, True), (9_000_000, False)):
        data = synth.generate("text", size, 2)
        arc = ace.ace_encode(data, 12, 4)
        db = DeviceBatch([arc, arc])
        shape = db.retune()
        assert (shape["window"] == 0) == one
        if one:
            assert (shape["grid"], shape["warps_per_cta"]) == ((2 * 3 * 15 + 3) // 4, 4)
        best = autotune(db, reps=1, cache_key=None)
        rows = [r for r in best["sweep"] if r["schedule"] == ace.ACE_SCHEDULE_PASSES]
        assert len(rows) == (1 if one else 24)
        db.out.zero_()
        db.decode()
        assert db.sync() == ace.ACE_OK
        assert np.array_equal(db.output(1).cpu().numpy(), data)
        db.close()
