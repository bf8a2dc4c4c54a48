"""The match pass's three ways through a block -- a CTA, a warp by rows, a warp
by rounds -- on matches where they can go wrong: lengths around the rows' limit
and the bit map's, every overlap, long runs (deep chains of copies), sources in
the same rows, sources across block and window boundaries, few and many
matches per block; the original bytes are the one correct answer."""
import numpy as np
import pytest

import oracle
import synth
import __graft_entry__

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2606_24531_gb300 import ace  # noqa: E402
from paper_2606_24531_gb300.archive import DeviceArchive  # noqa: E402
from paper_2606_24531_gb300.batch import DeviceBatch  # noqa: E402
from paper_2606_24531_gb300.serve import SeekCache  # noqa: E402
from conftest import with_dep_removed  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    torch.cuda.set_device(0)


def _copies(lengths, back, lit, total, seed):
    """lit random bytes, then a copy of the given length from at most back
    bytes earlier, in turn."""
    rng = np.random.default_rng(seed)
    out = bytearray(rng.integers(0, 256, 300).astype(np.uint8).tobytes())
    k = 0
    while len(out) < total:
        out += rng.integers(0, 256, int(rng.integers(0, lit + 1))).astype(np.uint8).tobytes()
        n = lengths[k % len(lengths)]
        d = int(rng.integers(1, min(back, len(out)) + 1))
        for _ in range(n):  # overlapping copies repeat
            out.append(out[-d])
        k += 1
    return np.frombuffer(bytes(out[:total]), np.uint8)


SHAPES = {
    "short, recent sources": ((5, 6, 9, 13), 60, 3),
    "around the rows' limit": ((31, 32, 33, 63, 64, 65), 4000, 40),
    "every overlap": (tuple(range(4, 70)), 70, 2),
    "runs": ((700, 3000), 9, 20),
    "a run of one value": ((40000,), 1, 1),
    "long": ((900, 2047, 2048, 2049, 5000), 30000, 300),
    "few": ((20, 40), 8000, 1500),
}


def _check(da, data):
    out = da.decode_all()
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy()[:data.size], data)


@pytest.mark.parametrize("log2b", [8, 10, 12, 14, 16])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_levels_seeks_batches_and_caches(shape, log2b):
    lengths, back, lit = SHAPES[shape]
    data = _copies(lengths, back, lit, 150_001, log2b)
    # the encoders' archives (few levels) and the oracle's (deep chains of blocks)
    arcs = [ace.ace_encode(data, log2b, 4), oracle.encode(data[:60_001], log2b, 4, 16)]
    datas = [data, data[:60_001]]
    for arc, d in zip(arcs, datas):
        da = DeviceArchive(arc, max_seek_blocks=700)
        _check(da, d)
        for coord, n in ((0, 1), (d.size - 5001, 5001), (d.size // 3, 20_000)):
            s = da.seek(coord, n)
            assert da.sync() == ace.ACE_OK
            assert np.array_equal(s.cpu().numpy(), d[coord:coord + n]), (coord, n)
        if log2b >= 10:
            cache = SeekCache([da], 800, 8, 1 << 17)
            for got, (coord, n) in zip(cache.seek_many([(0, 100, 30_000), (0, 40_000, 9_999)]), ((100, 30_000), (40_000, 9_999))):
                assert np.array_equal(got.cpu().numpy(), d[coord:coord + n])
            cache.close()
        da.close()
    db = DeviceBatch(arcs)
    db.decode()
    assert db.sync() == ace.ACE_OK
    for i, d in enumerate(datas):
        assert np.array_equal(db.output(i).cpu().numpy(), d)
    db.close()


@pytest.mark.parametrize("shape", ["short, recent sources", "around the rows' limit", "long", "every overlap"])
def test_levels_of_many_blocks(shape):
    """More blocks in a level than get a CTA each: the warp-per-block kernels
    (rows or rounds by the archive's matches) and the dense CTA kernel."""
    lengths, back, lit = SHAPES[shape]
    piece = _copies(lengths, back, lit, 1 << 20, 5)
    for thin in (0, 1, 2):  # fewer matches per 16 KiB each time
        rng = np.random.default_rng(thin)
        rows = [piece]
        for k in range(6):
            if thin:
                noise = rng.integers(0, 256, (1 << 20) * thin * 3).astype(np.uint8)
                rows.append(noise)
            rows.append(np.roll(piece, 4096 * k + k))
        data = np.concatenate(rows)
        arc = ace.ace_encode_gpu(torch.from_numpy(data).cuda(), 12, 4).cpu().numpy()
        da = DeviceArchive(arc)
        _check(da, data)
        da.close()


@pytest.mark.parametrize("off_width", [4, 5])
@pytest.mark.parametrize("log2b", [8, 12, 14, 16, "long"])
def test_match_pass_over_the_records_of_a_whole_decode(log2b, off_width):
    """A whole decode of few blocks leaves records with the literals before each
    match beside its source; the match pass by itself reads the same sources, by
    a CTA per block and (long: 1100 blocks, most of a level) by a warp per block."""
    if log2b == "long":
        piece = np.random.default_rng(7).integers(0, 256, 40_000).astype(np.uint8)
        data = np.concatenate([np.roll(piece, 1500 * k) for k in range(113)])[:1100 << 12]
        arc = ace.ace_encode_gpu(torch.from_numpy(data).cuda(), 12, 16, off_width=off_width).cpu().numpy()
    else:
        lengths, back, lit = SHAPES["every overlap"]
        data = _copies(lengths, back, lit, 30_001, log2b)
        arc = ace.ace_encode(data, log2b, 4, off_width=off_width)
    da = DeviceArchive(arc)
    out = da.decode_all()
    ace.ace_decode_pass(da.idx, 2, out, out.numel(), da.d_scratch, da.scratch_bytes, None, da.stream)
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy(), data)
    if log2b == "long":  # the sizes the case is for
        levels = ace.ace_index_levels(da.idx, da.info["n_levels"])
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        assert max(levels) > 4 * sms and da.info["n_blocks"] <= 8 * sms and arc.size < data.size // 4
    da.close()


def test_batches_of_either_size():
    """A batch that decodes a stream per warp and one, above 128 MiB, in three
    passes: blocks of every size, objects of a block and of many."""
    arcs, datas = [], []
    for k, log2b in enumerate((9, 12, 14, 16)):
        lengths, back, lit = SHAPES[sorted(SHAPES)[k]]
        for n in (77, 40_000, 700_001):
            datas.append(_copies(lengths, back, lit, n, k))
            arcs.append(ace.ace_encode(datas[-1], log2b, 4))
    per = sum(d.size for d in datas)
    for copies in (1, (128 << 20) // per + 2):
        db = DeviceBatch(arcs * copies)
        db.decode()
        assert db.sync() == ace.ACE_OK
        for k in range(len(datas)):
            want = torch.from_numpy(datas[k].copy()).cuda()
            for c in {0, copies // 2, copies - 1}:
                assert torch.equal(db.output(c * len(datas) + k), want)
        db.close()


@pytest.mark.parametrize("profile, log2b, size", [
    ("genome", 8, 300_000), ("fastq", 12, 900_000), ("genome", 16, 3_600_001),  # many blocks, few matches: a warp per block
    ("fastq", 15, 150_000), ("genome", 9, 20_001),                              # few blocks: a warp per stream
    ("text", 10, 700_000), ("mixed", 13, 2_400_000),                            # many blocks of many matches: a CTA per block
    ("text", 16, 900_000), ("mixed", 12, 90_000)])                              # few blocks: a warp per stream
def test_batch_routes(profile, log2b, size):
    """Every way a batch's passes take, on objects of one profile, and the same
    batch again (its epoch moved on)."""
    datas = [synth.generate(profile, size - 1009 * k, 31 * k + log2b) for k in range(12)]
    mm = {"genome": 20, "fastq": 16}.get(profile, 4)
    arcs = [ace.ace_encode_gpu(torch.from_numpy(d).cuda(), log2b, mm).cpu().numpy() for d in datas]
    db = DeviceBatch(arcs)
    for _ in range(2):
        db.out.zero_()
        db.decode()
        assert db.sync() == ace.ACE_OK
        for k, d in enumerate(datas):
            assert torch.equal(db.output(k), torch.from_numpy(d).cuda())
    db.close()


def test_batch_by_warps_reports_a_source_outside_its_levels():
    data = synth.generate("genome", 2_500_000, 3)
    arc = ace.ace_encode(data, 12, 20)
    bad = with_dep_removed(arc, int(np.nonzero(oracle.levels(arc) == 2)[0][-1]))  # it reads a block of level 1
    db = DeviceBatch([arc, bad])
    db.decode()
    assert db.sync() == ace.ACE_E_CORRUPT
    db.close()


@pytest.mark.parametrize("profile, log2b, size", [("text", 8, 120_000), ("fastq", 10, 700_000), ("fastq", 13, 500_000),
                                                  ("fastq", 14, 700_000), ("mixed", 9, 60_000)])
def test_whole_decodes_of_many_levels(profile, log2b, size):
    """Archives of more than 32 levels (the oracle takes the most recent
    sources), by warps and by CTAs waiting on one another's blocks; a block
    that reads past its levels is reported."""
    data = synth.generate(profile, size, 17 * log2b)
    arc = oracle.encode(data, log2b, {"fastq": 16}.get(profile, 4), 16)
    da = DeviceArchive(arc)
    assert da.info["n_levels"] > 32
    for _ in range(2):
        _check(da, data)
    bad = DeviceArchive(with_dep_removed(arc, int(np.argmax(oracle.levels(arc)))))
    bad.decode_all()
    assert bad.sync() == ace.ACE_E_CORRUPT
    da.close()
    bad.close()


@pytest.mark.parametrize("profile, mm", [("text", 4), ("text", 12), ("fastq", 16), ("genome", 20)])
@pytest.mark.parametrize("log2b", [8, 9, 10, 11, 12, 13, 14, 15, 16])
def test_levels_of_many_blocks_at_every_size(profile, mm, log2b):
    """More than four blocks per SM in a level where the size allows it: a CTA of
    32 to 256 threads per dense block, rows, rounds; and few blocks, in few levels
    and in many, with and without a warp per stream."""
    n = min(5000 << log2b, 24 << 20) - 7
    data = synth.generate(profile, n, log2b)
    da = DeviceArchive(ace.ace_encode_gpu(torch.from_numpy(data).cuda(), log2b, mm).cpu().numpy())
    _check(da, data)
    da.close()
    small = data[:26 << log2b]
    for arc in (ace.ace_encode(small, log2b, mm), oracle.encode(small, log2b, mm, 16)):
        da = DeviceArchive(arc)
        _check(da, small)
        da.close()


@pytest.mark.parametrize("log2b", [8, 12, 14, 16])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_fused_schedule(shape, log2b):
    """A match of up to 32 bytes by one lane in 8-byte words, at every length,
    alignment and overlap of the shapes, in whole decodes, seeks and batches."""
    lengths, back, lit = SHAPES[shape]
    data = _copies(lengths, back, lit, 90_001, 7 * log2b)
    arc = ace.ace_encode(data, log2b, 4)
    fused = ace.make_tune(schedule=ace.ACE_SCHEDULE_FUSED)
    da = DeviceArchive(arc, max_seek_blocks=400)
    out = da.decode_all(tune=fused)
    assert da.sync() == ace.ACE_OK
    assert np.array_equal(out.cpu().numpy(), data)
    ace.ace_index_set_tune(da.idx, fused)
    for coord, n in ((0, 1), (31_007, 20_002), (data.size - 5001, 5001)):
        s = da.seek(coord, n)
        assert da.sync() == ace.ACE_OK
        assert np.array_equal(s.cpu().numpy(), data[coord:coord + n])
    da.close()
    db = DeviceBatch([arc, arc], tune=fused)
    db.decode()
    assert db.sync() == ace.ACE_OK
    assert all(np.array_equal(db.output(k).cpu().numpy(), data) for k in range(2))
    db.close()
