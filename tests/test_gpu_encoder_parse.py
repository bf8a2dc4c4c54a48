"""The GPU encoder's streams against the oracle's rANS encoder, and its parse,
token by token, against a plain sequential model
of its rules (the earliest stride position of every 16-byte key, chains of
4-byte hashes inside a block, windows of 64 blocks, waves of at most 3, the
shallow preference), at the block sizes and input sizes where windows, bit
map words and chains end."""
import numpy as np
import pytest

import oracle
import synth
import __graft_entry__

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2606_24531_gb300 import ace  # noqa: E402

M64 = (1 << 64) - 1
WIN, HEAD = 64, 192


def _hash16(d, q, bits):
    a = int.from_bytes(d[q:q + 8], "little") * 0x9E3779B97F4A7C15 & M64
    b = int.from_bytes(d[q + 8:q + 16], "little") * 0xC2B2AE3D27D4EB4F & M64
    return ((a ^ ((b << 31 | b >> 33) & M64)) * 0x165667B19E3779F9 & M64) >> (64 - bits)


def _common(d, q, p, limit):
    n = 0
    while n + 64 <= limit and d[q + n:q + n + 64] == d[p + n:p + n + 64]:
        n += 64
    while n < limit and d[q + n] == d[p + n]:
        n += 1
    return n


def _model(data, log2b, mm, chain):
    """Tokens (run, length, source) per block."""
    d, n, B = data.tobytes(), data.size, 1 << log2b
    nb = (n + B - 1) // B
    bits = 10
    while bits < 27 and (1 << bits) < max(1, n // 8):
        bits += 1
    table = {}
    for q in range(0, n - 15, 8):
        table.setdefault(_hash16(d, q, bits), q)
    level, out = [0] * nb, []
    for b in range(nb):
        ws = b // WIN * WIN if b < HEAD else HEAD
        s, e = b * B, min(n, (b + 1) * B)
        prev, head = {}, {}
        for p in range(s, e - 3):
            h = (int.from_bytes(d[p:p + 4], "little") * 2654435761 & 0xFFFFFFFF) >> 20
            prev[p], head[h] = head.get(h), p

        def span(q, want):
            k, got = q >> log2b, 0
            while got < want and (k == b or (k < ws and level[k] < 3)):
                got = min(want, ((k + 1) << log2b) - q)
                k += 1
            return got

        wave, toks, run, p, lv = bytearray(e - s), [], 0, s, 0
        while p < e:
            room, lim = e - p, min(e - p, 32)
            li = le = qi = qe = 0
            if room >= mm:
                q = prev.get(p)
                for _ in range(chain):
                    if q is None:
                        break
                    c = _common(d, q, p, lim)
                    if c > li:
                        li, qi = c, q
                    q = prev.get(q)
                for j in range(8):
                    if p + j + 16 > n:
                        break
                    t = table.get(_hash16(d, p + j, bits))
                    if t is None or t < j or t - j >= p:
                        continue
                    q = t - j
                    c = _common(d, q, p, lim)
                    if q >= s:
                        if c > li or (c == li and q < qi):
                            li, qi = c, q
                        continue
                    c = span(q, c)
                    if c > le or (c == le and q < qe):
                        le, qe = c, q
            best = None
            for q, c, inside in ((qi, li, True), (qe, le, False)):
                if c < mm:
                    continue
                if c == 32:
                    c = _common(d, q, p, room)
                    c = c if inside else span(q, c)
                if c < mm:
                    continue
                lo, hi = max(q, s), min(q + c, p)
                w = 1 + (max(wave[lo - s:hi - s]) if hi > lo else 0)
                if w > 3:
                    continue
                if best is None:
                    take = True
                elif w < best[2]:
                    take = c + max(4, max(c, best[0]) // 8) >= best[0]
                elif w > best[2]:
                    take = c > best[0] + max(4, c // 8)
                else:
                    take = c > best[0] or (c == best[0] and q < best[1])
                if take:
                    best = (c, q, w)
            if best:
                c, q, w = best
                wave[p - s:p - s + c] = bytes([w]) * c
                toks.append((run, c, q))
                if q < s:
                    for k in range(q >> log2b, min((min(q + c, p) - 1) >> log2b, b - 1) + 1):
                        lv = max(lv, level[k] + 1)
                run, p = 0, p + c
            else:
                run, p = run + 1, p + 1
        toks.append((run, 0, 0))
        level[b] = lv
        out.append(toks)
    return out


def _inputs():
    rng = np.random.default_rng(11)
    text = synth.generate("text", 1 << 17, 5)
    period = np.tile(rng.integers(0, 4, 37).astype(np.uint8), 600)
    yield "text, 4 KiB blocks", text[:41_003], 12, 4
    yield "text, one 64 KiB block and a bit", text[:65_536 + 300], 16, 4
    yield "text, 256-byte blocks past three windows", text[:HEAD * 256 + 9_000], 8, 4
    yield "fastq", synth.generate("fastq", 40_000, 6), 13, 16
    yield "mixed, min match 33", synth.generate("mixed", 30_000, 7), 12, 33
    yield "one value", np.full(10_007, 65, np.uint8), 12, 4
    yield "period 37 with changes", np.where(rng.random(period.size) < 0.004, 9, period).astype(np.uint8), 14, 5
    yield "two values", rng.integers(0, 2, 9_001).astype(np.uint8), 10, 6
    for n in (1, 4, 31, 33, 255, 257, 4 * 256 + 31):
        yield "%d bytes" % n, rng.integers(0, 2, n).astype(np.uint8), 8, 4


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("name,data,log2b,mm", list(_inputs()), ids=lambda v: v if isinstance(v, str) else "")
@pytest.mark.parametrize("offset", [0, 3])
def test_parse_equals_the_sequential_model(name, data, log2b, mm, offset):
    """offset: the input's address modulo 16."""
    buf = torch.empty(data.size + 16, dtype=torch.uint8, device="cuda")
    d = buf[offset:offset + data.size]
    d.copy_(torch.from_numpy(np.ascontiguousarray(data)))
    arc = ace.ace_encode_gpu(d, log2b, mm).cpu().numpy()
    want = _model(np.ascontiguousarray(data), log2b, mm, 16)
    for b, toks in enumerate(want):
        run, length, src = oracle.block_tokens(arc, b)[:3]
        got = list(zip(run.tolist(), length.tolist(), src.tolist()))
        assert [t[:2] for t in got] == [t[:2] for t in toks], (name, b)
        assert [t[2] for t in got[:-1]] == [t[2] for t in toks[:-1]], (name, b)
    assert np.array_equal(oracle.decode(arc), data)


def _coded_like_the_oracle(arc):
    hdr = arc[:64].view(np.uint64)
    nb, dir_off, pay = int(hdr[3]), int(hdr[4]), int(hdr[6])
    d = arc[dir_off:dir_off + 64 * nb].reshape(nb, 64)
    offs, sizes, counts = (d[:, a:b].copy().view(t) for a, b, t in
                           ((0, 24, np.uint64), (24, 36, np.uint32), (36, 48, np.uint32)))
    for b in range(nb):
        for k in range(3):
            if not counts[b, k]:
                assert sizes[b, k] == 0
                continue
            p = arc[pay + int(offs[b, k]):pay + int(offs[b, k]) + int(sizes[b, k])]
            present = np.unpackbits(p[128:160], bitorder="little").astype(bool)
            freq = np.zeros(256, np.uint16)
            n = int(present.sum())
            freq[present] = p[160:160 + 2 * n].view(np.uint16)
            head = 160 + ((2 * n + 15) & ~15)
            sym = oracle.rans_decode(p[head:], p[:128].view(np.uint32), freq, int(counts[b, k]))
            assert np.array_equal(oracle.rans_freqs(sym), freq), (b, k)
            states, body = oracle.rans_encode(sym, freq)
            assert np.array_equal(states, p[:128].view(np.uint32)) and np.array_equal(body, p[head:]), (b, k)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 95, 96, 97, 128, 256, 700])
@pytest.mark.parametrize("values", [1, 3, 256])
def test_streams_equal_the_oracles_encoder(n, values):
    """Literal streams around the coder's rounds of 32 and its loads ahead,
    one value (frequency 4096) to all 256 (pushes of two bytes)."""
    rng = np.random.default_rng(n * 1000 + values)
    x = np.minimum(rng.integers(0, values, n), rng.integers(0, values, n)).astype(np.uint8)
    arc = ace.ace_encode_gpu(torch.from_numpy(x).cuda(), 10, 200).cpu().numpy()  # no matches
    assert np.array_equal(oracle.decode(arc), x)
    _coded_like_the_oracle(arc)
