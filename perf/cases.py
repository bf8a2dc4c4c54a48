"""The workloads whose speed counts: what users of the library have it do,
through its public entry points, from single small calls to whole-genome
decodes.  Inputs are seeded and made on the GPU, with the shapes of the four
profiles of the synth module (FASTQ records, a repetitive genome, Zipf text,
text with copied spans) and the encoder parameters the benchmark uses for
them; archives come from the GPU encoder.

A case is a dict: "op" (what is called), "profile", "size" in bytes,
"log2b" (block size 2^log2b), "adaptive" and "off_width" (encoder options),
and per op its counts.
"""
import numpy as np
import torch

from paper_2606_24531_gb300 import ace
from paper_2606_24531_gb300.archive import DeviceArchive
from paper_2606_24531_gb300.batch import DeviceBatch
from paper_2606_24531_gb300.serve import SeekCache

MIN_MATCH = {"fastq": 16, "genome": 20, "text": 4, "mixed": 4}
# decompressed over compressed size of the profiles at 16 KiB blocks
RATIO = {"fastq": 1.87, "genome": 20.0, "text": 2.2, "mixed": 2.3}
PROFILES = ("fastq", "genome", "text", "mixed")
KIB, MIB = 1 << 10, 1 << 20


def _case(name, op, profile, size, log2b=14, adaptive=False, off_width=0, count=0, length=0):
    c = {"op": op, "profile": profile, "size": size, "log2b": log2b, "adaptive": adaptive, "off_width": off_width,
         "count": count, "length": length}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small resident document decoded whole: launches and latency
        _case("decode_text_37KiB", "decode", "text", 37 * KIB + 411, 12),
        # the plain small configuration: 64 blocks, fewer than the GPU has SMs
        _case("decode_mixed_1MiB", "decode", "mixed", MIB),
        # a text collection: short matches, records as large as the output
        _case("decode_text_128MiB", "decode", "text", 128 * MIB),
        # the headline configuration: sequencing reads, mostly literals
        _case("decode_fastq_256MiB", "decode", "fastq", 256 * MIB),
        # the largest resident archive: long matches
        _case("decode_genome_1GiB", "decode", "genome", 1024 * MIB),
        # an archive that has just arrived in host memory (odd size, 4 KiB
        # blocks, streams stored where coding does not pay, 5-byte offsets):
        # upload, index, whole decode, status
        _case("open_mixed_24MiB", "open", "mixed", 24 * MIB + 4097, 12, True, 5),
        # random access: one unaligned 16 KiB range, with its status
        _case("seek_fastq_16KiB", "seek", "fastq", 128 * MIB, length=16 * KIB),
        # a range of 1001 blocks of a genome
        _case("seek_genome_16MiB", "seek", "genome", 192 * MIB, length=1001 * 16 * KIB),
        # seek serving through the block cache: two batches of requests of
        # 16 KiB to 1 MiB over four archives, more blocks than the cache holds
        _case("serve_128_requests", "serve", "all", 32 * MIB, count=128),
        # many uneven objects (4 KiB to 4 MiB, four profiles, three block
        # sizes) in one batched decode
        _case("batch_192_objects", "batch", "all", 4 * MIB, count=192),
        # archives written on the GPU: sequencing reads, and text of odd size
        _case("encode_fastq_64MiB", "encode", "fastq", 64 * MIB),
        _case("encode_text_11MiB", "encode", "text", 11 * MIB + 777),
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(lo * (hi / lo) ** rng.random())))


def draw(rng):
    op = rng.choice(("decode", "decode", "decode", "open", "seek", "seek", "serve", "batch", "encode", "encode"))
    profile = rng.choice(PROFILES)
    log2b = rng.choice((12, 14, 14, 16))
    adaptive, off_width = rng.random() < 0.3, rng.choice((0, 0, 5))
    if op == "decode":
        size = _log_uniform(rng, 4 * KIB, (512 if profile == "genome" else 192) * MIB)
        return _case("", op, profile, size, log2b, adaptive, off_width)
    if op == "open":
        return _case("", op, profile, _log_uniform(rng, 64 * KIB, 48 * MIB), log2b, adaptive, off_width)
    if op == "seek":
        size = _log_uniform(rng, 2 * MIB, 160 * MIB)
        return _case("", op, profile, size, log2b, adaptive, off_width,
                     length=_log_uniform(rng, 1, min(size // 2, 16 * MIB)))
    if op == "serve":
        return _case("", op, "all", _log_uniform(rng, 8 * MIB, 32 * MIB), log2b, adaptive, off_width,
                     count=_log_uniform(rng, 4, 128))
    if op == "batch":
        return _case("", op, "all", _log_uniform(rng, 64 * KIB, 4 * MIB), 0, adaptive, off_width,
                     count=_log_uniform(rng, 8, 192))
    size = _log_uniform(rng, 64 * KIB, (9 if profile in ("text", "mixed") else 48) * MIB)
    return _case("", op, profile, size, log2b, adaptive, off_width)


# ------------------------------------------------------------------- inputs

def _text(n, g):
    """Zipf(1.1) words of a 5,000-word vocabulary, each followed by a space."""
    dev, vocab = g.device, 5000
    length = torch.randint(2, 11, (vocab,), generator=g, device=dev)
    chars = torch.randint(97, 123, (vocab, 11), generator=g, device=dev, dtype=torch.uint8)
    chars.scatter_(1, length[:, None], 32)
    p = torch.arange(1, vocab + 1, device=dev, dtype=torch.float64) ** -1.1
    cdf = (p.cumsum(0) / p.sum()).float()
    parts, have = [], 0
    while have < n:
        m = min((n - have) // 5 + 64, 1 << 23)
        w = torch.searchsorted(cdf, torch.rand(m, generator=g, device=dev)).clamp_(max=vocab - 1)
        ln = length[w] + 1
        start = ln.cumsum(0) - ln
        k = torch.repeat_interleave(torch.arange(m, device=dev), ln)
        part = chars[w[k], torch.arange(k.numel(), device=dev) - start[k]]
        parts.append(part)
        have += part.numel()
    return torch.cat(parts)[:n].contiguous()


def _mixed(n, g):
    """Text in which two bytes in five belong to copies of earlier spans of
    32 to 512 bytes (copies of copies among them)."""
    dev = g.device
    out = _text(n, g)
    m = n // 600 + 8
    fresh = torch.randint(208, 609, (m,), generator=g, device=dev)
    copy = torch.randint(32, 513, (m,), generator=g, device=dev)
    fresh[0] += 512
    at = (fresh + copy).cumsum(0) - copy  # where each copy starts
    src = (torch.rand(m, generator=g, device=dev, dtype=torch.float64) * (at - copy)).long()
    k = torch.repeat_interleave(torch.arange(m, device=dev), copy)
    off = torch.arange(k.numel(), device=dev) - (copy.cumsum(0) - copy)[k]
    dst = at[k] + off
    keep = dst < n
    dst, src = dst[keep], (src[k] + off)[keep]
    idx = torch.arange(n, device=dev)
    idx[dst] = src
    for _ in range(40):  # every chain of copies ends at a fresh byte
        nxt = idx[idx]
        if torch.equal(nxt, idx):
            break
        idx = nxt
    return out[idx].contiguous()


def _fastq(n, g):
    """Records of a header, 150 order-2 Markov bases, "+" and 150 qualities."""
    dev = g.device
    rows = n // 325 + 2
    cum = torch.rand(16, 3, generator=g, device=dev).sort(1).values
    ctx = torch.randint(0, 16, (rows,), generator=g, device=dev)
    base = torch.empty(rows, 150, dtype=torch.uint8, device=dev)
    acgt = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=dev)
    for t in range(150):
        b = (torch.rand(rows, 1, generator=g, device=dev) >= cum[ctx]).sum(1)
        ctx = ((ctx << 2) | b) & 15
        base[:, t] = acgt[b]
    isn = torch.rand(rows, 150, generator=g, device=dev) < 1e-3
    mu = 38 - 10 * torch.arange(150, device=dev) / 149
    q = (mu + 3 * torch.randn(rows, 150, generator=g, device=dev) + 0.5).floor().clamp(2, 41)
    base[isn] = 78
    q[isn] = 2
    step = torch.randint(1, 21, (rows,), generator=g, device=dev).cumsum(0)
    y, x = step % 99999 + 1, 1000 + step // 99999
    tile = 1101 + torch.arange(rows, device=dev) // 1000000

    def lit(s):
        return torch.tensor(list(s), dtype=torch.uint8, device=dev).expand(rows, len(s))

    def digits(v, k):
        return torch.stack([v // 10 ** (k - 1 - j) % 10 + 48 for j in range(k)], 1).to(torch.uint8)

    row = torch.cat([lit(b"@SIM:1:FC:1:"), digits(tile, 4), lit(b":"), digits(x, 4), lit(b":"), digits(y, 5), lit(b"\n"),
                     base, lit(b"\n+\n"), (q + 33).to(torch.uint8), lit(b"\n")], 1)
    keep = torch.ones_like(row, dtype=torch.bool)
    for j in range(4):  # y without leading zeros
        keep[:, 22 + j] = y >= 10 ** (4 - j)
    return row[keep][:n].contiguous()


def _genome(n, g):
    """A random base of 10^6, then copies of it, each base with a SNP in 10^3
    and an indel of 1 to 5 in 10^4, a tandem repeat before each copy."""
    dev, period = g.device, 1000000
    acgt = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=dev)
    base = torch.randint(0, 4, (period,), generator=g, device=dev, dtype=torch.uint8)
    parts, have = [base], period
    while have < n:
        m = min(32, (n - have) // period + 1)
        unit = torch.randint(0, 4, (50,), generator=g, device=dev, dtype=torch.uint8)
        u = unit[:int(torch.randint(2, 51, (1,), generator=g, device=dev))]
        tandem = u.repeat(int(torch.randint(10, 201, (1,), generator=g, device=dev)))
        r = torch.rand(m * period, generator=g, device=dev)
        s = base.repeat(m)
        snp = r < 1e-3
        s = torch.where(snp, (s + torch.randint(1, 4, s.shape, generator=g, device=dev, dtype=torch.uint8)) & 3, s)
        count = torch.ones(m * period, dtype=torch.uint8, device=dev)
        indel = ((r >= 1e-3) & (r < 1.1e-3)).nonzero()[:, 0]
        ln = torch.randint(1, 6, indel.shape, generator=g, device=dev)
        ins = torch.rand(indel.shape, generator=g, device=dev) < 0.5
        for k in range(5):
            gone = indel[~ins & (ln > k)] + k
            count[gone[gone < count.numel()]] = 0
        count[indel[ins]] += ln[ins].to(torch.uint8)
        start = count.long().cumsum(0) - count
        k = torch.repeat_interleave(torch.arange(m * period, device=dev), count.long())
        new = torch.arange(k.numel(), device=dev) != start[k]  # inserted bases
        fill = torch.randint(0, 4, k.shape, generator=g, device=dev, dtype=torch.uint8)
        parts += [tandem, torch.where(new, fill, s[k])]
        have += tandem.numel() + k.numel()
    return acgt[torch.cat(parts)[:n].int()].contiguous()


_MAKE = {"fastq": _fastq, "genome": _genome, "text": _text, "mixed": _mixed}


def _data(profile, n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return _MAKE[profile](n, g)


def _archive(data, profile, case, log2b=0):
    arc = ace.ace_encode_gpu(data, log2b or case["log2b"], MIN_MATCH[profile], off_width=case["off_width"],
                             adaptive=case["adaptive"])
    return arc.cpu().numpy()


# -------------------------------------------------------------------- cases

def prepare(case, seed):
    op, size, profile = case["op"], case["size"], case["profile"]
    rng = np.random.default_rng(seed)
    if op == "encode":
        # where the program keeps its archives: room for one of this input's size
        store = torch.zeros(size + size // 4 + 64 * KIB, dtype=torch.uint8, device="cuda")
        return {"op": op, "data": _data(profile, size, seed), "log2b": case["log2b"], "min_match": MIN_MATCH[profile],
                "off_width": case["off_width"], "adaptive": case["adaptive"], "store": store}
    if op == "open":
        return {"op": op, "arc": _archive(_data(profile, size, seed), profile, case)}
    if op == "decode":
        da = DeviceArchive(_archive(_data(profile, size, seed), profile, case))
        return {"op": op, "da": da, "out": torch.empty(size, dtype=torch.uint8, device="cuda")}
    if op == "seek":
        blocks = (case["length"] >> case["log2b"]) + 2 + 512  # the range, and room for the blocks it reads
        da = DeviceArchive(_archive(_data(profile, size, seed), profile, case), max_seek_blocks=blocks)
        return {"op": op, "da": da, "coord": int(rng.integers(0, size - case["length"] + 1)), "length": case["length"],
                "out": torch.empty(case["length"], dtype=torch.uint8, device="cuda")}
    if op == "serve":
        das = [DeviceArchive(_archive(_data(p, size, seed * 8 + i), p, case)) for i, p in enumerate(PROFILES)]
        n, block = case["count"], 1 << case["log2b"]
        lens = rng.permutation(np.exp(np.linspace(np.log(16 * KIB), np.log(MIB), 2 * n)).astype(np.uint64))
        arcs = rng.integers(0, 4, 2 * n).astype(np.uint32)
        coords = (rng.random(2 * n) * (size - lens)).astype(np.uint64)
        # slots for one of the two batches and the blocks its matches read, not for both
        spans = (coords + lens - np.uint64(1)) // np.uint64(block) - coords // np.uint64(block) + np.uint64(1)
        slots = int(max(spans[:n].sum(), spans[n:].sum())) + 4 * 192 + 8
        pool = int(((lens + np.uint64(15)) & ~np.uint64(15)).sum())
        cache = SeekCache(das, slots, max(n, (slots + 31) // 32), pool, stream=torch.cuda.current_stream())
        cache.pool.zero_()
        a = cache.plan_arrays(arcs[:n], coords[:n], lens[:n])
        b = cache.plan_arrays(arcs[n:], coords[n:], lens[n:])
        b["out_off"] += a["out_off"][-1] + ((a["len"][-1] + np.uint64(15)) & ~np.uint64(15))
        return {"op": op, "cache": cache, "batches": (a, b)}
    assert op == "batch"
    n = case["count"]
    whole = [_data(p, max(8 * MIB, size), seed * 8 + i) for i, p in enumerate(PROFILES)]
    sizes = rng.permutation(np.exp(np.linspace(np.log(4 * KIB), np.log(size), n)).astype(np.int64))
    arcs = []
    for k in range(n):
        i = int(rng.integers(0, 4))
        at = int(rng.integers(0, whole[i].numel() - sizes[k] + 1))
        arcs.append(_archive(whole[i][at:at + int(sizes[k])].clone(), PROFILES[i], case, int(rng.choice((12, 14, 16)))))
    db = DeviceBatch(arcs)
    db.out.zero_()
    return {"op": op, "db": db}


def run(state):
    op = state["op"]
    if op == "decode":
        return state["da"].decode_all(state["out"])
    if op == "encode":
        arc, stats = ace.ace_encode_gpu(state["data"], state["log2b"], state["min_match"], stats=True,
                                        off_width=state["off_width"], adaptive=state["adaptive"])
        state["store"][:arc.numel()].copy_(arc)
        return {"archive": state["store"], "bytes": arc.numel(), "stats": stats}
    if op == "open":
        da = DeviceArchive(state["arc"])
        out = da.decode_all()
        status = da.sync()
        da.close()
        return {"out": out, "status": status}
    if op == "seek":
        out = state["da"].seek(state["coord"], state["length"], state["out"])
        return {"out": out, "status": state["da"].sync()}
    if op == "serve":
        for r in state["batches"]:
            state["cache"].run_batch(r)
        return state["cache"].pool
    state["db"].decode()
    return state["db"].out


def work(case):
    op, size = case["op"], case["size"]
    mean = sum(1 / r for r in RATIO.values()) / len(RATIO)
    part = 1 + (mean if case["profile"] == "all" else 1 / RATIO[case["profile"]])  # raw and compressed, once each
    if op == "seek":
        n = case["length"]
    elif op == "serve":  # 2 count requests, lengths log-uniform
        n = 2 * case["count"] * (MIB - 16 * KIB) / np.log(64)
    elif op == "batch":
        n = case["count"] * (size - 4 * KIB) / max(np.log(size / (4 * KIB)), 1e-9)
    else:
        n = size
    return {"bytes": float(n * part), "flops": 0.0}
