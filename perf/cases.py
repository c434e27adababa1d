"""Workloads of the library as its users run them, for timing.

Every case goes through the public binding (paper_2606_18900_gb300): archives
are encoded and opened in prepare(), which hands over what a program holds
before the call (the open handle, device or pinned host buffers), and run()
makes the call. Inputs come from the seeded generators in synth/, whose
sequence, quality, header and repeat statistics stand in for real FASTQ and
FASTA files.

All outputs are bytes, CRCs and status words: whole numbers, which must be
equal and have no value in floating point to be compared with, so exact()
gives none.
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2606_18900_gb300 as ace
import synth

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30
FASTQ_RATIO = 2.3   # compression of the generated FASTQ (16 KiB blocks, min_match 16)
FASTA_RATIO = 3.4   # and of a 200 MB generated genome (min_match 32)
LINE = 60           # bases per FASTA line of the generated genome


def listed():
    return [
        # one small sample, resident in L2: 2,000 single-end reads; latency of a whole-file decode
        {"name": "fastq tiny", "kind": "decode", "n": 675_000, "log2_B": 14, "cap": 8, "paired": False},
        # the headline: a 1 GiB paired-end FASTQ decoded in device memory
        {"name": "fastq 1 GiB", "kind": "decode", "n": GIB, "log2_B": 14, "cap": 8, "paired": True},
        # random access: record lookups by read ID, one after the other, as a pipeline that fetches reads does
        {"name": "read lookups", "kind": "reads", "n": 256 * MIB, "log2_B": 14, "cap": 8, "count": 32},
        # random access by coordinate: bases of chr:pos regions of a genome
        {"name": "region lookups", "kind": "regions", "n": 200_000_000, "log2_B": 14, "length": 150, "count": 32},
        # one ragged slice of a FASTQ in 1 MiB blocks, as a worker that takes its share of a file
        {"name": "range 9 MB", "kind": "range", "n": 128 * MIB, "log2_B": 20, "cap": 8, "length": 9_437_101},
        # a genome streamed through a device ring smaller than itself, checked by a CRC per window
        {"name": "genome ring", "kind": "stream", "n": 500_000_000, "log2_B": 14, "window": 128 * MIB},
        # many small files of uneven size in one launch
        {"name": "batch 512", "kind": "batch", "count": 512, "hi": 2 * MIB},
        # a FASTQ on the host to its bytes on the host in one call
        {"name": "host to host", "kind": "host", "n": 256 * MIB, "log2_B": 14, "cap": 8},
        # a decode by a program that forbids allocation: the archive is already in device memory
        {"name": "no allocation", "kind": "noalloc", "n": 64 * MIB, "log2_B": 14, "cap": 8},
        # a FASTQ stored as its four line streams, put back together on the device
        {"name": "line streams", "kind": "streams", "n": 192 * MIB},
        # making an archive: device input, the encoder's scratch kept between calls
        {"name": "encode fastq", "kind": "encode", "data": "fastq", "n": 192 * MIB, "log2_B": 14, "cap": 8},
        # a burst of read lookups and ranges through the serving engine
        {"name": "serve burst", "kind": "serve", "n": 200_000_000, "count": 1000},
    ]


def draw(rng):
    def size(lo, hi):  # log-uniform, mostly odd
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | rng.randint(0, 1)

    def block():
        return rng.choice([10, 12, 13, 14, 14, 14, 16, 20])

    kind = rng.choice(["decode", "decode", "reads", "regions", "range", "stream", "batch", "host", "noalloc",
                       "streams", "encode", "serve"])
    if kind == "decode":
        return {"kind": kind, "n": size(64 * KIB, 384 * MIB), "log2_B": block(), "cap": rng.choice([2, 8, 8]),
                "paired": rng.random() < 0.5}
    if kind == "reads":
        return {"kind": kind, "n": size(MIB, 256 * MIB), "log2_B": block(), "cap": rng.choice([2, 8, 8]),
                "count": rng.randint(8, 48)}
    if kind == "regions":
        return {"kind": kind, "n": size(4 * MIB, 256 * MIB), "log2_B": block(), "length": size(50, 20_000),
                "count": rng.randint(8, 48)}
    if kind == "range":
        n = size(4 * MIB, 192 * MIB)
        return {"kind": kind, "n": n, "log2_B": block(), "cap": 8, "length": size(KIB, n // 3)}
    if kind == "stream":
        return {"kind": kind, "n": size(16 * MIB, 500_000_000), "log2_B": block(), "window": rng.choice([8, 32, 128]) * MIB}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(4, 400), "hi": size(64 * KIB, 4 * MIB)}
    if kind == "host":
        return {"kind": kind, "n": size(MIB, 384 * MIB), "log2_B": rng.choice([14, 14, 20]), "cap": rng.choice([2, 8])}
    if kind == "noalloc":
        return {"kind": kind, "n": size(64 * KIB, 128 * MIB), "log2_B": rng.choice([12, 14, 14, 20]), "cap": 8}
    if kind == "streams":
        return {"kind": kind, "n": size(MIB, 256 * MIB)}
    if kind == "encode":
        return {"kind": kind, "data": rng.choice(["fastq", "fastq", "fasta"]), "n": size(64 * KIB, 192 * MIB),
                "log2_B": rng.choice([12, 14, 14, 20]), "cap": rng.choice([2, 8])}
    return {"kind": kind, "n": size(8 * MIB, 256 * MIB), "count": rng.randint(100, 1500)}


# ------------------------------------------------------------------- inputs

def _fastq(n, seed, paired=True):
    """About n bytes of FASTQ records (whole records, so the size is ragged);
    large files are written as several lanes of one library in parallel."""
    ref = synth.reference(seed, 0, min(50_000_000, max(200_000, n // 20)), repeat_frac=0.05, n_families=50)
    lanes = max(1, min(16, n // (8 * MIB)))
    share = -(-n // lanes)
    out = np.empty(share * lanes, dtype=np.uint8)

    def lane(i):
        d, _ = synth.fastq(ref, seed, 1 + i, paired=paired, max_bytes=share)
        return d

    with ThreadPoolExecutor(lanes) as ex:
        parts = list(ex.map(lane, range(lanes)))
    at = 0
    for p in parts:
        out[at:at + p.size] = p
        at += p.size
    return out[:at]


def _encode(data, **kw):
    with ace.GpuEncoder(0) as enc:
        return enc.encode(data, **kw)


def _positions(seed, count, bound):
    return [int(x) for x in synth.uniform(seed, 7, count, max(1, bound))]


def _u8(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def _pinned(n):
    return torch.empty(n, dtype=torch.uint8, pin_memory=True)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "decode":
        data = _fastq(case["n"], seed, case["paired"])
        s["arc"] = ace.Archive(_encode(data, log2_B=case["log2_B"], min_match=16, max_level=case["cap"]))
        s["out"] = _u8(data.size)
    elif kind == "reads":
        data = _fastq(case["n"], seed)
        arc = ace.Archive(_encode(data, log2_B=case["log2_B"], min_match=16, max_level=case["cap"],
                                  reads=ace.fastq_index(data)))
        s["ids"] = _positions(seed, case["count"], arc.stats()["n_reads"])
        s["arc"], s["out"] = arc, _u8(case["count"] * 1024).view(case["count"], 1024)
    elif kind == "regions":
        data = synth.fasta(case["n"], seed=seed)
        index, width = ace.fasta_index(data)
        s["arc"] = ace.Archive(_encode(data, log2_B=case["log2_B"], min_match=32, reads=index))
        chrom = _positions(seed, case["count"], 24)
        where = []
        for c, u in zip(chrom, _positions(seed + 1, case["count"], 1 << 30)):
            end = int(index[2 * c + 2]) if c < 23 else data.size
            room = (end - int(index[2 * c + 1])) * width // (width + 1) - case["length"] - width
            where.append((c, u % max(1, room)))
        s["where"], s["length"] = where, case["length"]
        s["out"] = _u8(case["count"] * case["length"]).view(case["count"], case["length"])
    elif kind == "range":
        data = _fastq(case["n"], seed)
        s["arc"] = ace.Archive(_encode(data, log2_B=case["log2_B"], min_match=16, max_level=case["cap"]))
        lo = _positions(seed, 1, data.size - case["length"])[0]
        s["lo"], s["hi"] = lo, lo + case["length"]
        s["out"] = _u8(case["length"])
    elif kind == "stream":
        data = synth.fasta(case["n"], seed=seed)
        D = case["window"]
        arc = ace.Archive(_encode(data, log2_B=case["log2_B"], min_match=32, dist_bound=D))
        s["ring"] = 4 * D  # the smallest power of two that holds a window, D and two segments
        s["arc"], s["window"], s["n"] = arc, case["window"], data.size
        s["crc"] = torch.zeros(-(-data.size // case["window"]), dtype=torch.int32, device="cuda")
    elif kind == "batch":
        sizes = synth.batch_sizes(case["count"], hi=case["hi"])  # one mix of sizes, other contents by the seed
        datas = synth.batch_fastq(sizes, seed=seed, ref_len=5_000_000)
        with ace.GpuEncoder(0) as enc:
            s["arcs"] = [ace.Archive(enc.encode(d, min_match=16)) for d in datas]
        ends = np.cumsum([d.size for d in datas])
        s["out"] = _u8(int(ends[-1]))
        s["outs"] = [s["out"][int(e) - d.size:int(e)] for e, d in zip(ends, datas)]
    elif kind == "host":
        data = _fastq(case["n"], seed)
        arc = _encode(data, log2_B=case["log2_B"], min_match=16, max_level=case["cap"])
        s["arc"], s["out"] = _pinned(arc.size), _pinned(data.size)
        s["arc"].copy_(torch.from_numpy(arc))
    elif kind == "noalloc":
        data = _fastq(case["n"], seed)
        s["arc"] = torch.from_numpy(_encode(data, log2_B=case["log2_B"], min_match=16, max_level=case["cap"])).cuda()
        s["out"], s["status"] = _u8(data.size), torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind == "streams":
        data = _fastq(case["n"], seed)
        parts, _ = ace.fastq_split(data)
        with ace.GpuEncoder(0) as enc:
            s["arcs"] = [ace.Archive(enc.encode(p, min_match=16)) for p in parts]
        s["out"] = _u8(data.size)
    elif kind == "encode":
        if case["data"] == "fasta":
            data, s["kw"] = synth.fasta(case["n"], seed=seed), {"min_match": 32}
        else:
            data = _fastq(case["n"], seed)
            s["kw"] = {"min_match": 16, "reads": ace.fastq_index(data)}
        s["kw"].update(log2_B=case["log2_B"], max_level=case["cap"])
        s["enc"], s["data"] = ace.GpuEncoder(0), torch.from_numpy(data).cuda()
        # the archive's length depends on the data: it is handed out as a head
        # of fixed length and the rest in a zero-padded array of fixed length
        big = 0.12 if case["data"] == "fasta" else 0.39
        s["head"] = int(data.size * (big if data.size > 16 * MIB and case["log2_B"] >= 14 else 0.1))
        s["rest"] = np.zeros(data.size + 64 * KIB, dtype=np.uint8)
    else:
        fq, fa = synth.tiny_fastq(seed), synth.fasta(case["n"], seed=seed)
        arcs = [ace.Archive(_encode(fq, min_match=16, reads=ace.fastq_index(fq))),
                ace.Archive(_encode(fa, min_match=32))]
        mix, rng = np.random.default_rng(5), np.random.default_rng(seed)  # one mix of lengths, other places by the seed
        reqs, room = [], []
        for _ in range(case["count"]):
            if mix.random() < 0.9:
                reqs.append((0, *arcs[0].read_lookup(int(rng.integers(0, 2000)))))
                room.append(512)
            else:
                length = int(np.exp(mix.uniform(np.log(1024), np.log(min(4 * MIB, fa.size // 4)))))
                lo = int(rng.integers(0, fa.size - length))
                reqs.append((1, lo, lo + length))
                room.append(length)
        starts = np.cumsum([0] + room)
        s["out"] = _u8(int(starts[-1]))
        s["outs"] = [s["out"][int(b):int(b) + hi - lo] for b, (_, lo, hi) in zip(starts, reqs)]
        s["reqs"], s["gaps"] = reqs, [0] * len(reqs)
        s["server"] = ace.Server(arcs, mem_budget=2 * GIB, slots=4)
    return s


def run(s):
    kind = s["kind"]
    if kind == "decode":
        s["arc"].decode_all(s["out"])
        return s["out"]
    if kind == "reads":
        for row, i in zip(s["out"], s["ids"]):
            s["arc"].decode_range(*s["arc"].read_lookup(i), row)
        return s["out"]
    if kind == "regions":
        for row, (chrom, pos) in zip(s["out"], s["where"]):
            s["arc"].decode_region(chrom, pos, s["length"], row, LINE)
        return s["out"]
    if kind == "range":
        s["arc"].decode_range(s["lo"], s["hi"], s["out"])
        return s["out"]
    if kind == "stream":
        s["arc"].stream_range(0, s["n"], s["ring"], s["window"], s["crc"])
        return s["crc"]
    if kind == "batch":
        ace.decode_batch(s["arcs"], s["outs"])
        return s["out"]
    if kind == "host":
        ace.decode_host(s["arc"], s["out"])
        return s["out"]
    if kind == "noalloc":
        code = ace.decode_all_noalloc(s["arc"], s["arc"].numel(), s["out"], s["status"])
        return [code, s["status"], s["out"]]
    if kind == "streams":
        ace.decode_fastq_streams(s["arcs"], s["out"])
        return s["out"]
    if kind == "encode":
        arc = s["enc"].encode(s["data"], **s["kw"])
        s["rest"][:arc.size - s["head"]] = arc[s["head"]:]
        return [arc.size, arc[:s["head"]], s["rest"]]
    tickets, status, _ = s["server"].replay(s["reqs"], s["outs"], s["gaps"])
    for t in tickets:
        s["server"].wait(t)
    return [np.array(status, dtype=np.int32), s["out"]]


def exact(case, seed):
    """None: bytes, CRCs and status words are compared for equality."""
    return None


def work(case):
    """Archive bytes read and output bytes written, once each. For a lookup
    these are its own blocks' and its record's (a source closure adds to
    them, by the data); nothing is computed in floating point."""
    kind = case["kind"]
    if kind == "batch":
        # mean of the log-uniform sizes in [16 KiB, hi)
        mean = (case["hi"] - 16 * KIB) / math.log(case["hi"] / (16 * KIB)) if case["hi"] > 16 * KIB else 16 * KIB
        out = case["count"] * mean
        return {"bytes": out + out / FASTQ_RATIO, "flops": 0}
    if kind in ("reads", "regions"):
        length = case.get("length", 350)
        block = min(16 * KIB, 1 << case["log2_B"])
        ratio = FASTQ_RATIO if kind == "reads" else FASTA_RATIO
        return {"bytes": case["count"] * (length + (length // block + 1) * block / ratio), "flops": 0}
    if kind == "range":
        return {"bytes": case["length"] * (1 + 1 / FASTQ_RATIO), "flops": 0}
    if kind == "stream":
        return {"bytes": case["n"] / FASTA_RATIO + 2 * case["n"], "flops": 0}  # written to the ring, read by the CRC
    if kind == "streams":
        # each line is decoded to its stream, read there and written to its place
        return {"bytes": case["n"] * (3 + 1 / FASTQ_RATIO), "flops": 0}
    if kind == "serve":
        top = min(4 * MIB, case["n"] // 4)
        out = case["count"] * (0.9 * 350 + 0.1 * (top - 1024) / math.log(top / 1024))
        return {"bytes": out * (1 + 1 / FASTA_RATIO), "flops": 0}
    ratio = FASTA_RATIO if case.get("data") == "fasta" else FASTQ_RATIO
    return {"bytes": case["n"] * (1 + 1 / ratio), "flops": 0}
