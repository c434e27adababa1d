"""Window CRCs whose pieces are larger than a segment: small segments, windows
that are not a multiple of the piece, starts inside a piece and unaligned
starts, rings of one piece, against zlib."""
import zlib

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def genome():
    return synth.fasta(70_000_003, seed=5)


@pytest.mark.parametrize("log2_B,n,window,lo", [
    (3, 2_000_003, 1_900_000, 0), (3, 2_000_003, 1_900_008, 8), (3, 2_000_003, 1_900_000, 24), (4, 3_000_001, 2_900_016, 48),
    (8, 70_000_003, 60_000_256, 0), (8, 70_000_003, 33_333_248, 256 * 7), (10, 70_000_003, 1 << 26, 0),
    (10, 70_000_003, 60_000_256, 1024 * 3), (12, 70_000_003, 40_960_000, 4096 * 5), (13, 70_000_003, 8192 * 7001, 8192),
    (14, 70_000_003, 1 << 25, 0)])
def test_pieces(genome, log2_B, n, window, lo):
    import paper_2606_18900_gb300 as ace

    data = genome[:n]
    D = 1 << 16
    window = window >> log2_B << log2_B
    ring = 1
    while ring < window + D + (2 << log2_B):
        ring *= 2
    with ace.GpuEncoder(0) as enc:
        arc = enc.encode(data, log2_B=log2_B, min_match=16, dist_bound=D)
    with ace.Archive(arc) as a:
        k = -(-(n - lo) // window)
        crc = torch.zeros(k, dtype=torch.int32, device="cuda")
        for _ in range(2):
            crc.zero_()
            a.stream_range(lo, n, ring, window, crc)
            a.check()
            got = [int(c) & 0xFFFFFFFF for c in crc.cpu().tolist()]
            assert got == [zlib.crc32(data[lo + i * window:min(n, lo + (i + 1) * window)].tobytes()) for i in range(k)]
