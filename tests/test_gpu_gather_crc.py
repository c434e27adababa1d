"""Range gathers at every alignment of source and destination, across segment
ends, and window CRCs of pieces of all lengths."""
import zlib

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("log2_B", [2, 4, 5, 10, 14])
def test_gather(log2_B):
    import paper_2606_18900_gb300 as ace

    n = 40_003 if log2_B > 2 else 3_001
    data = synth.random_bytes(9, log2_B, n, b"ACGTN\n")
    with ace.Archive(ace.encode(data, log2_B=log2_B, min_match=4)) as a:
        for lo in (0, 1, 15, 16, 17, 1000, n - 40, n - 1):
            for length in (1, 2, 15, 16, 17, 31, 33, 64, 1500):
                hi = min(n, lo + length)
                shift = (lo + length) % 19
                buf = torch.full((hi - lo + 64,), 7, dtype=torch.uint8, device="cuda")
                a.decode_range(lo, hi, buf[16 + shift:16 + shift + hi - lo])
                got = buf.cpu().numpy()
                assert np.array_equal(got[16 + shift:16 + shift + hi - lo], data[lo:hi])
                assert (got[:16 + shift] == 7).all() and (got[16 + shift + hi - lo:] == 7).all()
        a.check()


@pytest.mark.parametrize("log2_B,windows,n", [(2, 8, 999), (4, 3, 5_001), (9, 5, 40_001), (10, 1, 70_000), (14, 3, 500_001),
                                              (14, 1, 16_384), (14, 1, 16_385), (14, 64, 3_000_007)])
def test_window_crc(log2_B, windows, n):
    import paper_2606_18900_gb300 as ace

    data = synth.random_bytes(11, n, n, b"ACGTN\n")
    S = 1 << min(log2_B, 14)
    window = -(-n // windows // S) * S
    D = max(S, 64)
    ring = 1
    while ring < window + D + 16 + 2 * S:
        ring *= 2
    with ace.Archive(ace.encode(data, log2_B=log2_B, min_match=4, dist_bound=D)) as a:
        k = -(-n // window)
        crc = torch.zeros(k, dtype=torch.int32, device="cuda")
        for _ in range(2):
            a.stream_range(0, n, ring, window, crc)
            a.check()
            got = [int(c) & 0xFFFFFFFF for c in crc.cpu().tolist()]
            assert got == [zlib.crc32(data[i * window:(i + 1) * window].tobytes()) for i in range(k)]
