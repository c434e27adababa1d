"""Short work lists (staged_kernel: a team of warps builds each segment in
shared memory) against the source bytes and against the one-warp-per-segment
path (which a launch of one warp per CTA always takes): segment sizes from 4
bytes to 16 KiB, aligned and unaligned output, commands in one batch per warp
and in several, matches of one block and of hundreds, chains of matches inside
a segment, and the list lengths around the limits of the rule."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

GRID = 152


def mixed(n, seed):
    """Random bases, copies of earlier text of 4 to 3,000 bytes (some of them
    of text copied a moment before) and runs."""
    rng = np.random.default_rng(seed)
    out = np.empty(n + 4096, dtype=np.uint8)
    at = 0
    while at < n:
        kind = rng.random()
        if at < 64 or kind < 0.4:
            k = int(rng.integers(1, 60))
            out[at:at + k] = rng.integers(65, 85, k)
        elif kind < 0.95:
            k = int(min(at, np.exp(rng.uniform(np.log(4), np.log(3000)))))
            back = int(rng.integers(k, at + 1)) if rng.random() < 0.6 else int(min(at, k + rng.integers(0, 200)))
            out[at:at + k] = out[at - back:at - back + k]
        else:
            k = int(rng.integers(8, 400))
            out[at:at + k] = 65
        at += k
    return out[:n]


def decoded(arc, n, shift, one_warp):
    import paper_2606_18900_gb300 as ace

    with ace.Archive(arc) as a:
        if one_warp:
            a.set_launch(0, 1, 0)
        buf = torch.full((n + 64,), 7, dtype=torch.uint8, device="cuda")
        a.decode_all(buf[32 + shift:32 + shift + n])
        a.check()
    got = buf.cpu().numpy()
    assert (got[:32 + shift] == 7).all() and (got[32 + shift + n:] == 7).all()
    return got[32 + shift:32 + shift + n]


@pytest.mark.parametrize("shift", [0, 1, 8])
@pytest.mark.parametrize("log2_B,min_match,n", [
    (14, 4, 1), (14, 4, 127), (14, 4, 128), (14, 4, 16384), (14, 4, 16385), (14, 4, 700_001), (14, 16, 700_001),
    (10, 4, 300_001), (7, 4, 60_001), (4, 4, 9_001), (3, 2, 4_001), (2, 1, 2_001), (20, 16, 1_500_003)])
def test_short_list(log2_B, min_match, n, shift):
    import paper_2606_18900_gb300 as ace

    data = mixed(n, 10 * log2_B + min_match)
    arc = ace.encode(data, log2_B=log2_B, min_match=min_match)
    assert np.array_equal(decoded(arc, n, shift, False), data)
    assert np.array_equal(decoded(arc, n, shift, True), data)


@pytest.mark.parametrize("segments", [GRID - 1, GRID, GRID + 1, 6 * GRID, 6 * GRID + 1, 12 * GRID, 12 * GRID + 1])
def test_list_lengths(segments):
    import paper_2606_18900_gb300 as ace

    n = 256 * segments - 3
    data = mixed(n, segments)
    arc = ace.encode(data, log2_B=8, min_match=4)
    assert np.array_equal(decoded(arc, n, 0, False), data)


def test_ranges():
    """The paged view: closures of a few and of many segments."""
    import paper_2606_18900_gb300 as ace

    data = synth.tiny_fastq(5)
    arc = ace.encode(data, log2_B=12, min_match=16)
    with ace.Archive(arc) as a:
        for lo, hi in [(0, 1), (5_000, 5_001), (4_095, 4_097), (300_000, 360_001), (0, data.size), (data.size - 1, data.size)]:
            out = torch.zeros(hi - lo, dtype=torch.uint8, device="cuda")
            a.decode_range(lo, hi, out)
            a.check()
            assert np.array_equal(out.cpu().numpy(), data[lo:hi])


def test_corrupt_and_late_segments():
    """A damaged payload is reported and a segment that is never published
    runs the others into the wait limit; the handle decodes afterwards."""
    import paper_2606_18900_gb300 as ace

    data = synth.tiny_fastq(6)
    arc = ace.encode(data, min_match=16)
    bad = arc.copy()
    at = int(arc[104:112].view(np.uint64)[0])
    bad[at:at + 4] = 0  # a lane's initial state below 2^16
    with ace.Archive(bad) as a:
        out = torch.zeros(data.size, dtype=torch.uint8, device="cuda")
        a.decode_all(out)
        assert a.last_error() == ace.ECORRUPT
    off_deps = int(arc[88:96].view(np.uint64)[0])
    source = int(arc[off_deps:off_deps + 4].view(np.uint32)[0])  # a segment that another one reads
    with ace.Archive(arc) as a:
        out = torch.zeros(data.size, dtype=torch.uint8, device="cuda")
        a.debug_block_segments([source])
        a.set_wait_limit(20_000_000)
        a.decode_all(out)
        assert a.last_error() == ace.ETIMEOUT
        a.debug_block_segments([])
        a.set_wait_limit(0)
        a.decode_all(out)
        a.check()
        assert np.array_equal(out.cpu().numpy(), data)
