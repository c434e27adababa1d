"""Gathers of long ranges at every alignment, requests packed back to back in
one buffer through the serving engine, and ranges on both sides of the length
up to which a work list goes to the device by value."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("log2_B", [2, 10, 14])
@pytest.mark.parametrize("length", [16_383, 16_384, 16_385, 70_001, 200_003])
def test_long_ranges(log2_B, length):
    import paper_2606_18900_gb300 as ace

    if log2_B == 2:
        length //= 4
    n = length + 5_000
    data = synth.random_bytes(3, log2_B, n, b"ACGTN\n")
    with ace.Archive(ace.encode(data, log2_B=log2_B, min_match=4)) as a:
        buf = torch.empty(length + 64, dtype=torch.uint8, device="cuda")
        for shift in range(19):
            lo = 37 * shift + shift // 2
            buf.fill_(7)
            a.decode_range(lo, lo + length, buf[16 + shift:16 + shift + length])
            got = buf.cpu().numpy()
            assert np.array_equal(got[16 + shift:16 + shift + length], data[lo:lo + length])
            assert (got[:16 + shift] == 7).all() and (got[16 + shift + length:] == 7).all()
        a.check()


def test_packed_requests():
    import paper_2606_18900_gb300 as ace

    rng = np.random.default_rng(8)
    data = synth.pe_fastq(3 << 20, seed=8, ref_len=500_000)
    lengths = [1, 2, 15, 16, 17, 65_535, 65_536, 65_537, 131_071, 131_073, 300_001] + [int(x) for x in rng.integers(1, 90_000, 60)]
    order = rng.permutation(len(lengths))
    with ace.Archive(ace.encode(data, min_match=16)) as a, ace.Server([a], mem_budget=256 << 20, slots=3) as srv:
        for lead in (0, 1, 7):
            buf = torch.full((64 + sum(lengths),), 7, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            at, want, tickets = 16 + lead, [], []
            for i in order:
                lo = int(rng.integers(0, data.size - lengths[i]))
                tickets.append(srv.submit(0, lo, lo + lengths[i], buf[at:at + lengths[i]]))
                want.append(data[lo:lo + lengths[i]])
                at += lengths[i]
            for t in tickets:
                srv.wait(t)
            got = buf.cpu().numpy()
            assert np.array_equal(got[16 + lead:at], np.concatenate(want))
            assert (got[:16 + lead] == 7).all() and (got[at:] == 7).all()


@pytest.mark.parametrize("log2_B", [2, 4, 6])
def test_lists_by_value_and_copied(log2_B):
    import paper_2606_18900_gb300 as ace

    n = 1100 << log2_B
    data = np.random.default_rng(log2_B).integers(0, 256, n, dtype=np.uint8)  # (no matches: a range is its own closure)
    with ace.Archive(ace.encode(data, log2_B=log2_B, min_match=8)) as a:
        for segments in (992, 993, 1, 991, 1050, 2):
            for first in (0, 17):
                lo, hi = first << log2_B, (first + segments) << log2_B
                assert a.range_closure(lo, hi)[0] == segments
                out = torch.zeros(hi - lo, dtype=torch.uint8, device="cuda")
                a.decode_range(lo, hi, out)
                a.check()
                assert np.array_equal(out.cpu().numpy(), data[lo:hi])


def test_page_table_cleared_with_the_gather_or_apart():
    """Short ranges of 4,095 to 4,097 segments, each followed by others."""
    import paper_2606_18900_gb300 as ace

    data = np.random.default_rng(2).integers(0, 256, 20_000, dtype=np.uint8)
    with ace.Archive(ace.encode(data, log2_B=2, min_match=8)) as a:
        for lo, hi, segments in ((0, 16_380, 4095), (0, 16_384, 4096), (1, 16_385, 4097), (3, 5, 2), (3_000, 19_384, 4096),
                                 (3_001, 19_385, 4097), (0, 20_000, 5000)):
            assert a.range_closure(lo, hi)[0] == segments
            out = torch.zeros(hi - lo, dtype=torch.uint8, device="cuda")
            a.decode_range(lo, hi, out)
            a.check()
            assert np.array_equal(out.cpu().numpy(), data[lo:hi])
