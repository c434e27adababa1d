"""decode_fastq_streams on a caller's stream: its parts decode on streams of
their own, so the output has to be complete for whatever follows on the
caller's stream, under capture, and with two sets at once. Streams that are not
the lines of a FASTQ are reported or put together within the output's bounds."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def opened(parts):
    import paper_2606_18900_gb300 as ace

    return [ace.Archive(ace.encode(p, min_match=16)) for p in parts]


@pytest.fixture(scope="module")
def sets():
    import paper_2606_18900_gb300 as ace

    out = []
    for seed in (3, 4):
        data = synth.pe_fastq(6 << 20, seed=seed, ref_len=1_000_000)
        out.append((data, opened(ace.fastq_split(data)[0])))
    return out


def test_output_is_ready_on_the_callers_stream(sets):
    import paper_2606_18900_gb300 as ace

    data, arcs = sets[0]
    want = torch.from_numpy(data).cuda()
    out = torch.zeros(data.size, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for _ in range(5):
        with torch.cuda.stream(st):
            out.zero_()
            ace.decode_fastq_streams(arcs, out, st)
            same = (out == want).all()
        st.synchronize()
        assert bool(same)
    for a in arcs:
        a.check()


def test_two_sets_at_once(sets):
    import paper_2606_18900_gb300 as ace

    streams = [torch.cuda.Stream() for _ in sets]
    outs = [torch.zeros(d.size, dtype=torch.uint8, device="cuda") for d, _ in sets]
    torch.cuda.synchronize()
    for _ in range(4):
        for (_, arcs), o, st in zip(sets, outs, streams):
            ace.decode_fastq_streams(arcs, o, st)
    for st in streams:
        st.synchronize()
    for (d, arcs), o in zip(sets, outs):
        for a in arcs:
            a.check()
        assert np.array_equal(o.cpu().numpy(), d)


def test_capture(sets):
    import paper_2606_18900_gb300 as ace

    data, arcs = sets[1]
    out = torch.zeros(data.size, dtype=torch.uint8, device="cuda")
    st = torch.cuda.Stream()
    ace.decode_fastq_streams(arcs, out, st)  # (the first call makes streams and scratch)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        ace.decode_fastq_streams(arcs, out, st)
    for _ in range(3):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        for a in arcs:
            a.check()
        assert np.array_equal(out.cpu().numpy(), data)


@pytest.mark.parametrize("which", [(0,), (1,), (3,), (0, 1, 2, 3)])
def test_streams_of_empty_lines(which):
    """More newlines than a stream's index holds: reported by parts[0], nothing
    written outside the output, and a handle that still decodes."""
    import paper_2606_18900_gb300 as ace

    rng = np.random.default_rng(5)
    lines = np.frombuffer(b"".join(b"%d\n" % x for x in rng.integers(10, 10**6, 20_000)), np.uint8)
    parts = [np.full(150_001, 10, np.uint8) if k in which else lines for k in range(4)]
    arcs = opened(parts)
    n = sum(p.size for p in parts)
    buf = torch.full((n + 64,), 7, dtype=torch.uint8, device="cuda")
    ace.decode_fastq_streams(arcs, buf[32:32 + n])
    assert arcs[0].last_error() == ace.ECORRUPT
    assert all(a.last_error() == ace.OK for a in arcs[1:])
    assert bool((buf[:32] == 7).all()) and bool((buf[32 + n:] == 7).all())
    good = opened([lines] * 4)
    if 0 not in which:
        good[0] = arcs[0]
    out = torch.zeros(4 * lines.size, dtype=torch.uint8, device="cuda")
    ace.decode_fastq_streams(good, out)
    for a in good:
        a.check()
    want = b"".join(x + b"\n" for x in lines.tobytes().split(b"\n")[:-1] for _ in range(4))
    assert out.cpu().numpy().tobytes() == want


def test_unequal_line_counts():
    """Lines of the first stream lead; what the others lack is empty, and what
    they have more goes with the last lines or is left out."""
    import paper_2606_18900_gb300 as ace

    parts = [np.frombuffer(b"".join(b"%d\n" % (k * 1000 + i) for i in range(c)), np.uint8)
             for k, c in enumerate((900, 1000, 5, 700))]
    arcs = opened(parts)
    n = sum(p.size for p in parts)
    buf = torch.full((n + 64,), 7, dtype=torch.uint8, device="cuda")
    ace.decode_fastq_streams(arcs, buf[32:32 + n])
    for a in arcs:
        a.check()
    got = buf.cpu().numpy()
    assert (got[:32] == 7).all() and (got[32 + n:] == 7).all()
    lines = [p.tobytes().split(b"\n")[:-1] for p in parts]
    want = b"".join(ls[r] + b"\n" for r in range(900) for ls in lines if r < len(ls))
    assert got[32:32 + len(want)].tobytes() == want
