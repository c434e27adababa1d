"""FASTQ reassembly from line streams: line lengths from empty to longer than
an index chunk, files cut inside a record, outputs at any alignment, newline
counts on both sides of a row and a chunk of the index, and one handle given
for two parts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def fastq(records, lengths, seed, cut=0):
    rng = np.random.default_rng(seed)
    lines = []
    for r in range(records):
        n = int(lengths[r % len(lengths)])
        seq = rng.choice(np.frombuffer(b"ACGT", np.uint8), n).tobytes()
        qual = rng.integers(35, 74, n).astype(np.uint8).tobytes()
        lines.append(b"@r%d\n%s\n+\n%s\n" % (r, seq, qual))
    data = np.frombuffer(b"".join(lines), np.uint8)
    return data[:data.size - cut] if cut else data


@pytest.mark.parametrize("shift", [0, 5])
@pytest.mark.parametrize("records,lengths,cut", [
    (1, [1], 0), (3, [10], 0), (2000, [150], 0), (2000, [150], 40), (2000, [150], 200), (500, [0, 1, 2, 15, 16, 17, 33], 0),
    (9, [70_000, 3], 0), (8, [131_072], 1), (40_000, [1], 0), (7, [150], 3)])
def test_lines(records, lengths, cut, shift):
    import paper_2606_18900_gb300 as ace

    data = fastq(records, lengths, records + cut, cut)
    parts, _ = ace.fastq_split(data)
    arcs = [ace.Archive(ace.encode(p, min_match=16)) for p in parts]
    buf = torch.full((data.size + 64,), 7, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        buf.fill_(7)
        ace.decode_fastq_streams(arcs, buf[32 + shift:32 + shift + data.size])
        for a in arcs:
            a.check()
        got = buf.cpu().numpy()
        assert np.array_equal(got[32 + shift:32 + shift + data.size], data)
        assert (got[:32 + shift] == 7).all() and (got[32 + shift + data.size:] == 7).all()


def test_one_handle_for_two_parts():
    import paper_2606_18900_gb300 as ace

    line = np.frombuffer(b"ACGTACGTTTGACA\n" * 5000, np.uint8)
    parts = [np.frombuffer(b"".join(b"@%d\n" % i for i in range(5000)), np.uint8), line,
             np.frombuffer(b"+\n" * 5000, np.uint8)]
    a = [ace.Archive(ace.encode(p, min_match=16)) for p in parts]
    want = b"".join(b"@%d\nACGTACGTTTGACA\n+\nACGTACGTTTGACA\n" % i for i in range(5000))
    out = torch.zeros(len(want), dtype=torch.uint8, device="cuda")
    ace.decode_fastq_streams([a[0], a[1], a[2], a[1]], out)
    for x in a:
        x.check()
    assert out.cpu().numpy().tobytes() == want
