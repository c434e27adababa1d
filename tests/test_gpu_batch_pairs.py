"""A batch of more archives than CTAs: large archives, small ones that share a
CTA two by two, empty ones, several segment sizes, and command streams that do
not fit the shared stage."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("count,sizes,log2_B,min_match", [
    (153, (1, 40_000), (14,), 16), (400, (0, 200_000), (14, 10, 4), 4), (310, (140_000, 160_000), (14,), 4),
    (200, (100, 147_456), (14,), 4)])
def test_more_archives_than_ctas(count, sizes, log2_B, min_match):
    import paper_2606_18900_gb300 as ace

    rng = np.random.default_rng(count)
    text = synth.tiny_fastq(8)
    datas, arcs = [], []
    with ace.GpuEncoder(0) as enc:
        for i in range(count):
            b = log2_B[i % len(log2_B)]
            n = int(rng.integers(*sizes)) >> max(0, 2 * (10 - b) // 3)
            at = int(rng.integers(0, text.size - n))
            datas.append(text[at:at + n].copy())
            arcs.append(ace.Archive(enc.encode(datas[-1], log2_B=b, min_match=min_match)))
    ends = np.cumsum([0] + [d.size for d in datas])
    out = torch.zeros(int(ends[-1]) + 1, dtype=torch.uint8, device="cuda")
    outs = [out[int(ends[i]):int(ends[i + 1])] if datas[i].size else out[:1] for i in range(count)]
    for _ in range(2):
        out.zero_()
        ace.decode_batch(arcs, outs)
        arcs[0].check()
        assert np.array_equal(out.cpu().numpy()[:-1], np.concatenate(datas))
