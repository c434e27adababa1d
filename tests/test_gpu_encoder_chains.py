"""The GPU encoder's match search over hash chains of every length around a
warp's 32 sorted slots (pairs spread over the lanes, counted warps of long
chains, uncounted ones): the CPU encoder's archive, byte for byte."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("dist_bound", [0, 5000])
@pytest.mark.parametrize("copies", [1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 64, 65, 200])
def test_chain_lengths(copies, dist_bound):
    import paper_2606_18900_gb300 as ace

    rng = np.random.default_rng(copies)
    blocks = [rng.integers(0, 256, 40, dtype=np.uint8) for _ in range(max(3, 600 // copies))]
    order = rng.permutation(np.repeat(np.arange(len(blocks)), copies))
    data = np.concatenate([np.concatenate([blocks[i], rng.integers(0, 256, 3, dtype=np.uint8)]) for i in order])
    with ace.GpuEncoder(0) as enc:
        for mm in (8, 16):
            kw = dict(log2_B=12, min_match=mm, dist_bound=dist_bound)
            assert np.array_equal(enc.encode(data, **kw), ace.encode(data, **kw))
