"""The wait limit bounds waits for other segments and nothing else: archives
whose segments depend on no other decode under the shortest limit, whatever
chains of matches a segment holds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def chains(n, seed):
    """Literals and copies of text from just before, so that most matches of a
    segment read an earlier match of it."""
    rng = np.random.default_rng(seed)
    out = np.empty(n + 512, dtype=np.uint8)
    out[:64] = rng.integers(65, 85, 64)
    at = 64
    while at < n:
        k = int(rng.integers(24, 60))
        out[at:at + k] = out[at - k:at]
        out[at + k:at + k + 6] = rng.integers(65, 85, 6)
        at += k + 6
    return out[:n]


@pytest.mark.parametrize("segments", [1, 40, 900])
def test_segments_without_sources(segments):
    import paper_2606_18900_gb300 as ace

    n = 16384 * segments - 7
    data = chains(n, segments)
    with ace.Archive(ace.encode(data, min_match=16, max_level=0)) as a:
        assert a.stats()["max_level"] == 0
        a.set_wait_limit(1)
        for _ in range(5):
            out = torch.zeros(n, dtype=torch.uint8, device="cuda")
            a.decode_all(out)
            a.check()
            assert np.array_equal(out.cpu().numpy(), data)
