"""Lists around the limits of the rule that gives short lists to teams (one or
two segments per team by the archive's depth, none for small segments), at this
GPU's number of CTAs, against the source bytes and the one-warp-per-segment
path."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def words(n, seed):
    """Text of short words, so that segments have many commands."""
    rng = np.random.default_rng(seed)
    pool = [rng.integers(65, 85, int(k), dtype=np.uint8) for k in rng.integers(6, 30, 400)]
    return np.concatenate([pool[i] for i in rng.integers(0, 400, n // 6)])[:n]


@pytest.mark.parametrize("cap", [0, 1, 8])
@pytest.mark.parametrize("per_cta,more,log2_B", [
    (1, 0, 12), (1, 1, 12), (6, -1, 12), (6, 0, 12), (6, 1, 12), (7, 0, 12), (7, 1, 12), (12, 0, 12), (12, 1, 12),
    (1, -144, 10), (6, 1, 10), (1, -144, 11), (6, 0, 11), (6, 1, 11), (12, 1, 11)])
def test_limits(per_cta, more, log2_B, cap):
    import paper_2606_18900_gb300 as ace

    with ace.Archive(ace.encode(np.zeros(64, np.uint8))) as a:
        a.set_launch(0, 0, 0)  # (looks the number of CTAs up)
        segments = per_cta * a.get_launch()["max_ctas"] + more
    n = (segments << log2_B) - 5
    data = words(n, segments)
    with ace.Archive(ace.encode(data, log2_B=log2_B, min_match=8, max_level=cap)) as a:
        for warps in (0, 1):  # the default, and one warp per CTA, which is never a team
            a.set_launch(0, warps, 0)
            buf = torch.full((n + 64,), 7, dtype=torch.uint8, device="cuda")
            a.decode_all(buf[16:16 + n])
            a.check()
            got = buf.cpu().numpy()
            assert np.array_equal(got[16:16 + n], data)
            assert (got[:16] == 7).all() and (got[16 + n:] == 7).all()
