"""aceapex_decode_all_noalloc over the launches it chooses between: lists that
teams of warps take and longer ones, command streams that fit a warp's usual
shared stage and ones that need the largest, and a table that is one symbol."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def phrases(n, seed, lo, hi):
    """Text of phrases of lo to hi bytes from a small dictionary."""
    rng = np.random.default_rng(seed)
    book = [rng.integers(65, 91, int(rng.integers(lo, hi + 1))).astype(np.uint8) for _ in range(400)]
    out = np.concatenate([book[i] for i in rng.integers(0, 400, n // lo + 1)])
    return out[:n]


def stage_bytes(arc):
    n_seg = int(arc[40:48].view(np.uint64)[0])
    cmds = arc[2176:2176 + 24 * n_seg].view(np.uint32).reshape(-1, 6)[:, 3]
    return n_seg, int(cmds.max()) * (4 + int(arc[26])) + 4


@pytest.mark.parametrize("log2_B,lo,hi,n,big", [
    (14, 40, 200, 600_001, False),     # teams
    (14, 5, 9, 600_001, True),         # short list, large command stages
    (8, 12, 60, 256 * 1825 - 7, False),  # one segment more than the teams take
    (12, 12, 60, 9_000_001, False),
    (14, 5, 9, 33_000_001, True),      # long list, large command stages
])
def test_lists(log2_B, lo, hi, n, big):
    import paper_2606_18900_gb300 as ace

    data = phrases(n, log2_B + lo, lo, hi)
    with ace.GpuEncoder(0) as enc:
        arc = enc.encode(data, log2_B=log2_B, min_match=4)
    assert (stage_bytes(arc)[1] > 3072) == big
    d_arc = torch.from_numpy(arc).cuda()
    out = torch.zeros(n, dtype=torch.uint8, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        out.fill_(0)
        assert ace.decode_all_noalloc(d_arc, arc.size, out, status) == ace.OK
        torch.cuda.synchronize()
        assert int(status.item()) == ace.OK
        assert np.array_equal(out.cpu().numpy(), data)


@pytest.mark.parametrize("n", [1, 31, 5_000, 100_000])
def test_one_symbol(n):
    import paper_2606_18900_gb300 as ace

    data = np.full(n, 65, dtype=np.uint8)
    arc = ace.encode(data, min_match=255)
    out = torch.zeros(n, dtype=torch.uint8, device="cuda")
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    assert ace.decode_all_noalloc(torch.from_numpy(arc).cuda(), arc.size, out, status) == ace.OK
    torch.cuda.synchronize()
    assert int(status.item()) == ace.OK
    assert np.array_equal(out.cpu().numpy(), data)
