"""Closures searched on the device in memory that other archives have used:
several archives are opened, decoded and closed, so that the library's pool
hands their buffers (random payload among them) to the next handles, and wide
closures (more than the 16,384 dependency entries that the host walks) on new
handles must give the source bytes and latch nothing."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def edges_of(sec, lo, hi):
    """Dependency entries that a walk of the closure of [lo, hi) visits."""
    ptr, deps, shift = sec["dep_ptr"], sec["deps"], sec["log2_S"]
    seen = set(range(lo >> shift, ((hi - 1) >> shift) + 1))
    stack, edges = list(seen), 0
    while stack:
        s = stack.pop()
        new = [int(d) for d in deps[int(ptr[s]):int(ptr[s + 1])]]
        edges += len(new)
        for d in new:
            if d not in seen:
                seen.add(d)
                stack.append(d)
    return edges


@pytest.mark.parametrize("log2_B,mib", [(10, 12), (12, 16), (14, 48)])
def test_wide_closures_in_used_memory(log2_B, mib):
    import paper_2606_18900_gb300 as ace

    rng = np.random.default_rng(log2_B)
    data = synth.pe_fastq(mib << 20, seed=log2_B, ref_len=2_000_000)
    with ace.GpuEncoder(0) as enc:
        arc = enc.encode(data, log2_B=log2_B, min_match=16, reads=ace.fastq_index(data))
        noise = [enc.encode(rng.integers(0, 256, k << 20, dtype=np.uint8)) for k in (1, 3, 9, 27)]
    for a in [ace.Archive(x) for x in noise]:
        out = torch.empty(a.size, dtype=torch.uint8, device="cuda")
        a.decode_all(out)
        a.check()
        a.close()
    sec, wide = oracle.sections(arc), 0
    for k in range(3):
        with ace.Archive(arc) as a:
            n_reads = a.stats()["n_reads"]
            ranges = [a.read_lookup(int(r)) for r in synth.uniform(9, k, 6, n_reads)]
            ranges += [(data.size - (300_001 << k), data.size), (data.size // 2, data.size // 2 + 1)]
            for lo, hi in ranges:
                wide += edges_of(sec, lo, hi) > 16384
                buf = torch.zeros(hi - lo, dtype=torch.uint8, device="cuda")
                a.decode_range(lo, hi, buf)
                a.check()
                assert np.array_equal(buf.cpu().numpy(), data[lo:hi]), (lo, hi)
    assert wide >= 3
