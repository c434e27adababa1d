"""The library's host code over a CUDA runtime that runs on the CPU
(tests/support/host_on_fake_cuda.cpp): each entry point is called with each of
its runtime calls failing in turn and then called again, which has to work and
to launch nothing on memory that is missing, too small or not initialised."""
import os
import shutil
import subprocess

import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cuda = "/usr/local/cuda/include"
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no g++ or no CUDA headers")
    csrc = os.path.join(ROOT, "paper_2606_18900_gb300", "csrc")
    d = tmp_path_factory.mktemp("fake_cuda")
    sources = [os.path.join(ROOT, "tests", "support", "host_on_fake_cuda.cpp")]
    sources += [os.path.join(csrc, f) for f in ("host.cpp", "server.cpp", "encoder.cpp")]
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I" + csrc, "-I" + os.path.join(ROOT, "include"), "-I" + cuda,
                        *sources, "-o", str(d / "program"), "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    synth.pe_fastq(16 << 20, seed=12, ref_len=2_000_000).tofile(d / "in.fastq")

    synth.fasta(16 << 20, seed=12).tofile(d / "in.fasta")

    def run(mode, name="in.fastq"):
        r = subprocess.run([str(d / "program"), mode, str(d / name)], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
        return r.stdout

    return run


def test_calls_after_a_failure(program):
    out = program("calls")
    assert out.count("ok ") == 9


def test_server(program):
    """The engine's lock is free while it reads a batch's error word back; a
    handle's stage may be made smaller while it is served; a batch whose event
    or error word cannot be read ends with an error, and is waited for no
    longer."""
    assert "ok requests" in program("server")


def test_depth_of_short_lists(program):
    """Teams may take two segments each in FASTQ (eight levels, many commands)
    and only one in a genome (two or three levels), where two were slower than
    a warp per segment."""
    assert "depth 2" in program("depth")
    assert "depth 0" in program("depth", "in.fasta")


def test_blocks_of_a_line(program):
    """The pieces in which a line is copied, up to the longest line that a
    stream may hold: sums in 32 bits wrapped from 2^32 - 30 bytes on."""
    assert "ok blocks" in program("blocks")
