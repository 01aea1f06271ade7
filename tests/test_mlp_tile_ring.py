"""The weight-tile ring of the tensor-core evaluators: after an error in any
warp, the copies that tiles_landed waits for are the ones that may be in
flight (host code over ring_first)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_28514_gb300", "csrc")


@pytest.fixture(scope="module")
def ring_first(tmp_path_factory):
    nvcc = os.environ.get("NVCC", "nvcc")
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("ring")
    (d / "ring.cu").write_text('#include "ns_mlp.cuh"\nextern "C" unsigned first(unsigned a, unsigned b, unsigned s) '
                               '{ return nsd::ring_first(a, b, s); }\n')
    so = str(d / "ring.so")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                        "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, str(d / "ring.cu"), "-o", so],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = ctypes.CDLL(so).first
    f.restype = ctypes.c_uint
    return f


@pytest.mark.parametrize("stages", [3, 4, 5])
def test_every_copy_in_flight_is_waited_for(ring_first, stages):
    for item0 in (0, 1, 7, 228):
        for issued in range(0, 4 * stages + 2):
            # the consumer stopped at any tile the producer can have got to
            for consumed in range(max(0, issued - stages), issued + 1):
                in_flight = set(range(item0 + consumed, item0 + issued))
                first = ring_first(item0, item0 + issued, stages)
                waited = set(range(first, item0 + issued))
                assert in_flight <= waited and len(waited) <= stages, (item0, issued, consumed)
