"""The one-pass attention's operand ring, its order compiled on the host: what is requested before the
previous kernel has finished holds prefix keys alone, whatever the head dim and the prefix length."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37772_gb300", "csrc")
SLOTS = 5
SRC = """
#include "attn_ring.cuh"
using namespace uad;
extern "C" int early(int kp, int nck, int slots, int prefix) { return AttnRing{kp, nck}.early(slots, prefix); }
extern "C" int total(int kp, int nck) { return AttnRing{kp, nck}.total(); }
extern "C" int k_entry(int kp, int nck, int c, int j) { return AttnRing{kp, nck}.k_entry(c, j); }
extern "C" int v_entry(int kp, int nck, int c, int h) { return AttnRing{kp, nck}.v_entry(c, h); }
extern "C" void at(int kp, int nck, int e, int* out) {
  const AttnRing::Entry x = AttnRing{kp, nck}.at(e);
  out[0] = x.k; out[1] = x.chunk; out[2] = x.part; out[3] = AttnRing::end_key(x);
}
"""


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("ring")
    (d / "ring.cc").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-x", "c++", "-I", CSRC, "-o", str(d / "ring.so"), str(d / "ring.cc")],
                   check=True)
    return ctypes.CDLL(str(d / "ring.so"))


@pytest.mark.parametrize("kp", [1, 2])   # head dim 64; 128 and 256
def test_entries_come_in_the_order_they_are_read(ring, kp):
    out = (ctypes.c_int * 4)()
    for nck in range(1, 9):
        want = [(1, 0, j) for j in range(kp)]
        for c in range(nck):
            want += [(1, c + 1, j) for j in range(kp)] if c + 1 < nck else []
            want += [(0, c, h) for h in range(2)]
        assert ring.total(kp, nck) == len(want)
        for e, (k, c, part) in enumerate(want):
            ring.at(kp, nck, e, out)
            assert tuple(out[:3]) == (k, c, part)
            assert (ring.k_entry if k else ring.v_entry)(kp, nck, c, part) == e
            assert out[3] == (128 * (c + 1) if k else 128 * c + 64 * (part + 1))


@pytest.mark.parametrize("kp", [1, 2])
@pytest.mark.parametrize("chunk", [1, 16, 50, 256])
def test_early_entries_hold_prefix_keys_alone(ring, kp, chunk):
    out = (ctypes.c_int * 4)()
    for prefix in range(0, 700):
        nck = (prefix + chunk + 127) // 128
        n = ring.early(kp, nck, SLOTS, prefix)
        for e in range(n):
            ring.at(kp, nck, e, out)
            assert out[3] <= prefix, (prefix, e)
        if prefix >= 256:   # K of two chunks and the Vt of the first are prefix keys
            assert n == min(SLOTS, 2 * kp + 2, ring.total(kp, nck))
