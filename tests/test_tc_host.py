"""The tensor-core kernels' host-checkable arithmetic (csrc/kd_tc_host.h), compiled here with
the host compiler."""

import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2609_11687_gb300", "csrc")

SHIM = r"""
#include "kd_tc_host.h"
extern "C" int last_parity(int issued, int slots, int s) { return kd::ring_last_parity(issued, slots, s); }
extern "C" int smem_floor(int cols) { return kd::tc_smem_floor(cols); }
extern "C" int smem_per_sm() { return kd::kSmemPerSM; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("tc_host")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


class _Barrier:
    """An mbarrier's phase: waiting for a parity succeeds once the phase of that parity, the
    current one or the one before, is complete."""

    def __init__(self):
        self.complete = 0  # phases completed

    def reads_complete(self, parity):
        return (self.complete & 1) != parity


def test_ring_drain_waits_for_every_copy(lib):
    """After any number of copies, with any of the last ones (one per slot at most) still in
    flight, the wait for the returned parity holds exactly while the slot's copy is missing; a
    slot that no copy used is not waited for."""
    for slots in range(1, 9):
        for issued in range(0, 4 * slots + 3):
            for in_flight in range(0, min(slots, issued) + 1):  # a slot's next copy follows its last one's landing
                bars = [_Barrier() for _ in range(slots)]
                for i in range(issued - in_flight):
                    bars[i % slots].complete += 1
                missing = {i % slots for i in range(issued - in_flight, issued)}
                for s in range(slots):
                    parity = lib.last_parity(issued, slots, s)
                    if s >= issued:
                        assert parity == -1
                        continue
                    assert bars[s].reads_complete(parity) == (s not in missing)
                    # either parity, as a loop's end, would not have waited
                    assert bars[s].reads_complete(0) or bars[s].reads_complete(1)


def test_ctas_that_fit_on_an_sm_have_their_tmem_there(lib):
    """Any set of CTAs of 256 and 512 columns whose shared memory fits (1 KB reserved each, at
    least the floor of dynamic memory) needs no more than the SM's 512 columns; two of 256 or one
    of 512 do fit, beside 2 KB of static memory."""
    total = lib.smem_per_sm()
    assert total == 228 * 1024
    size = {c: lib.smem_floor(c) + 1024 for c in (256, 512)}
    for a in range(8):
        for b in range(4):
            if a * size[256] + b * size[512] <= total:
                assert 256 * a + 512 * b <= 512, (a, b)
    assert 2 * (size[256] + 2048) <= total and size[512] + 2048 <= total
    assert all(lib.smem_floor(c) <= 227 * 1024 for c in (256, 512))
