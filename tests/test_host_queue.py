"""Arrow queues of the one-walker kernels (csrc/kc_host_plan.h), compiled with the
host C++ compiler."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_16356_gb300", "csrc")

SHIM = r"""
#include "kc_host_plan.h"
extern "C" int hq_bits(int64_t d) { return kc_host::queue_bits(d); }
extern "C" int hq_slots(int b) { return kc_host::queue_slots(b); }
extern "C" int hq_group(int64_t B, int64_t sms) { return kc_host::queue_group(B, sms); }
extern "C" int hq_max_bits() { return kc_host::kMaxQueueBits; }
extern "C" int hq_width() { return kc_host::kQueueWidth; }
"""


@pytest.fixture(scope="module")
def queue(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("hostqueue")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"),
                    "-o", str(d / "shim.so")], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "shim.so"))
    lib.hq_bits.argtypes = [ctypes.c_int64]
    lib.hq_group.argtypes = [ctypes.c_int64, ctypes.c_int64]
    return lib


def test_arrow_queues_fit_their_words(queue):
    """Every neighbour index of the largest degree fits the bits, and the queue
    (last arrow, the next ones, end mark) its width."""
    for max_deg in list(range(1, 300)) + [1 << k for k in range(9, 31)]:
        b = queue.hq_bits(max_deg)
        assert b >= 1 and max_deg <= 1 << b and (b == 1 or max_deg > 1 << (b - 1))
        if b <= queue.hq_max_bits():
            slots = queue.hq_slots(b)
            assert slots >= 1
            assert b + slots * b + 1 <= queue.hq_width() < b + (slots + 1) * b + 1


def test_every_wave_size_has_a_group(queue):
    got = [queue.hq_group(B, 152) for B in range(1, 20000)]
    assert set(got) == {32, 16, 8} and got == sorted(got, reverse=True)
