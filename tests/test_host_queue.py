"""Arrow queues of the one-walker kernels and block shapes of cycle popping
(csrc/kc_host_plan.h), compiled with the host C++ compiler."""
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
extern "C" uint64_t hq_pop_bytes(int64_t n) { return kc_host::pop_small_bytes(n); }
extern "C" int hq_pop_threads(int64_t n) { return kc_host::pop_small_threads(n); }
extern "C" int hq_pop(int64_t n, int64_t twom, int64_t d) { return kc_host::pop_kind(n, twom, d); }
extern "C" uint64_t hq_trees_bytes(int64_t n) { return kc_host::pop_trees_bytes(n); }
extern "C" int64_t hq_trees_max(int contract) {
    return contract ? kc_host::kPopContractMax : kc_host::kPopTreesMax;
}
extern "C" int hq_pop_noalloc(int64_t n, int64_t t) { return kc_host::pop_noalloc(n, t); }
extern "C" int hq_serves(int64_t B, int64_t sms, int bit, int reject) {
    return kc_host::queue_serves(B, sms, bit, reject);
}
extern "C" int hq_in_order(int64_t B, int64_t n, int64_t sms, int bit) {
    return kc_host::transform_in_order(B, n, sms, bit);
}
extern "C" int64_t hq_pop_max() { return kc_host::kPopSmallMax; }
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
    lib.hq_pop_bytes.restype = ctypes.c_uint64
    lib.hq_pop_max.restype = ctypes.c_int64
    lib.hq_trees_bytes.restype = ctypes.c_uint64
    lib.hq_trees_max.restype = ctypes.c_int64
    for f in (lib.hq_pop_bytes, lib.hq_pop_threads, lib.hq_trees_bytes):
        f.argtypes = [ctypes.c_int64]
    lib.hq_pop.argtypes = [ctypes.c_int64] * 3
    lib.hq_serves.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int]
    lib.hq_in_order.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int64, ctypes.c_int]
    lib.hq_pop_noalloc.argtypes = [ctypes.c_int64] * 2
    return lib


def test_arrow_queues_fit_their_words(queue):
    """Every neighbour index of the largest degree fits the bits, and the queue
    (last arrow, the next ones, end mark) a half word."""
    for max_deg in list(range(1, 300)) + [1 << k for k in range(9, 31)]:
        b = queue.hq_bits(max_deg)
        assert b >= 2 and max_deg <= 1 << b and (b == 2 or max_deg > 1 << (b - 1))
        if b <= queue.hq_max_bits():
            slots = queue.hq_slots(b)
            assert slots >= 1
            assert b + slots * b + 1 <= 32 < b + (slots + 1) * b + 2


def test_every_wave_size_has_a_group(queue):
    for B in range(1, 20000):
        per_sm = -(-B // 152)
        assert queue.hq_group(B, 152) == (16 if 32 < per_sm <= 48 else 32)


def test_popped_trees_fit_a_block(queue):
    """14 bytes a vertex within 227 KB less the static part, ids in 16 bits."""
    top = queue.hq_pop_max()
    assert top < 1 << 16 and queue.hq_pop_bytes(top) + 64 <= 227 * 1024
    for n in (2, 3, 1024, 1025, 4096, 4097, top):
        assert 14 * n <= queue.hq_pop_bytes(n) <= 14 * n + 2
        assert queue.hq_pop_threads(n) in (128, 256, 512, 1024)
        assert queue.hq_pop(n, 10 * n, 1) == 1
    for contract, each in ((1, 6), (0, 4)):
        n = queue.hq_trees_max(contract)
        assert queue.hq_trees_bytes(n) == each * n <= 227 * 1024 - 64


def test_popping_follows_size_and_root(queue):
    small, trees = queue.hq_pop_max(), queue.hq_trees_max(1)
    assert queue.hq_pop(small + 1, 10 * small, small) == 2  # a hub: in memory
    assert queue.hq_pop(small + 1, 10 * small, 20) == 3     # else in a block
    assert queue.hq_pop(trees + 1, 10 * trees, 20) == 0     # until it does not fit
    assert queue.hq_pop(4000000, 68000000, 8000) == 2
    assert queue.hq_pop(9000, 1 << 32, 8999) == 3           # 32-bit volumes do not hold 2m


def test_many_trees_of_few_vertices_are_walked(queue):
    """Past 128 trees a vertex; from 256 vertices on the scratch limit (n x trees at most
    8 Mi) lets no call get there."""
    for n in (2, 3, 40, 100, 255):
        assert queue.hq_pop_noalloc(n, 128 * n) and not queue.hq_pop_noalloc(n, 128 * n + 1)
    for n in (256, 2000, queue.hq_trees_max(0)):
        assert queue.hq_pop_noalloc(n, (8 << 20) // n)
    assert not queue.hq_pop_noalloc(queue.hq_trees_max(0) + 1, 1)


@pytest.mark.parametrize("bit,reject,per_sm", [(0, 0, 160), (0, 1, 160), (1, 0, 320),
                                               (1, 1, 184)])
def test_waves_of_very_many_trees_take_a_lane_each(queue, bit, reject, per_sm):
    assert queue.hq_serves(1, 152, bit, reject)
    assert queue.hq_serves(per_sm * 152 - 1, 152, bit, reject)
    assert not queue.hq_serves(per_sm * 152, 152, bit, reject)


def test_many_transformed_trees_are_traversed_in_order(queue):
    for n in (2, 40, 2000, 1000000):
        assert not queue.hq_in_order(607, n, 152, 1) and queue.hq_in_order(608, n, 152, 1)
        line = 608 + n // 10
        assert not queue.hq_in_order(line - 1, n, 152, 0) and queue.hq_in_order(line, n, 152, 0)
