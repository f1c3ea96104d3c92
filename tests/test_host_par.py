"""Words of the order-free traversal (csrc/kc_host_par.h), compiled with the host C++
compiler: sizes by reports in any order of the vertices' threads."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_16356_gb300", "csrc")

SHIM = r"""
#include "kc_host_par.h"
// word: children counted; a vertex's thread after the other, in the order given.  Returns
// the number of vertices that reached the root with a wrong size.
extern "C" int hp_up(int n, int root, const int32_t *par, const int32_t *order, uint64_t *word,
                     int32_t *size) {
    int bad = 0;
    for (int i = 0; i < n; ++i) {
        int32_t x = order[i], sx = 1;
        if (!kc_host::par_is_leaf(word[x], x, root)) continue;
        for (;;) {
            const int32_t p = par[x];
            size[x] = sx;
            if (p < 0) {
                word[x] = kc_host::par_at(0, x);
                bad += sx != n;
                break;
            }
            const uint64_t old = word[p];
            word[p] = old + kc_host::par_report(sx);
            word[x] = kc_host::par_at((uint32_t)kc_host::par_sizes(old) + 1u, p);
            if (!kc_host::par_was_last(old)) break;
            sx = 1 + kc_host::par_sizes(old) + sx;
            x = p;
        }
    }
    return bad;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("hostpar")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"),
                    "-o", str(d / "shim.so")], check=True, capture_output=True)
    return ctypes.CDLL(str(d / "shim.so"))


@pytest.mark.parametrize("root", [0, 1, 4])
@pytest.mark.parametrize("n", [5, 40, 700])
def test_reports_in_any_order_of_the_threads(lib, n, root):
    """Also when the root's own thread comes to it after the tree is finished."""
    rng = random.Random(100 * n + root)
    for trial in range(20):
        ids = [root] + rng.sample([v for v in range(n) if v != root], n - 1)
        par = [-1] * n
        for k in range(1, n):
            par[ids[k]] = ids[rng.randrange(k)]
        sizes = [1] * n
        for v in reversed(ids[1:]):
            sizes[par[v]] += sizes[v]
        order = rng.sample(range(n), n)
        if trial % 2:
            order.remove(root)
            order.append(root)
        word = [0] * n
        for p in par:
            if p >= 0:
                word[p] += 1 << 32
        a32 = ctypes.c_int32 * n
        c_word, c_size = (ctypes.c_uint64 * n)(*word), a32()
        assert lib.hp_up(n, root, a32(*par), a32(*order), c_word, c_size) == 0
        assert list(c_size) == sizes
