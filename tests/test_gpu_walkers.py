"""GPU tests of the walkers' waves against the CPU oracle: failed trees of a
pipelined wave, segment tables across waves."""
import numpy as np
import pytest

import oracle as O
from paper_2511_16356_gb300 import synth as S

pytestmark = pytest.mark.gpu

kc = pytest.importorskip("paper_2511_16356_gb300.kc")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2511_16356_gb300 import build as kbuild

    kbuild.build()
    kc.load()


def _cfg(**kw):
    c = kc.kc_config_default()
    c.keep_trees = 0
    for k, v in kw.items():
        setattr(c, k, v)
    return c


def _check(g, got, seed, first, count):
    f_ref, st_ref = O.sample_batch(g, O.tau0(g), seed, first, count)
    assert np.array_equal(got["steps"], st_ref)
    assert np.array_equal(got["f"], f_ref)


@pytest.fixture(scope="module")
def grid260():
    return S.grid_perturbed(260, 260, 0.25, 2)  # large enough for pipelined waves


@pytest.mark.parametrize("walker", [kc.KC_WALK_AUTO, kc.KC_WALK_LANE, kc.KC_WALK_WARP])
def test_step_limit_in_a_pipelined_wave(grid260, walker):
    """Trees that stop at the step cap are never traversed: the call reports
    the cap and leaves the pool as it was."""
    with kc.KemenyGraph.from_graph(grid260, _cfg(walker=walker, step_cap=5000)) as G:
        st = kc.kc_sample(G.h, 3, 8, check=False)
        assert kc.STATUS[st] == "KC_ERR_STEP_LIMIT"
        assert G.stats()["pool_trees"] == 0


def test_segment_tables_survive_a_later_pipelined_wave(grid260):
    """The autotuner's plain pilot waves size the segment tables; a smaller
    pipelined wave after them still has its tables."""
    with kc.KemenyGraph.from_graph(grid260, _cfg(autotune=1)) as G:
        G.sample(5, 64)
        G.sample(5, 4)
        _check(grid260, G.samples(), 5, 0, 68)
