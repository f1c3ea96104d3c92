"""GPU tests of the walkers' waves against the CPU oracle: failed trees of a
pipelined wave, segment tables across waves."""
import ctypes

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


SMALL = {
    "K2": lambda: S.complete(2), "K3": lambda: S.complete(3), "star40": lambda: S.star(40),
    "cycle500": lambda: S.cycle(500),  # paths of more than 32 vertices are committed in chunks
    "er300": lambda: S.er_lcc(300, 0.02, 7), "grid17x13": lambda: S.grid_perturbed(17, 13, 0.25, 3),
    "cl3000": lambda: S.chung_lu(3000, 2.1, 8.0, 5),
}


@pytest.mark.parametrize("name,trees", [(k, 40) for k in SMALL] +
                         [("K3", 100000), ("star40", 3000), ("er300", 5000),
                          ("grid17x13", 6000), ("er300", 7200),
                          ("grid17x13", 9800), ("er300", 20000), ("grid17x13", 40000)])
def test_arrows_drawn_ahead_match_oracle(name, trees):
    """One walker per tree, one and two trees per warp (5000 and 6000 trees)."""
    g = SMALL[name]()
    with kc.KemenyGraph.from_graph(g, _cfg(walker=kc.KC_WALK_LANE)) as G:
        G.sample(17, trees)
        _check(g, G.samples(), 17, 0, trees)


@pytest.mark.parametrize("name,trees", [("cycle500", 64), ("grid17x13", 3600)])
def test_arrows_drawn_ahead_reject_match_oracle(name, trees):
    """Rejection by walk length, one tree and several trees per warp."""
    g = SMALL[name]()
    t0 = O.tau0(g)
    _, st = O.sample_batch(g, t0, 23, 0, 256)
    cap = int(np.quantile(st, 0.6))
    ids, f_ref, st_ref = O.accepted_samples(lambda a, c: O.sample_batch(g, t0, 23, a, c), cap,
                                            trees, block=2 * trees)
    with kc.KemenyGraph.from_graph(g, _cfg(walker=kc.KC_WALK_LANE, reject_steps=cap)) as G:
        G.sample(23, trees)
        got = G.samples()
    assert np.array_equal(got["sid"], ids)
    assert np.array_equal(got["steps"], st_ref)
    assert np.array_equal(got["f"], f_ref)


@pytest.mark.parametrize("n", [2, 3, 31, 33, 1024, 1025, 4096, 4097, 8192, 8193, 16000, 16001])
def test_popped_trees_match_oracle(n):
    """Cycle popping in shared memory (up to 16000 vertices; past them the walkers),
    at the edges of its block sizes: f, step counts and a kept tree."""
    g = S.complete(n) if n < 4 else S.complete_bipartite(min(25, n // 2), n - min(25, n // 2))
    t0 = O.tau0(g)
    with kc.KemenyGraph.from_graph(g, _cfg(keep_trees=1)) as G:
        G.sample(41, 20)
        G.sample(41, 13)
        _check(g, G.samples(), 41, 0, 33)
        for k in (0, 32):
            tr, ref = G.tree(k), O.tree(g, t0, 41, k)
            for key in ("parent", "depth", "din", "dout", "vol"):
                assert np.array_equal(tr[key], getattr(ref, key)), key


def test_popped_trees_at_the_step_cap():
    """A tree past the cap is left to the 32-walker kernel, whose cap is per walker."""
    g = SMALL["er300"]()
    with kc.KemenyGraph.from_graph(g, _cfg(step_cap=400)) as G:  # S is about 540
        G.sample(3, 40)
        _check(g, G.samples(), 3, 0, 40)
    with kc.KemenyGraph.from_graph(g, _cfg(step_cap=5)) as G:
        st = kc.kc_sample(G.h, 3, 40, check=False)
        assert kc.STATUS[st] == "KC_ERR_STEP_LIMIT"


@pytest.mark.parametrize("n", [16500, 38000, 38400])
def test_popped_trees_of_random_graphs_match_oracle(n):
    """No hub: trees in shared memory up to 38000 vertices, walkers past them."""
    g = S.er_lcc(n, 8.0 / n, 9)
    with kc.KemenyGraph.from_graph(g, _cfg(keep_trees=1)) as G:
        G.sample(47, 20)
        _check(g, G.samples(), 47, 0, 20)


@pytest.mark.parametrize("trees", [1, 40, 200])
def test_popped_trees_in_memory_match_oracle(trees):
    """Power-law graph with a hub as root, too large for shared memory; fewer trees
    than SMs and more, a kept tree, and trees conditioned on an edge (BSM insertion)."""
    g = S.chung_lu(20000, 2.1, 8.0, 5)
    t0 = O.tau0(g)
    with kc.KemenyGraph.from_graph(g, _cfg(keep_trees=1)) as G:
        G.sample(43, trees)
        _check(g, G.samples(), 43, 0, trees)
        tr, ref = G.tree(trees - 1), O.tree(g, t0, 43, trees - 1)
        for key in ("parent", "depth", "din", "dout", "vol"):
            assert np.array_equal(tr[key], getattr(ref, key)), key


@pytest.mark.parametrize("n,trees", [(2, 5), (1000, 40), (5000, 20), (56000, 3), (56001, 3)])
@pytest.mark.parametrize("cap", [0, 30000])
def test_trees_without_allocation_match_oracle(n, trees, cap):
    """kc_wilson_noalloc at the edges of its two ways: trees, step counts and the
    status, also where some trees pass the step cap."""
    torch = pytest.importorskip("torch")
    g = S.complete(2) if n == 2 else S.complete_bipartite(25, n - 25)
    t0 = O.tau0(g)
    ro, co = torch.from_numpy(g.row_off).cuda(), torch.from_numpy(g.col).cuda()
    par = torch.full((trees, n), -7, dtype=torch.int32, device="cuda")
    steps = torch.zeros(trees, dtype=torch.int64, device="cuda")
    status = torch.full((1,), 5, dtype=torch.int32, device="cuda")
    st = kc.load().kc_wilson_noalloc(n, ro.data_ptr(), co.data_ptr(), t0.r, 71, 4, trees, cap,
                                     par.data_ptr(), steps.data_ptr(), status.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    assert st == kc.KC_OK
    torch.cuda.synchronize()
    _, want = O.sample_batch(g, t0, 71, 4, trees)
    over = want > cap if cap else want < 0
    got = steps.cpu().numpy()
    assert int(status.item()) == int(over.any())
    assert np.array_equal(got[~over], want[~over])
    assert np.all(got[over] == cap + 1)
    for k in np.flatnonzero(~over)[:3]:
        assert np.array_equal(par[k].cpu().numpy(), O.tree(g, t0, 71, 4 + int(k)).parent)


@pytest.mark.parametrize("n", [60, 3000, 6000, 12000])
def test_noalloc_is_captured_after_a_first_call_of_another_size(n):
    """A call of any size can be captured once one call was made on the device: the
    replay gives the trees that a plain call gives."""
    torch = pytest.importorskip("torch")
    trees = 6

    def buffers(g):
        return (torch.from_numpy(g.row_off).cuda(), torch.from_numpy(g.col).cuda(),
                torch.zeros((trees, g.n), dtype=torch.int32, device="cuda"),
                torch.zeros(trees, dtype=torch.int64, device="cuda"),
                torch.zeros(1, dtype=torch.int32, device="cuda"))

    def call(g, b, stream):
        assert kc.load().kc_wilson_noalloc(g.n, b[0].data_ptr(), b[1].data_ptr(), 0, 5, 9, trees,
                                           0, b[2].data_ptr(), b[3].data_ptr(), b[4].data_ptr(),
                                           stream.cuda_stream) == kc.KC_OK

    first = S.complete(5)
    call(first, buffers(first), torch.cuda.current_stream())
    g = S.complete_bipartite(25, n - 25)
    b, plain = buffers(g), buffers(g)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side):
        call(g, b, side)
    graph.replay()
    torch.cuda.synchronize()
    call(g, plain, torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(b[2:], plain[2:]))
    assert int(b[3].min()) >= n - 1


def _hubs_first(n):
    """Vertex 0 joined to the next ones (up to 63), the others spread under those: a root 0
    whose neighbours in id are internal."""
    hubs = max(1, min(63, (n - 1) // 2))
    u = np.arange(1, n)
    return S.csr_from_edges(n, u, np.where(u <= hubs, 0, 1 + (u - 1 - hubs) % hubs))


@pytest.mark.parametrize("n", [2, 3, 128, 129, 3000, 20000])
def test_root_zero_is_never_taken_for_a_leaf(n):
    """The path tree, popped trees and single-tree reads of a graph rooted at vertex 0."""
    g = _hubs_first(n)
    t0 = O.tau0(g, 0)
    cfg = _cfg(keep_trees=1, root=0)
    with kc.KemenyGraph.from_graph(g, cfg) as G:
        tau = G.tau0()
        assert np.array_equal(tau["in0"], t0.in0) and np.array_equal(tau["out0"], t0.out0)
        G.sample(29, 40)
        f_ref, st_ref = O.sample_batch(g, t0, 29, 0, 40)
        got = G.samples()
        assert np.array_equal(got["f"], f_ref) and np.array_equal(got["steps"], st_ref)
        for k in range(0, 40, 13):
            tr, ref = G.tree(k), O.tree(g, t0, 29, k)
            for key in ("parent", "depth", "din", "dout", "vol"):
                assert np.array_equal(tr[key], getattr(ref, key)), key


@pytest.mark.parametrize("n", [40, 4000, 16001])
@pytest.mark.parametrize("cap", [5, -1, 0])
def test_step_cap_holds_for_trees_without_a_cycle(n, cap):
    """A star rooted at its centre pops nothing: a tree still departs n - 1 times, and
    a cap below that (cap <= 0: n - 1 + cap) ends it."""
    torch = pytest.importorskip("torch")
    g, trees = S.star(n), 40
    cap = cap if cap > 0 else n - 1 + cap
    root = int(np.argmax(np.diff(g.row_off)))
    ro, co = torch.from_numpy(g.row_off).cuda(), torch.from_numpy(g.col).cuda()
    par = torch.zeros((trees, n), dtype=torch.int32, device="cuda")
    steps = torch.zeros(trees, dtype=torch.int64, device="cuda")
    status = torch.full((1,), 5, dtype=torch.int32, device="cuda")
    assert kc.load().kc_wilson_noalloc(n, ro.data_ptr(), co.data_ptr(), root, 5, 0, trees, cap,
                                       par.data_ptr(), steps.data_ptr(), status.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream) == kc.KC_OK
    torch.cuda.synchronize()
    assert int(status.item()) == int(cap < n - 1)
    assert np.all(steps.cpu().numpy() == min(n - 1, cap + 1))
    # AUTO: the 32-walker kernel decides, whose cap is per walker
    said = []
    for walker in (kc.KC_WALK_AUTO, kc.KC_WALK_WARP):
        with kc.KemenyGraph.from_graph(g, _cfg(walker=walker, step_cap=cap)) as G:
            said.append(kc.STATUS[kc.kc_sample(G.h, 3, trees, check=False)])
    assert said[0] == said[1]
    assert cap < n - 1 or said[0] == "KC_OK"


@pytest.mark.parametrize("trees", [128 * 60, 128 * 60 + 1, 140000])
@pytest.mark.parametrize("cap", [0, 100])
def test_many_small_trees_without_allocation_match_oracle(trees, cap):
    """Either side of the line between a block per tree and a lane per tree, and the largest
    call that the scratch array takes: step counts, parents and the status."""
    torch = pytest.importorskip("torch")
    g = S.complete_bipartite(7, 53)
    n, t0 = g.n, O.tau0(g)
    if trees > (8 << 20) // n:
        trees = (8 << 20) // n
    ro, co = torch.from_numpy(g.row_off).cuda(), torch.from_numpy(g.col).cuda()
    par = torch.full((trees, n), -7, dtype=torch.int32, device="cuda")
    steps = torch.zeros(trees, dtype=torch.int64, device="cuda")
    status = torch.full((1,), 5, dtype=torch.int32, device="cuda")
    assert kc.load().kc_wilson_noalloc(n, ro.data_ptr(), co.data_ptr(), t0.r, 73, 2, trees, cap,
                                       par.data_ptr(), steps.data_ptr(), status.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream) == kc.KC_OK
    torch.cuda.synchronize()
    _, want = O.sample_batch(g, t0, 73, 2, trees)
    over = want > cap if cap else want < 0
    assert int(status.item()) == int(over.any())
    got = steps.cpu().numpy()
    assert np.array_equal(got[~over], want[~over]) and np.all(got[over] == cap + 1)
    for k in [*np.flatnonzero(~over)[:2], *np.flatnonzero(~over)[-2:]]:
        assert np.array_equal(par[k].cpu().numpy(), O.tree(g, t0, 73, 2 + int(k)).parent)


@pytest.mark.parametrize("name,variant,per_sm", [("K3", 1, 160), ("er300", 1, 160),
                                                 ("er300", 2, 320), ("grid17x13", 2, 320)])
def test_a_lane_per_tree_matches_oracle(name, variant, per_sm):
    """So many trees that the LANE walker takes a lane for each, both variants of f."""
    g, trees = SMALL[name](), per_sm * 152
    with kc.KemenyGraph.from_graph(g, _cfg(walker=kc.KC_WALK_LANE, ttf_variant=variant)) as G:
        G.sample(19, trees)
        _check(g, G.samples(), 19, 0, trees)


@pytest.mark.parametrize("variant", [1, 2])
def test_a_lane_per_tree_under_rejection_matches_oracle(variant):
    g = SMALL["grid17x13"]()
    t0 = O.tau0(g)
    _, st = O.sample_batch(g, t0, 31, 0, 256)
    cap, trees = int(np.quantile(st, 0.6)), 184 * 152
    ids, f_ref, st_ref = O.accepted_samples(lambda a, c: O.sample_batch(g, t0, 31, a, c), cap,
                                            trees, block=2 * trees)
    with kc.KemenyGraph.from_graph(g, _cfg(walker=kc.KC_WALK_LANE, reject_steps=cap,
                                           ttf_variant=variant)) as G:
        G.sample(31, trees)
        got = G.samples()
    assert np.array_equal(got["sid"], ids)
    assert np.array_equal(got["steps"], st_ref) and np.array_equal(got["f"], f_ref)


@pytest.mark.parametrize("pinned", [True, False])
def test_creation_waits_for_copies_into_its_arrays(pinned):
    """A handle from host arrays that an asynchronous copy queued before the call still
    fills, and one from device arrays under the host flag: the runtime orders and finds both."""
    torch = pytest.importorskip("torch")
    g = SMALL["er300"]()
    dev = [torch.from_numpy(x).cuda() for x in (g.row_off, g.col)]
    src = dev
    if pinned:
        src = [torch.zeros(x.shape, dtype=x.dtype).pin_memory() for x in dev]
    with kc.KemenyGraph.from_graph(g):  # sets the device up: no step of the next one waits
        pass
    torch.cuda.synchronize()
    if pinned:
        with torch.cuda.stream(torch.cuda.default_stream()):
            torch.cuda._sleep(200_000_000)
            for h, d in zip(src, dev):
                h.copy_(d, non_blocking=True)
    h, cfg = ctypes.c_void_p(), _cfg()
    st = kc.load().kc_graph_create(g.n, src[0].data_ptr(), src[1].data_ptr(), ctypes.byref(cfg),
                                   ctypes.byref(h))
    assert kc.STATUS[st] == "KC_OK"
    try:
        kc.kc_sample(h, 17, 20)
        _check(g, kc.kc_get_samples(h, 0, 20), 17, 0, 20)
    finally:
        kc.kc_graph_destroy(h)


@pytest.mark.parametrize("n", [40002, 70002])
def test_lane_walker_without_queues_matches_oracle(n):
    """Neighbour indices too wide for an arrow queue (a vertex of degree n - 2): a lane per
    tree, in plain and (70002 vertices) pipelined waves, also rejecting and at the cap."""
    g = S.complete_bipartite(2, n - 2)
    t0 = O.tau0(g)
    with kc.KemenyGraph.from_graph(g, _cfg(walker=kc.KC_WALK_LANE)) as G:
        G.sample(53, 12)
        _check(g, G.samples(), 53, 0, 12)
    _, st = O.sample_batch(g, t0, 59, 0, 32)
    cap = int(np.quantile(st, 0.6))
    ids, f_ref, st_ref = O.accepted_samples(lambda a, c: O.sample_batch(g, t0, 59, a, c), cap,
                                            10, block=32)
    with kc.KemenyGraph.from_graph(g, _cfg(walker=kc.KC_WALK_LANE, reject_steps=cap)) as G:
        G.sample(59, 10)
        got = G.samples()
    assert np.array_equal(got["sid"], ids)
    assert np.array_equal(got["steps"], st_ref) and np.array_equal(got["f"], f_ref)
    with kc.KemenyGraph.from_graph(g, _cfg(walker=kc.KC_WALK_LANE, step_cap=5000)) as G:
        assert kc.STATUS[kc.kc_sample(G.h, 3, 8, check=False)] == "KC_ERR_STEP_LIMIT"
        assert G.stats()["pool_trees"] == 0


def _clique_on_a_path(k, length):
    """K_k with a path of `length` edges from its vertex k - 1; its far end is the last id.
    A clique vertex departs about k x length times from there on the way to that end."""
    iu, iv = np.triu_indices(k, 1)
    p = np.arange(k - 1, k + length - 1)
    return S.csr_from_edges(k + length, np.r_[iu, p], np.r_[iv, p + 1])


def test_pops_past_their_count_field_are_walked():
    """More pops of one vertex (about 10000) than a popped tree counts (8191): the walkers
    give the oracle's trees, through a handle and without allocation."""
    torch = pytest.importorskip("torch")
    g, trees = _clique_on_a_path(100, 100), 6
    root = g.n - 1
    t0 = O.tau0(g, root)
    f_ref, st_ref = O.sample_batch(g, t0, 61, 0, trees)
    with kc.KemenyGraph.from_graph(g, _cfg(keep_trees=1, root=root, ttf_variant=1)) as G:
        G.sample(61, trees)
        got = G.samples()
        assert np.array_equal(got["steps"], st_ref) and np.array_equal(got["f"], f_ref)
        assert np.array_equal(G.tree(3)["parent"], O.tree(g, t0, 61, 3).parent)
    ro, co = torch.from_numpy(g.row_off).cuda(), torch.from_numpy(g.col).cuda()
    par = torch.zeros((trees, g.n), dtype=torch.int32, device="cuda")
    steps = torch.zeros(trees, dtype=torch.int64, device="cuda")
    status = torch.full((1,), 5, dtype=torch.int32, device="cuda")
    assert kc.load().kc_wilson_noalloc(g.n, ro.data_ptr(), co.data_ptr(), root, 61, 0, trees, 0,
                                       par.data_ptr(), steps.data_ptr(), status.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream) == kc.KC_OK
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and np.array_equal(steps.cpu().numpy(), st_ref)
    for k in range(trees):
        assert np.array_equal(par[k].cpu().numpy(), O.tree(g, t0, 61, k).parent)


def test_a_batched_wave_past_a_cap_is_drawn_again():
    """One graph of a batched call passes its cap under popping, another under the queue
    walk: the wave is repeated with 32 walkers, whose cap is per walker."""
    graphs = [SMALL[k]() for k in ("er300", "cycle500", "cl3000", "K3")]
    caps = []
    for g in graphs:
        _, st = O.sample_batch(g, O.tau0(g), 67, 0, 40)
        caps.append(int(st.max()) - 1)
    for capped in ([0], [1], [0, 1]):
        Gs = [kc.KemenyGraph.from_graph(g, _cfg(step_cap=caps[k] if k in capped else 0))
              for k, g in enumerate(graphs)]
        try:
            kc.kc_sample_multi([G.h for G in Gs], [67] * 4, [40] * 4)
            for g, G in zip(graphs, Gs):
                _check(g, G.samples(), 67, 0, 40)
        finally:
            for G in Gs:
                G.close()


def test_kept_trees_of_every_popped_kind_in_a_batched_call():
    """In one call: trees in shared memory with and without f (16500 vertices, no hub), in
    memory (20000, a hub), and the walkers' trees; f, step counts and kept trees."""
    graphs = [SMALL["er300"](), S.er_lcc(16500, 8.0 / 16500, 9), S.chung_lu(20000, 2.1, 8.0, 5),
              SMALL["grid17x13"](), S.er_lcc(40000, 8.0 / 40000, 9)]
    Gs = [kc.KemenyGraph.from_graph(g, _cfg(keep_trees=1)) for g in graphs]
    try:
        for first in (0, 9):
            kc.kc_sample_multi([G.h for G in Gs], [71] * 5, [9] * 5)
            for g, G in zip(graphs, Gs):
                _check(g, G.samples(first, 9), 71, first, 9)
        for g, G in zip(graphs, Gs):
            t0 = O.tau0(g)
            for k in (0, 8, 9, 17):
                tr, ref = G.tree(k), O.tree(g, t0, 71, k)
                for key in ("parent", "depth", "din", "dout", "vol"):
                    assert np.array_equal(tr[key], getattr(ref, key)), key
    finally:
        for G in Gs:
            G.close()
