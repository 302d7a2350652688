"""The lane sampler (one tree per warp or block, cycle popping in rounds)
where it can go wrong: the edges of its word layout, of its shared-memory and
global-memory variants and of the stack of pending ends.  Trees are compared
with the oracle's sequential Wilson bit for bit."""
import numpy as np
import pytest
import torch

import paper_2510_20604_gb300 as rwc
import synth
from oracle import wilson as ow

pytestmark = pytest.mark.gpu


def _exact(g, T, opt=None, seed=1, tree0=0, flags=0, root=-1):
    G = rwc.Graph.from_synth(g, root=root, flags=flags)
    sums, st, par, vis = G.sample(T, seed=seed, tree0=tree0, want_trees=True, opt=opt)
    ref = ow.Sampler(g, root=G.root, seed=seed).sample(tree0, T, want_trees=True, nthreads=min(T, 8))
    assert np.array_equal(par.cpu().numpy(), ref["parents"])
    assert np.array_equal(vis.cpu().numpy(), ref["visits"])
    assert np.array_equal(sums.cpu().numpy(), ref["sums"])
    return st


def _heavy_pair(n, ratio):
    """A BA graph with one edge `ratio` times heavier than the others, between
    two vertices of small degree: a walk that enters the pair goes to and fro
    about `ratio` times, so two counts are large.  Returns (graph, hub)."""
    b = synth.ba(n, 2, seed=9)
    deg = np.diff(b.row_ptr)
    u, v, _ = b.undirected()
    w = np.ones(len(u), np.float32)
    w[np.argmin(deg[u] + deg[v])] = ratio
    return synth.from_edges(n, u, v, w), int(np.argmax(deg))


@pytest.mark.parametrize("n", [61, 62, 63, 126, 127, 190, 192, 193, 255, 256, 257, 1023])
def test_sizes_around_the_word_layout_and_the_stack(n):
    # p' takes one more bit at n + lanes + 2 = 2^b; the stack of pending ends
    # spills to global memory only for n > 192
    _exact(synth.ba(n, 2, seed=n), 40)
    _exact(synth.cycle(n), 6)


@pytest.mark.parametrize("mode", [rwc.MODE_AUTO, rwc.MODE_WALKER])
@pytest.mark.parametrize("T", [1, 3, 160, 700])
def test_threads_per_tree_follow_the_trees_per_sm(mode, T):
    _exact(synth.rgg(1500, 9.0, seed=3, sigma=0.5), T, rwc.Options(mode=mode), tree0=5)


@pytest.mark.parametrize("n", [55000, 57000, 58000])
@pytest.mark.parametrize("sigma", [None, 0.7])
def test_shared_and_global_words_meet(n, sigma):
    _exact(synth.rmat(16, 8, seed=2, sigma=sigma) if n == 57000 else synth.rgg(n, 8.0, seed=n, sigma=sigma), 3,
           flags=rwc.GRAPH_INT64_OFFSETS if sigma else 0)


def test_long_chains_spill_the_stack():
    # a grid above the shared-memory size (global words, inline rows) and a
    # path: long popped cycles fill the stack of pending ends
    _exact(synth.grid2d(250, 245), 2)
    _exact(synth.path(900), 5)


def test_counts_beyond_the_word_are_sampled_again():
    # 40000 vertices leave 15 bits for the count in a 32-bit word
    g, hub = _heavy_pair(40000, 300000.0)
    opt = rwc.Options(mode=rwc.MODE_WALKER)
    st = _exact(g, 3, opt, root=hub)
    assert st.chunks == 1
    G = rwc.Graph.from_synth(g, root=hub)
    ref, _, _, vis = G.sample(3, want_trees=True, opt=opt)
    assert int(vis.max()) > 32768
    s = torch.zeros(g.n, dtype=torch.float64, device="cuda")
    rwc.rwc_sample_trees(G.handle, 1, 0, 3, s, None, None, rwc.Options(mode=rwc.MODE_WALKER, async_status=1))
    rwc.rwc_sync_status(G.handle)
    assert torch.equal(s, ref)


@pytest.mark.parametrize("mode,ratio", [(rwc.MODE_SHARED, 1e6), (rwc.MODE_WALKER, 2e7)])
def test_count_limits_are_reported(mode, ratio):
    # SHARED allows 65535 pops of a vertex, WALKER 2^20 - 1
    g, hub = _heavy_pair(300, ratio)
    G = rwc.Graph.from_synth(g, root=hub)
    with pytest.raises(rwc.RWCError) as e:
        G.sample(16, opt=rwc.Options(mode=mode))
    assert e.value.status == 6 and "popped more than" in str(e.value)


@pytest.mark.parametrize("sched", [None, (128, 2600, 2, 0, 0), (64, 700, 3, 1, 1)])
def test_batch_bins_and_block_sizes(sched):
    # sizes on both sides of the bins' and block sizes' bounds, one kernel per
    # bin on forked streams or one after the other, and one launch per graph
    ns = [2, 3, 191, 193, 640, 641, 1281, 2500, 2501, 5000, 5001]
    gs = [synth.path(2) if n == 2 else synth.ba(n, 2, seed=n) if n > 5 else synth.cycle(n) for n in ns]
    B = rwc.Batch(gs)
    if sched:
        B.set_schedule(*sched)
    T = 5
    s, st = B.sample(T, seed=7)
    one, _ = B.sample(T, seed=7, per_graph_launch=1)
    assert torch.equal(s, one)
    roots, o = B.roots(), B.offsets
    sums = s.cpu().numpy()
    for i, g in enumerate(gs):
        ref = ow.Sampler(g, root=int(roots[i]), seed=7, graph_id=i).sample(0, T)
        assert np.array_equal(sums[o[i]:o[i + 1]], ref["sums"]), ns[i]
    assert st.trees == T * len(gs) and st.draws == int(sums.sum()) and st.rounds > 0


@pytest.mark.parametrize("T", [1, 2, 3, 5, 6, 7])
def test_batch_takes_every_tree_once(T):
    # more blocks than trees of one graph, tree counts of every remainder of
    # the schedule's trees per item, blocks of several warps
    gs = [synth.ba(n, 2, seed=n) for n in range(120, 190, 2)] * 5
    B = rwc.Batch(gs)
    B.set_schedule(512, 0, 4, 0, 1)
    s, st = B.sample(T, seed=3)
    sums, roots, o = s.cpu().numpy(), B.roots(), B.offsets
    for i in range(0, len(gs), 7):
        ref = ow.Sampler(gs[i], root=int(roots[i]), seed=3, graph_id=i).sample(0, T)
        assert np.array_equal(sums[o[i]:o[i + 1]], ref["sums"]), i
    assert st.draws == int(sums.sum()) and st.trees == T * len(gs)


@pytest.mark.parametrize("side,T", [(130, 2), (70, 160), (70, 900), (70, 1600)])
def test_stacks_are_refilled_from_global_memory(side, T):
    # popped cycles of a grid overflow the 192 ends of a warp's stack; once all
    # stacks are empty the overflow comes back (blocks of 256, 256, 128 and 64
    # threads by the trees that an SM gets)
    _exact(synth.grid2d(side, side), T, rwc.Options(mode=rwc.MODE_SHARED))


def test_stacks_are_refilled_in_a_batch():
    gs = [synth.grid2d(a, b) for a, b in ((45, 47), (60, 50), (69, 70), (90, 100))]
    for sched in ((512, 0, 4, 0, 1), (512, 2600, 4, 1, 1)):     # blocks only; the smallest by a warp
        B = rwc.Batch(gs)
        B.set_schedule(*sched)
        s, _ = B.sample(6, seed=11)
        sums, roots, o = s.cpu().numpy(), B.roots(), B.offsets
        for i, g in enumerate(gs):
            ref = ow.Sampler(g, root=int(roots[i]), seed=11, graph_id=i).sample(0, 6)
            assert np.array_equal(sums[o[i]:o[i + 1]], ref["sums"]), (sched, i)


@pytest.mark.parametrize("chunk", [0, 1, 2])
def test_counts_beyond_global_words_repeat_only_their_trees(chunk):
    # above the shared-memory size 32-bit words leave 15 bits for the count; one
    # tree, a part or all of a chunk's trees are listed
    g, hub = _heavy_pair(60000, 3e5)
    opt = rwc.Options(mode=rwc.MODE_WALKER, trees_per_chunk=chunk)
    G = rwc.Graph.from_synth(g, root=hub)
    _, _, _, vis = G.sample(7, want_trees=True, opt=opt)
    big = (vis.max(1).values > 32768).sum().item()
    assert 0 < big < 7
    _exact(g, 7, opt, root=hub)
    g, hub = _heavy_pair(60000, 2e6)
    _exact(g, 5, opt, root=hub)


@pytest.mark.parametrize("n", [2, 3, 33, 93, 94, 95, 222, 223, 448, 449])
def test_small_trees_by_one_warp(n):
    # p' takes one more bit at n + 34 = 2^b; blocks of one warp up to 448 vertices
    for g in (synth.path(n), synth.ba(n, 2, seed=n) if n > 5 else synth.complete(n)):
        st = _exact(g, 5)
        _exact(g, 5, rwc.Options(mode=rwc.MODE_WALKER), tree0=9)
        assert st.block_threads == (32 if n <= 448 else 256)
    if n >= 3:
        _exact(synth.cycle(n), 3)


@pytest.mark.parametrize("n", [30000, 60000])
def test_memory_budget_bounds_the_scratch(n):
    # words in shared memory (the blocks' pending ends are the scratch) and in global
    # memory; what the call takes from the device's pool
    import ctypes
    rt = ctypes.CDLL("libcudart.so.13")
    pool, high, budget = ctypes.c_void_p(), ctypes.c_uint64(0), 6 << 20
    g = synth.rgg(n, 8.0, seed=n)
    G = rwc.Graph.from_synth(g)
    ref, *_ = G.sample(200, seed=4, opt=rwc.Options(mode=rwc.MODE_WALKER))
    torch.cuda.synchronize()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    used_current, used_high = 7, 8
    before = ctypes.c_uint64()
    assert rt.cudaMemPoolGetAttribute(pool, used_current, ctypes.byref(before)) == 0
    assert rt.cudaMemPoolSetAttribute(pool, used_high, ctypes.byref(high)) == 0
    s, *_ = G.sample(200, seed=4, opt=rwc.Options(mode=rwc.MODE_WALKER, memory_budget=budget))
    assert rt.cudaMemPoolGetAttribute(pool, used_high, ctypes.byref(high)) == 0
    assert torch.equal(s, ref)
    assert 0 < high.value - before.value <= budget
