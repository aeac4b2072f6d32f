"""The lockstep target walks and their end filters against the CPU oracle.

All outputs are integers or functions of one integer, so every comparison is
exact.  The cases sit at the edges of the kernel's tiles: 448 targets per pass
of a block's threads, 3 per thread, groups of 16 pairs, 32 nodes of a pair in
a warp's lanes, the smallest and the largest filter, lists around the bounds
of what goes to shared memory, hubs within and beyond the cached records.
"""
import numpy as np
import pytest

from test_gpu_parity import assert_parity, gpu_query, oracle_query, srk  # noqa: F401

pytestmark = pytest.mark.gpu


def ring_lists(n, d, seed):
    """Every node has exactly d in-neighbours (so the number of targets is n)."""
    rng = np.random.default_rng(seed)
    col = np.sort((np.arange(n)[:, None] + rng.integers(1, n, size=(n, d))) % n, axis=1)
    return np.arange(0, n * d + 1, d, dtype=np.int32), col.astype(np.int32).ravel()


@pytest.mark.parametrize("n", [2, 31, 447, 448, 449, 1343, 1345, 2689])
def test_target_blocks(srk, n):
    # repeated entries in a list are separate draws: keep the duplicates
    rp, col = ring_lists(n, 3, n)
    kw = dict(z_override=700.0, L_override=12)
    assert_parity(gpu_query(srk, rp, col, n // 2, 0.5, 3, **kw),
                  oracle_query(rp, col, n // 2, 0.5, 3, **kw))


@pytest.mark.parametrize("d", [1, 8, 9, 33, 64, 65, 200])
def test_own_lists(srk, d):
    rp, col = ring_lists(1500, d, d)
    kw = dict(z_override=3000.0, L_override=9)
    assert_parity(gpu_query(srk, rp, col, 7, 0.5, 4, **kw),
                  oracle_query(rp, col, 7, 0.5, 4, **kw))


@pytest.mark.parametrize("z,L", [(1.0, 0), (2.0, 1), (40.0, 2), (90.0, 3), (60.0, 33), (50.0, 70),
                                 (9000.0, 34)])
def test_pair_counts_and_lengths(srk, z, L):
    # long pairs: two nodes with one shared in-neighbour chain that never ends
    rp, col = ring_lists(400, 2, 11)
    kw = dict(z_override=z, L_override=L)
    assert_parity(gpu_query(srk, rp, col, 3, 0.5, 5, **kw), oracle_query(rp, col, 3, 0.5, 5, **kw))


@pytest.mark.parametrize("layout", ["narrow", "wide", "csr"])
@pytest.mark.parametrize("hubs", [1, 600])
def test_hubs_and_filter_sizes(srk, layout, hubs):
    """Hubs of in-degree 2,500 (600 of them: more than the cached records) that
    are also in-neighbours of up to 12,000 nodes (filters of the largest size),
    beside nodes that are in-neighbours of one or two (the smallest)."""
    import torch
    from srk_inputs import csr_from_edges
    rng = np.random.default_rng(hubs)
    n = 12000
    h = rng.choice(n, size=hubs, replace=False)
    src = [rng.integers(0, n, size=2500) for _ in h]
    dst = [np.full(2500, x) for x in h]
    src += [h[rng.integers(0, hubs, size=n)], rng.integers(0, n, size=n)]
    dst += [np.arange(n), np.arange(n)]
    rp, col = csr_from_edges(n, np.concatenate(src), np.concatenate(dst))
    s = int(h[0])
    dev = torch.device("cuda:0")
    with srk.srk_graph_load(torch.from_numpy(rp).to(dev), torch.from_numpy(col).to(dev),
                            layout=layout) as g:
        scores = torch.empty(n, dtype=torch.float64, device=dev)
        out = [torch.empty(n, dtype=t, device=dev) for t in (torch.int32, torch.int64, torch.int32)]
        stats = srk.SrkStats()
        srk.srk_single_source(g, s, 0.6, 0.5, 9, scores, out[0], out[1], step_counts=out[2],
                              stats=stats, z_override=900.0, L_override=15)
        again = torch.empty_like(scores)
        srk.srk_single_source(g, s, 0.6, 0.5, 9, again, z_override=900.0, L_override=15)
        torch.cuda.synchronize()
    gpu = (scores.cpu().numpy(), out[0].cpu().numpy().view(np.uint32),
           out[1].cpu().numpy().view(np.uint64), out[2].cpu().numpy().view(np.uint32), stats)
    assert_parity(gpu, oracle_query(rp, col, s, 0.5, 9, z_override=900.0, L_override=15))
    assert torch.equal(again, scores)  # the kernel that does not count steps


@pytest.mark.parametrize("lo,hi", [(0, 1), (100, 100), (17, 465), (999, 1000)])
def test_short_target_ranges_without_filters(srk, lo, hi):
    rp, col = ring_lists(1000, 5, 2)
    kw = dict(z_override=300.0, L_override=10)
    ref = oracle_query(rp, col, 20, 0.5, 6, **kw)
    got = gpu_query(srk, rp, col, 20, 0.5, 6, target_range=(lo, hi), **kw)
    for a, b in zip(got[:4], (ref.scores, ref.count, ref.wsum, ref.steps)):
        assert np.array_equal(a[lo:hi].astype(b.dtype), b[lo:hi])
    assert got[4].target_steps == int(ref.steps[lo:hi].sum())


@pytest.mark.parametrize("n", [447, 449, 895, 897, 1793])
def test_target_blocks_wide(srk, n):
    """8-byte entries: one target per thread for a query, two for shared walks."""
    import torch
    rp, col = ring_lists(n, 3, n)
    dev = torch.device("cuda:0")
    kw = dict(z_override=500.0, L_override=12)
    sources, c = [0, n // 2, n - 1], 0.6
    out = torch.empty((3, n), dtype=torch.float64, device=dev)
    cnt = torch.empty((3, n), dtype=torch.int32, device=dev)
    with srk.srk_graph_load(torch.from_numpy(rp).to(dev), torch.from_numpy(col).to(dev),
                            layout="wide") as g:
        for shared in (False, True):
            if shared:
                srk.srk_multi_source(g, sources, c, [0.5] * 3, 3, out, cnt, shared_walks=True, **kw)
            else:
                for i, s in enumerate(sources):
                    srk.srk_single_source(g, s, c, 0.5, 3, out[i], cnt[i], **kw)
            torch.cuda.synchronize()
            for i, s in enumerate(sources):
                ref = oracle_query(rp, col, s, 0.5, 3, shared_walks=shared, **kw)
                assert np.array_equal(out[i].cpu().numpy(), ref.scores)
                assert np.array_equal(cnt[i].cpu().numpy().view(np.uint32), ref.count)


@pytest.mark.parametrize("polls", ["0", "1"])
def test_waits_for_filters_that_give_up(srk, monkeypatch, polls):
    """SRK_WAIT_POLLS = 0: every block's first wait gives up, so the filters are
    read from global memory from then on; 1: some waits may.  Integers: equal."""
    rp, col = ring_lists(5000, 12, 8)
    kw = dict(z_override=4000.0, L_override=14)
    ref = oracle_query(rp, col, 9, 0.5, 21, **kw)
    monkeypatch.setenv("SRK_WAIT_POLLS", polls)
    for _ in range(3):
        assert_parity(gpu_query(srk, rp, col, 9, 0.5, 21, **kw), ref)


def batch_and_singles(srk, g, n, sources, eps, seed, **kw):
    """Dense batch outputs and the same queries one by one, as (scores, counts)."""
    import torch
    dev = torch.device("cuda:0")
    k = len(sources)
    out = [(torch.full((k, n), -3.0, dtype=torch.float64, device=dev),
            torch.full((k, n), 7, dtype=torch.int32, device=dev)) for _ in range(2)]
    st = srk.SrkStats()
    srk.srk_multi_source(g, sources, 0.6, eps, seed, *out[0], stats=st, **kw)
    steps = 0
    for i, s in enumerate(sources):
        one = srk.SrkStats()
        srk.srk_single_source(g, s, 0.6, eps[i], seed, out[1][0][i], out[1][1][i], stats=one)
        steps += one.target_steps
    torch.cuda.synchronize()
    return out, st.target_steps, steps


# 256 sources to a group, one cluster of 1 to 8 blocks a source; sources of 5e8 pairs
# x targets are walked by launches of their own beside the others of their group
@pytest.mark.parametrize("n,k,eps", [(2, 3, [0.9]), (447, 1, [0.2]), (449, 33, [0.3, 0.1]),
                                     (1345, 255, [0.4]), (1000, 256, [0.3]), (1000, 257, [0.3, 0.5]),
                                     (20000, 5, [0.008, 0.3, 0.1])])
def test_groups_of_sources(srk, n, k, eps):
    import torch
    rp, col = ring_lists(n, 5 if n > 5 else 1, n)
    if n >= 1000:  # every third node loses its list: no targets, and sources that meet nobody
        keep = np.repeat(np.arange(n) % 3 != 2, 5)
        col = col[keep]
        rp = np.concatenate([[0], np.cumsum(5 * (np.arange(n) % 3 != 2))]).astype(np.int32)
    eps = [eps[i % len(eps)] for i in range(k)]
    if n == 2:
        eps = [0.9] * k
    sources = [(i * 7) % n for i in range(k)]
    kw = dict(z_override=20.0) if n == 2 else {}
    dev = torch.device("cuda:0")
    with srk.srk_graph_load(torch.from_numpy(rp).to(dev), torch.from_numpy(col).to(dev)) as g:
        if n == 2:
            out = torch.empty((k, n), dtype=torch.float64, device=dev)
            srk.srk_multi_source(g, sources, 0.6, eps, 5, out, **kw)
            torch.cuda.synchronize()
            for i, s in enumerate(sources):
                assert np.array_equal(out[i].cpu().numpy(),
                                      oracle_query(rp, col, s, 0.9, 5, **kw).scores)
            return
        for kw in ({}, dict(no_graph=True)):
            (a, b), steps, want = batch_and_singles(srk, g, n, sources, eps, 5, **kw)
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and steps == want
        ref = oracle_query(rp, col, sources[-1], eps[-1], 5)
        assert np.array_equal(a[0][k - 1].cpu().numpy(), ref.scores)


@pytest.mark.parametrize("layout", ["narrow", "wide", "csr"])
@pytest.mark.parametrize("budget", [None, 1 << 20, 3 << 20, 6 << 20])
def test_groups_within_a_scratch_budget(srk, monkeypatch, layout, budget):
    """Budgets that leave room for no filters, for some, and for some groups."""
    import torch
    from srk_inputs import rmat_in_csr
    rp, col = rmat_in_csr(13, seed=4)
    n = rp.size - 1
    sources = [int(s) for s in np.argsort(-np.diff(rp), kind="stable")[:24]]
    eps = [0.1, 0.07, 0.2] * 8
    dev = torch.device("cuda:0")
    if budget:
        monkeypatch.setenv("SRK_BATCH_BYTES", str(budget))
    with srk.srk_graph_load(torch.from_numpy(rp).to(dev), torch.from_numpy(col).to(dev),
                            layout=layout) as g:
        (a, b), steps, want = batch_and_singles(srk, g, n, sources, eps, 8)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and steps == want


def test_small_sources_of_a_batch_run_together(srk):
    """64 queries that are small by themselves, as one batch: well below the time
    of as many calls (0.57 to 0.63 of it when the batch ran them one by one)."""
    import time

    import torch
    from srk_inputs import er_in_csr
    rp, col = er_in_csr(2000, 8.0, seed=2)
    n = rp.size - 1
    dev = torch.device("cuda:0")
    sources = [int(s) for s in np.flatnonzero(np.diff(rp) > 0)[:64]]
    out = torch.empty((64, n), dtype=torch.float64, device=dev)

    def best_of(f):
        times = []
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            f()
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
        return min(times)

    with srk.srk_graph_load(torch.from_numpy(rp).to(dev), torch.from_numpy(col).to(dev)) as g:
        batch = best_of(lambda: srk.srk_multi_source(g, sources, 0.6, [0.1] * 64, 7, out))
        loop = best_of(lambda: [srk.srk_single_source(g, s, 0.6, 0.1, 7, out[i])
                                for i, s in enumerate(sources)])
    assert batch < 0.4 * loop


@pytest.fixture(scope="module")
def far_graph(srk):
    """Lists of 13 on 2^20 nodes, with the wide layout (117 MB: beyond the L2, units of
    one target block in a row) and the narrow one (54 MB: within it)."""
    import torch
    n, d = 1 << 20, 13
    gen = torch.Generator(device="cuda")
    gen.manual_seed(6)
    col = torch.randint(0, n, (n * d,), generator=gen, device="cuda").to(torch.int32)
    rp = torch.arange(0, n * d + 1, d, dtype=torch.int32, device="cuda")
    with srk.srk_graph_load(rp, col, layout="wide") as far, \
            srk.srk_graph_load(rp, col, layout="narrow") as near:
        yield n, rp, col, far, near


@pytest.mark.parametrize("lo,hi", [(0, 1 << 20), (0, (1 << 20) - 1), (5, 453), (1000, 90001)])
def test_far_and_near_adjacency_agree(srk, far_graph, lo, hi):
    import torch
    n, rp, col, far, near = far_graph
    out = []
    for g in (far, near):
        sc = torch.zeros(n, dtype=torch.float64, device="cuda")
        ct, st = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
        ws = torch.zeros(n, dtype=torch.int64, device="cuda")
        srk.srk_single_source(g, 77, 0.6, 0.12, 3, sc, ct, ws, step_counts=st, target_range=(lo, hi))
        out.append((sc, ct, ws, st))
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(*out))
    some = np.unique(np.linspace(lo, hi - 1, 300).astype(np.int32))
    ref = oracle_query(rp.cpu().numpy(), col.cpu().numpy(), 77, 0.12, 3, targets=some)
    assert np.array_equal(out[0][0].cpu().numpy()[some], ref.scores)


@pytest.mark.parametrize("shared", [False, True])
def test_far_and_near_batches_agree(srk, far_graph, shared):
    import torch
    n, rp, col, far, near = far_graph
    sources, eps = [1, 77, 500000], [0.2, 0.12, 0.3]
    out = [torch.empty((3, n), dtype=torch.float64, device="cuda") for _ in range(2)]
    for g, o in zip((far, near), out):
        srk.srk_multi_source(g, sources, 0.6, eps, 9, o, shared_walks=shared)
    torch.cuda.synchronize()
    assert torch.equal(*out)


@pytest.mark.parametrize("z,part", [(1137.0, 1), (1137.0, 2), (1137.0, 20), (1137.0, 60), (100.0, 1),
                                    (100.0, 7)])
def test_ways_to_walk_agree(srk, far_graph, z, part):
    """Lists of 13 on 2^20 nodes: as the targets get fewer the layouts go over from end
    filters to a warp per target and to lockstep without filters, at lines of their
    own (117, 54 and 58 MB; 68, 30, 3, 1, 6 and 0.8 pairs x targets an edge)."""
    import torch
    n, rp, col, far, near = far_graph
    lo, hi = n // 9, n // 9 + (n - n // 9) // part
    if part == 1:
        lo, hi = 0, n
    some = np.unique(np.linspace(lo, hi - 1, 100).astype(np.int32))
    ref = oracle_query(rp.cpu().numpy(), col.cpu().numpy(), 77, 0.12, 3, targets=some, z_override=z)
    with srk.srk_graph_load(rp, col, layout="csr") as csr:
        for g in (far, near, csr):
            sc = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
            ct, st = (torch.full((n,), 9, dtype=torch.int32, device="cuda") for _ in range(2))
            ws = torch.full((n,), 9, dtype=torch.int64, device="cuda")
            stats = srk.SrkStats()
            srk.srk_single_source(g, 77, 0.6, 0.12, 3, sc, ct, ws, step_counts=st, stats=stats,
                                  z_override=z, target_range=(lo, hi))
            assert np.array_equal(sc.cpu().numpy()[some], ref.scores)
            assert np.array_equal(ct.cpu().numpy()[some].view(np.uint32), ref.count)
            assert np.array_equal(ws.cpu().numpy()[some].view(np.uint64), ref.wsum)
            assert np.array_equal(st.cpu().numpy()[some].astype(np.uint64), ref.steps)
            assert stats.target_steps == int(st[lo:hi].sum())
            assert bool((sc[:lo] == -1.0).all()) and bool((sc[hi:] == -1.0).all())
            assert bool((ct[:lo] == 9).all()) and bool((ws[hi:] == 9).all())


def pool_peak(srk, f):
    """Bytes that the library's pool handed out at most while f ran."""
    import torch
    torch.cuda.synchronize()
    _, used, _ = srk.srk_pool_stats(0, reset_high=True)
    f()
    torch.cuda.synchronize()
    return srk.srk_pool_stats(0)[2] - used


def test_scratch_budgets_hold(srk, monkeypatch):
    """SRK_BATCH_BYTES bounds the batch's scratch with its filters (the descriptors of 64
    sources, 4 KB each, come on top), SRK_TOPK_ROWS_BYTES the top-k rows with their
    histograms (per row some 200 bytes, and a batch of one small source, on top)."""
    import torch
    from srk_inputs import rmat_in_csr
    rp, col = rmat_in_csr(13, seed=4)
    n = rp.size - 1
    dev = torch.device("cuda:0")
    sources = [int(s) for s in np.argsort(-np.diff(rp), kind="stable")[:64]]
    out = torch.empty((64, n), dtype=torch.float64, device=dev)
    with srk.srk_graph_load(torch.from_numpy(rp).to(dev), torch.from_numpy(col).to(dev)) as g:
        for mb in (2, 4, 16):
            monkeypatch.setenv("SRK_BATCH_BYTES", str(mb << 20))
            peak = pool_peak(srk, lambda: srk.srk_multi_source(g, sources, 0.6, [0.1] * 64, 7, out))
            assert 0 < peak <= (mb << 20) + 64 * 4096 + 65536
        monkeypatch.setenv("SRK_BATCH_BYTES", "1")
        budget = 64 * 8 * n
        monkeypatch.setenv("SRK_TOPK_ROWS_BYTES", str(budget))
        o = [torch.empty((64, 10), dtype=t, device=dev) for t in (torch.int32, torch.float64)]
        peak = pool_peak(srk, lambda: srk.srk_multi_source_topk(
            g, sources, 0.6, [0.5] * 64, 7, 10, *o, z_override=60.0))
        assert 0 < peak <= budget + 64 * 256 + (200 << 10)


@pytest.mark.parametrize("n,d", [(1, 1), (3, 2), (1024, 5), (1025, 40), (4095, 16), (4096, 16),
                                 (4096, 17), (4097, 3)])
def test_graphs_ranked_by_one_block(srk, n, d):
    """At most 4,096 nodes and 65,536 edges; lists of 0, d or 2 d entries."""
    rng = np.random.default_rng(n + d)
    deg = np.array([0, d, 2 * d])[rng.integers(0, 3, size=n)] if n > 3 else np.full(n, d)
    if (n, d) in ((4096, 16), (4096, 17)):
        deg = np.full(n, d)
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    col = rng.integers(0, n, size=int(rp[-1])).astype(np.int32)
    s = int(np.flatnonzero(deg)[0])
    kw = dict(z_override=300.0, L_override=10)
    assert_parity(gpu_query(srk, rp, col, s, 0.5, 3, **kw), oracle_query(rp, col, s, 0.5, 3, **kw))
