"""Paths that ordinary sizes do not reach, brought within reach of small data by
a context's test limits: the allocation-free join whose waits run out or whose
task queue fills (its launch behind then redoes every pair, and the next call
clears the queue), joins whose list of handed-over parity rays fills, dataset joins that leave the
joint walk at a queue or the list of leaf pairs, and the tiled join with the
host gathering the cells.  All against the oracle."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2609_24513_gb300 import pierce, synth
from test_gpu_join import _bipyramid
from test_zz_no_alloc import _noalloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = pierce.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def dense():
    # bipyramids: nearly all their node pairs overlap, so that stacks fill
    m, tw = (_bipyramid(300, (0.5, 0.5, 0.5), 0.2, 0.2, phase=p) for p in (0.0, 0.5))
    A, B = synth.concat([m, m, tw]), synth.concat([m, tw, synth.translate(m, (1.0, 0.0, 0.0))])
    cand = np.array([(i, j) for i in range(3) for j in range(3)], np.int32)
    truth = oracle.join(A, B, cand, tier=2).astype(bool)
    return A, B, np.tile(cand, (4, 1)), np.tile(truth, 4)


@pytest.mark.parametrize("W,L", [(2, 1), (4, 2), (8, 1)])
@pytest.mark.parametrize("limits", [dict(noalloc_polls=1), dict(noalloc_queue=1),
                                    dict(noalloc_queue=40), dict(noalloc_queue=2000)])
def test_noalloc_join_that_fails_over(ctx, dense, W, L, limits):
    torch = pytest.importorskip("torch")
    A, B, cand, truth = dense
    assert truth.any() and not truth.all()
    ha, hb = ctx.load(A), ctx.load(B)
    ctx.build(ha, W, L)
    ctx.build(hb, W, L)

    def call():
        before = ctx.counters()["pairs_refined"]
        k, pairs, flags = _noalloc(ctx, ha, hb, cand, torch)
        assert np.array_equal(flags.astype(bool), truth)
        assert k == int(truth.sum()) and np.array_equal(pairs, cand[truth])
        return ctx.counters()["pairs_refined"] - before

    assert call() == len(cand)            # the streaming launch did it
    for _ in range(2):                    # the limit, then a call without it
        pierce.pj_set_test_limits(ctx.h, **limits)
        refined = [call() for _ in range(2)]
        pierce.pj_set_test_limits(ctx.h)
        if limits.get("noalloc_polls") or limits.get("noalloc_queue") == 1:
            assert min(refined) > len(cand)   # the launch behind it redid the pairs
        assert call() == len(cand)
    pierce.pj_free_dataset(ctx.h, ha)
    pierce.pj_free_dataset(ctx.h, hb)


def test_touching_boxes_beyond_the_parity_list(ctx):
    # the same two boxes 2,200,000 times: both directions' first vertices lie on
    # the other's surface, more directions than 2^22.  Threads look at further
    # vertices themselves, so that nothing is redone
    box = synth.concat([synth.box((1000, 1000, 1000), (9000, 9000, 9000))])
    ha, hb = ctx.load(box), ctx.load(box)
    ctx.build(ha, 4, 2)
    ctx.build(hb, 4, 2)
    launches = []
    for n in (2000, 2200000):
        before = ctx.counters()["kernel_launches"]
        got, info = ctx.join(ha, hb, cand=np.zeros((n, 2), np.int32))
        assert info["n_candidates"] == n and len(got) == 0      # identical meshes
        launches.append(ctx.counters()["kernel_launches"] - before)
    assert launches[0] == launches[1]
    pierce.pj_free_dataset(ctx.h, ha)
    pierce.pj_free_dataset(ctx.h, hb)


@pytest.fixture(scope="module")
def walls():
    # towers of 8 to 441 wall vertices against neighbours that share the wall,
    # stand inside against it, are the same, or touch in an edge
    sets = []
    for per, bands in ((1, 1), (2, 1), (3, 2), (4, 15), (20, 20)):
        foot = np.rint(synth._rect(8000, 8000, per) + 50000)
        t = synth.building(foot, 1000, 8000, 100, bands)
        sets.append((t, [synth.translate(t, (8000, 0, 0)), t, synth.translate(t, (8000, 8000, 0)),
                         synth.box((46000, 47000, 2000), (48000, 51000, 6000))]))
    A = synth.concat([t for t, _ in sets])
    B = synth.concat([m for _, ms in sets for m in ms])
    cand = np.array([(i, 4 * i + k) for i in range(len(sets)) for k in range(4)], np.int32)
    return A, B, cand, {p: oracle.join(A, B, cand, predicate=p).astype(bool)
                        for p in ("intersects", "contains", "within")}


@pytest.mark.parametrize("limit", [0, 1, 7, 64])
@pytest.mark.parametrize("W,L,levels", [(2, 1, 0), (4, 2, 0), (8, 4, 0), (4, 2, 4)])
def test_surface_vertices_over_parity_list_sizes(ctx, walls, limit, W, L, levels):
    # no limit: the first directions go to warps, then those past 8, 16, ...
    # vertices; small lists: threads go on to the last vertex
    A, B, cand, truth = walls
    assert truth["intersects"].any() and truth["contains"].any()
    ha, hb = ctx.load(A), ctx.load(B)
    ctx.build(ha, W, L)
    ctx.build(hb, W, L)
    pierce.pj_set_test_limits(ctx.h, parity_list=limit)
    for reps in (1, 1500):
        c = np.tile(cand, (reps, 1))
        for pred, t in truth.items():
            got, _ = ctx.join(ha, hb, cand=c, width=W, leaf_size=L, predicate=pred,
                              wave_levels=levels)
            assert np.array_equal(got, c[np.tile(t, reps)]), (pred, reps)
    pierce.pj_set_test_limits(ctx.h)
    pierce.pj_free_dataset(ctx.h, ha)
    pierce.pj_free_dataset(ctx.h, hb)


@pytest.mark.parametrize("n", [1, 31, 400, 90000])
def test_noalloc_join_finds_bad_ids_and_replays(ctx, n):
    # ids out of range anywhere in a warp's share; then the queued launches
    # captured once and replayed over other candidates
    torch = pytest.importorskip("torch")
    A, B = synth.tiny_spheres(1001)
    every = np.array([(i, j) for i in range(A.nmesh) for j in range(B.nmesh)], np.int32)
    truth = oracle.join(A, B, every, tier=2).astype(bool)
    rng = np.random.default_rng(n)
    pick = rng.integers(0, len(every), size=n)
    ha, hb = ctx.load(A), ctx.load(B)
    ctx.build(ha, 4, 2)
    ctx.build(hb, 4, 2)
    for at, bad in ((0, (A.nmesh, 0)), (n - 1, (0, B.nmesh)), (n // 2, (-1, 0)), (n // 3, (0, -1))):
        cand = every[pick]
        cand[at] = bad
        k, _, flags = _noalloc(ctx, ha, hb, cand, torch)
        want = truth[pick].copy()
        want[at] = False
        assert k == -1 and np.array_equal(flags.astype(bool), want)
    d_cand = torch.from_numpy(every[pick]).cuda()
    d_flags = torch.zeros(n, dtype=torch.uint8, device="cuda")
    d_pairs = torch.zeros((n, 2), dtype=torch.int32, device="cuda")
    d_count = torch.zeros(1, dtype=torch.int64, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        pierce.pj_join_intersects_noalloc(ctx.h, ha, hb, d_cand, d_flags, d_pairs, d_count,
                                          stream=torch.cuda.current_stream())
    for _ in range(3):
        pick = rng.integers(0, len(every), size=n)
        d_cand.copy_(torch.from_numpy(every[pick]))
        g.replay()
        torch.cuda.synchronize()
        t = truth[pick]
        assert int(d_count.item()) == t.sum()
        assert np.array_equal(d_flags.cpu().numpy().astype(bool), t)
        assert np.array_equal(d_pairs[:int(t.sum())].cpu().numpy(), every[pick][t])
    pierce.pj_free_dataset(ctx.h, ha)
    pierce.pj_free_dataset(ctx.h, hb)


def test_noalloc_join_of_the_full_tissue(ctx, pathology_truth):
    # more tasks change hands than a queue of 131,072 entries took, and all of
    # them fit
    torch = pytest.importorskip("torch")
    A, B, cand, truth = pathology_truth
    truth = truth.astype(bool)
    ha, hb = ctx.load(A), ctx.load(B)
    ctx.build(ha, 2, 2)
    ctx.build(hb, 2, 2)
    for _ in range(2):
        ctx.reset_counters()
        k, pairs, flags = _noalloc(ctx, ha, hb, cand, torch)
        assert np.array_equal(flags.astype(bool), truth)
        assert k == int(truth.sum()) and np.array_equal(pairs, cand[truth])
        c = ctx.counters()
        assert c["pairs_refined"] == len(cand)            # nothing was redone
        assert 131072 < c["tasks_spilled"] < 1 << 20
    pierce.pj_free_dataset(ctx.h, ha)
    pierce.pj_free_dataset(ctx.h, hb)


@pytest.mark.parametrize("W,L", [(2, 1), (4, 2), (8, 8)])
@pytest.mark.parametrize("predicate", ["intersects", "overlap"])
def test_dataset_join_leaves_the_walk(ctx, W, L, predicate):
    # from limits that the first level passes to one nothing passes: either the
    # packets do it (their launches besides) or the walk, with the same counts
    A, B = synth.tiny_spheres(1002)
    cand = oracle.mbb_candidates(A, B)
    want = cand[oracle.join(A, B, cand, predicate=predicate).astype(bool)]
    ha, hb = ctx.load(A), ctx.load(B)

    def call(mat, limit):
        pierce.pj_set_test_limits(ctx.h, dataset_walk=limit)
        before = ctx.counters()["kernel_launches"]
        got, st = pierce.pj_dataset_join(ctx.h, ha, hb, width=W, leaf_size=L,
                                         predicate=predicate, materialize=mat, fixed_slots=4096)
        assert np.array_equal(got, want)
        return ctx.counters()["kernel_launches"] - before, st

    for mat in ("estimated", "two_pass", "fixed"):
        call(mat, 0)
        n, st = call(mat, 0)
        left = []
        for limit in (1, 33, 64, 500, 3000, 20000, 1 << 20):
            m, s2 = call(mat, limit)
            left.append(m > n)
            assert m == n + left[-1] * (2 if predicate == "intersects" else 1)
            assert s2["hits"] == st["hits"] and s2["recheck_pairs"] == st["recheck_pairs"]
        assert left[0] and not left[-1] and left == sorted(left, reverse=True)
    pierce.pj_set_test_limits(ctx.h)
    pierce.pj_free_dataset(ctx.h, ha)
    pierce.pj_free_dataset(ctx.h, hb)


@pytest.mark.parametrize("grid", [1, 2, 3])
def test_tiled_join_gathered_by_the_host(ctx, grid):
    A, B = synth.tiny_spheres(1003)
    U = synth.urban(5001, n_buildings=400, n_parts=40)
    want, want_u = oracle.join_all(A, B), oracle.join_all(U, U, self_join=True)
    cut = synth.MeshSet(A.xyz, A.tris, A.voff[3:], A.toff[3:])
    for host in (1, 0):
        pierce.pj_set_test_limits(ctx.h, tiled_host_gather=host)
        got, st = pierce.pj_join_tiled(ctx.h, A, B, grid=grid)
        assert np.array_equal(got, want) and st["grid"] == grid
        got, _ = pierce.pj_join_tiled(ctx.h, U, self_join=True, grid=grid)
        assert np.array_equal(got, want_u)
        got, _ = pierce.pj_join_tiled(ctx.h, cut, B, grid=grid)
        assert np.array_equal(got, want[want[:, 0] >= 3] - [3, 0])
        if host:
            assert st["ms_gather"] > 0    # it was the host
    bad = synth.MeshSet(A.xyz.copy(), A.tris, A.voff, A.toff)
    bad.xyz[5, 1] += 0.5
    for host in (1, 0):
        pierce.pj_set_test_limits(ctx.h, tiled_host_gather=host)
        with pytest.raises(pierce.PierceError) as e:
            pierce.pj_join_tiled(ctx.h, bad, B, grid=grid)
        assert e.value.code == 2          # PJ_ERR_NOT_QUANTIZED
    pierce.pj_set_test_limits(ctx.h)


def test_tiled_budget_counts_memory_the_context_keeps():
    # with almost no free memory left a tiled join still has what the context
    # keeps of a freed dataset, and need not split its space
    V = synth.urban(5001, n_buildings=400, n_parts=40)
    U = synth.urban(5002, n_buildings=3000, n_parts=300)
    want = oracle.join_all(V, V, self_join=True)
    with pierce.Context(0) as c:
        pierce.pj_set_test_limits(c.h, tiled_free=4096)
        got, st = pierce.pj_join_tiled(c.h, V, self_join=True)
        assert np.array_equal(got, want) and st["grid"] > 1
        h = c.load(U)
        c.build(h, 4, 2)
        pierce.pj_free_dataset(c.h, h)
        got, st = pierce.pj_join_tiled(c.h, V, self_join=True)
        assert np.array_equal(got, want) and st["grid"] == 1
        with pytest.raises(pierce.PierceError) as e:          # a given budget is kept
            pierce.pj_join_tiled(c.h, V, self_join=True, device_budget=4096)
        assert e.value.code == 4                              # PJ_ERR_NO_MEMORY


def test_limits_refuse_no_context():
    assert pierce.load().pj_set_test_limits(None, ctypes.byref(pierce.pj_test_limits())) == 1
