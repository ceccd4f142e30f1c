"""The bounding-box filter join by sort and sweep (Sec. 3.1, the filter step),
taken when the all-pairs count passes 2^24: the device candidate list must be
the oracle's, in the oracle's order (checked through the per-candidate flags,
which line up with the device list), and the refined pair set the oracle's,
for a self join and for a join of two different datasets."""
import numpy as np
import pytest

import oracle
from conftest import oracle_flags
from paper_2609_24513_gb300 import pierce, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = pierce.Context(0)
    yield c
    c.close()


def _check(ctx, name, A, B, self_join):
    ma, mb = A.nmesh, B.nmesh
    assert (ma * (ma - 1) // 2 if self_join else ma * mb) > (1 << 24)  # the sweep path
    cand = oracle.mbb_candidates(A, B, self_join=self_join)
    flags = oracle_flags(name, A, B, cand)
    ha = ctx.load(A)
    hb = ha if self_join else ctx.load(B)
    ctx.build(ha, 4, 2)
    if not self_join:
        ctx.build(hb, 4, 2)
    res = pierce.pj_join_intersects_ex(ctx.h, ha, hb, self_join=self_join, width=4, leaf_size=2,
                                       out_host=True, keep_flags=True)
    n = int(res.n_candidates)
    got_flags = pierce.device_to_numpy(res.flags, n, np.uint8)
    got = pierce.pairs_to_numpy(res)
    pierce.pj_free_pairs(ctx.h, res)
    assert n == len(cand)
    assert np.array_equal(got_flags, flags)     # the same list, in the same order
    assert np.array_equal(got, cand[flags.astype(bool)])
    again, info = ctx.join(ha, hb, self_join=self_join, use_graph=True)
    assert info["n_candidates"] == len(cand) and np.array_equal(again, got)
    return len(cand), len(got)


def test_self_join(ctx):
    U = synth.urban(5003, n_buildings=5600, n_parts=600)
    c, k = _check(ctx, "urban self join 6,200 meshes", U, U, True)
    assert c > 1000 and k > 100


def test_two_datasets(ctx):
    A = synth.urban(5004, n_buildings=3900, n_parts=400)
    B = synth.urban(5005, n_buildings=3900, n_parts=400)
    c, k = _check(ctx, "urban x urban 4,300 x 4,300 meshes", A, B, False)
    assert c > 1000 and k > 100


def _boxes(rng, n, side, span=(262143, 262143, 262143)):
    lo = rng.integers(0, [max(1, s - d) for s, d in zip(span, side)], size=(n, 3))
    hi = lo + rng.integers(1, np.array(side) + 1, size=(n, 3))
    return [synth.box(tuple(a), tuple(np.minimum(b, 262143))) for a, b in zip(lo, hi)]


@pytest.mark.parametrize("kind", ["sparse", "dense", "long", "huge", "two_sided", "one_bucket"])
def test_sweep_over_box_shapes(ctx, kind):
    # sparse: a few pairs a box; dense: more pairs than the list first has
    # room for; long: ranges past the 16 steps of a box's own warp, thousands
    # of them; huge: meshes with more pairs than are ordered in place;
    # two_sided: few long boxes against many small ones; one_bucket: every
    # low x in one bucket of 16 grid units
    rng = np.random.default_rng(7)
    B = None
    if kind == "sparse":
        A = _boxes(rng, 5900, (6000, 6000, 6000))
    elif kind == "dense":
        A = _boxes(rng, 5900, (30000, 60000, 60000))
    elif kind == "long":
        A = _boxes(rng, 5900, (200000, 2000, 2000))
    elif kind == "huge":
        A = [synth.box((k, 2 * k, 0), (262143 - k, 262143, 262143)) for k in range(1, 4)] + \
            _boxes(rng, 5900, (3000, 3000, 3000))
    elif kind == "two_sided":
        A = _boxes(rng, 210, (90000, 5000, 5000))
        B = _boxes(rng, 81000, (900, 900, 900))
    else:
        A = _boxes(rng, 5900, (9, 9000, 9000), (20, 262143, 262143))
    A = synth.concat(A)
    B = synth.concat(B) if B else None
    c, k = _check(ctx, "sweep " + kind, A, B if B is not None else A, B is None)
    assert c > 200 and k > 50
    if kind == "dense":
        assert c > 4 * 5900


def test_sweep_graph_beside_a_host_list_graph(ctx):
    # a sweep join and a join over a host list of the same length use the same
    # buffers, but only the latter's flags are cleared before its graph runs:
    # the sweep must not replay the list's graph over another join's flags
    U = synth.urban(5003, n_buildings=5600, n_parts=600)
    h = ctx.load(U)
    ctx.build(h, 4, 2)
    want, info = ctx.join(h, h, self_join=True)
    n = info["n_candidates"]
    cand = oracle.mbb_candidates(U, U, self_join=True)
    assert n == len(cand) and 100 < len(want) < n
    flags = oracle_flags("sweep beside a list", U, U, cand).astype(bool)
    assert np.array_equal(want, cand[flags])
    order = np.random.default_rng(11).permutation(n)
    for _ in range(2):                                    # captured, then replayed
        got, _ = ctx.join(h, h, cand=cand[order], use_graph=True)
        assert np.array_equal(got, cand[order][flags[order]])
    # every flag set by an unrelated join of the same length
    ctx.join(h, h, cand=want[np.arange(n) % len(want)])
    for _ in range(2):
        got, _ = ctx.join(h, h, self_join=True, use_graph=True)
        assert np.array_equal(got, want)
    got, _ = ctx.join(h, h, cand=cand[order], use_graph=True)
    assert np.array_equal(got, cand[order][flags[order]])
