"""The dataset-level join (pj_dataset_join: one BVH per dataset, every owned
edge traced both ways with all of its crossings, one parity ray per object,
pairs deduplicated by a hashmap sized by the estimate, by counting two-pass
or by a fixed hashmap; paper Sec. 3.1-3.5) against the oracle, for the
intersects and overlap predicates: tiny spheres at three BVH shapes,
hand-built solids in both roles, exhaustive lattice placements (many parity
vertices on the other surface: the per-pair recheck), a self join of urban
buildings and the full pathology workload.  Pair sets compared exactly."""
import numpy as np
import pytest

import oracle
from cases import HAND, lattice_case_sets
from paper_2609_24513_gb300 import pierce, synth

pytestmark = pytest.mark.gpu

MATS = ("estimated", "two_pass", "fixed")


@pytest.fixture(scope="module")
def ctx():
    c = pierce.Context(0)
    yield c
    c.close()


def _truth(A, B, pred, self_join=False):
    cand = oracle.mbb_candidates(A, B, self_join)
    return cand[oracle.join(A, B, cand, predicate=pred, threads=None).astype(bool)]


@pytest.mark.parametrize("W,L", [(4, 2), (8, 4), (2, 1)])
def test_tiny_spheres(ctx, W, L):
    for seed in (1001, 1002, 1003):
        A, B = synth.tiny_spheres(seed)
        ha, hb = ctx.load(A), ctx.load(B)
        for pred in ("intersects", "overlap"):
            want = _truth(A, B, pred)
            for mat in MATS:
                got, st = pierce.pj_dataset_join(ctx.h, ha, hb, width=W, leaf_size=L,
                                                 predicate=pred, materialize=mat)
                assert np.array_equal(got, want), (seed, pred, mat)
                assert st["hits"] >= 0 and st["edges"] > 0


def test_hand_built_both_roles(ctx):
    for name, (ma, mb, _) in sorted(HAND.items()):
        for X, Y in ((ma, mb), (mb, ma)):
            A, B = synth.concat([X]), synth.concat([Y])
            ha, hb = ctx.load(A), ctx.load(B)
            for pred in ("intersects", "overlap"):
                want = _truth(A, B, pred)
                for mat in MATS:
                    got, _ = pierce.pj_dataset_join(ctx.h, ha, hb, predicate=pred, materialize=mat)
                    assert np.array_equal(got, want), (name, pred, mat)
            pierce.pj_free_dataset(ctx.h, ha)
            pierce.pj_free_dataset(ctx.h, hb)


def test_lattice_placements_recheck(ctx):
    A, B, cand, _ = lattice_case_sets()
    ha, hb = ctx.load(A), ctx.load(B)
    want = _truth(A, B, "intersects")
    for mat in MATS:
        got, st = pierce.pj_dataset_join(ctx.h, ha, hb, materialize=mat)
        assert np.array_equal(got, want), mat
    assert st["recheck_pairs"] > 0          # vertices on the other surface were rechecked


def test_urban_self_join(ctx):
    U = synth.urban(5001, n_buildings=2000, n_parts=200)
    h = ctx.load(U)
    want = _truth(U, U, "intersects", self_join=True)
    for mat in MATS:
        got, _ = pierce.pj_dataset_join(ctx.h, h, h, self_join=True, materialize=mat)
        assert np.array_equal(got, want), mat
        assert np.all(got[:, 0] < got[:, 1])


def test_overflowing_fixed_hashmap_relaunches(ctx):
    A, B = synth.tiny_spheres(1002)
    ha, hb = ctx.load(A), ctx.load(B)
    want = _truth(A, B, "intersects")
    got, st = pierce.pj_dataset_join(ctx.h, ha, hb, materialize="fixed", fixed_slots=16)
    assert np.array_equal(got, want)
    assert st["relaunches"] > 0 and st["slots"] > 16


def test_pathology_full(ctx, pathology_truth):
    A, B, cand, flags = pathology_truth
    want = cand[flags.astype(bool)]
    ha, hb = ctx.load(A), ctx.load(B)
    for mat in MATS:
        got, st = pierce.pj_dataset_join(ctx.h, ha, hb, materialize=mat)
        assert np.array_equal(got, want), mat
        print("dataset join %s: %d pairs, %.2f ms (trace %.2f, materialise %.2f), %d edges, "
              "%d crossings, %d slots, %d relaunches, %d rechecked"
              % (mat, len(got), st["ms_total"], st["ms_trace"], st["ms_materialize"],
                 st["edges"], st["hits"], st["slots"], st["relaunches"], st["recheck_pairs"]))


@pytest.mark.parametrize("sides,bands", [(6, 0), (5, 2), (8, 1), (17, 1), (3, 10), (64, 19)])
@pytest.mark.parametrize("W,L", [(2, 8), (4, 1), (8, 2)])
def test_packet_sizes(ctx, sides, bands, W, L):
    # 12, 30, 32, 68, 66 and 2,560 triangles a mesh: around the 32 of a warp's
    # packet; five meshes, so that packets hold the ends of several; the last
    # one's triangles are far larger than the others' whole meshes
    th = 2 * np.pi * np.arange(sides) / sides

    def prism(x, y, z, r):
        foot = np.rint(np.stack([r * np.cos(th) + x, r * np.sin(th) + y], 1))
        return synth.building(foot, z, 9000, 1500, max(1, bands)) if bands else \
            synth.box((x - r, y - r, z), (x + r, y + r, z + 9000))

    A = synth.concat([prism(50000 + 6000 * k, 50000, 20000, 4000 + 100 * k) for k in range(5)])
    B = synth.concat([prism(52000 + 7000 * k, 51000 + 900 * k, 21000, 3000) for k in range(4)] +
                     [synth.box((0, 0, 0), (262143, 262143, 262143))])
    ha, hb = ctx.load(A), ctx.load(B)
    for pred in ("intersects", "overlap"):
        want = _truth(A, B, pred)
        assert len(want) > 0
        hits = set()
        for mat in MATS:
            got, st = pierce.pj_dataset_join(ctx.h, ha, hb, width=W, leaf_size=L, predicate=pred,
                                             materialize=mat)
            assert np.array_equal(got, want), (pred, mat)
            hits.add(st["hits"])
        assert len(hits) == 1


def test_dense_datasets_leave_the_walk(ctx):
    # 16 x 16 mutually crossing spheres of 20,480 triangles: far more
    # overlapping leaf pairs (at least 9.5 M) than the joint walk's
    # list holds, so that the packets trace the edges; against the per-pair
    # join, which other tests hold to the oracle
    V, F = synth.icosphere(5)
    rng = np.random.default_rng(3)
    R = synth.random_rotations(rng, 32)
    ball = [(synth.quantize(0.5 + (V @ R[k].T) * (0.2 + 1e-6 * k)), F) for k in range(32)]
    A, B = synth.concat(ball[:16]), synth.concat(ball[16:])
    ha, hb = ctx.load(A), ctx.load(B)
    ctx.build(ha, 4, 2)
    ctx.build(hb, 4, 2)
    for pred in ("intersects", "overlap"):
        want, _ = ctx.join(ha, hb, predicate=pred)
        assert len(want) > 100
        for mat in MATS:
            got, st = pierce.pj_dataset_join(ctx.h, ha, hb, predicate=pred, materialize=mat)
            assert np.array_equal(got, want), (pred, mat)
            assert st["hits"] > 50_000
            assert st["edges"] == 3 * (len(A.tris) + len(B.tris)) // 2
    pierce.pj_free_dataset(ctx.h, ha)
    pierce.pj_free_dataset(ctx.h, hb)
