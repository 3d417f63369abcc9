"""Batched lattices on the GPU: one persistent launch per tick for every
lattice must reproduce, bit for bit, what each lattice does in its own
context (itself checked against the oracle), before and after the footprint
autotuner; the bounded grid barrier must give up cleanly."""
import time

import numpy as np
import pytest

import oracle as O
import paper_1803_04782_gb300 as sfm
import scenegen as SG
from paper_1803_04782_gb300 import build as B
from parity import OracleRun, assert_field, compare_choices

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()
    sfm.lib()


def _mixed_batch():
    """Ten lattices of uneven size, crowd and radius (every class-table row
    stride: 34, 50, ..., 114 and the narrow 102), closed, periodic and torus
    boundaries."""
    sc = [
        SG.random_scene(64, 64, 300, r=5, seed=201, exits=("east",)),
        SG.random_scene(150, 97, 1500, r=12, seed=202, obstacles=3, exits=("north", "west"),
                        goal_mode="mixed", heading_mode="random"),
        SG.random_scene(90, 60, 900, r=9, seed=203, periodic_x=1, exits=("south",),
                        goal_mode="fixed", heading_mode="goal"),
        SG.random_scene(70, 70, 1200, r=20, seed=204, periodic_x=1, periodic_y=1, ring=False,
                        exits=(), goal_mode="fixed", heading_mode="random"),
        SG.random_scene(200, 130, 2500, r=28, seed=205, obstacles=5, exits=("east",),
                        goal_mode="mixed", heading_mode="random"),
        SG.random_scene(33, 41, 200, r=0, seed=206, exits=("west",)),
        SG.random_scene(260, 180, 3000, r=36, seed=207, exits=("north",), heading_mode="random"),
        SG.random_scene(120, 230, 2000, r=47, seed=208, periodic_y=1, exits=("east",),
                        goal_mode="mixed", heading_mode="random"),
        SG.random_scene(40, 40, 38 * 38 - 3, r=3, seed=209, exits=("east", "west"), exit_len=6),
        SG.random_scene(11, 60, 100, r=5, seed=210, periodic_x=1, exits=("south",),
                        goal_mode="mixed", heading_mode="random"),
    ]
    for i, s in enumerate(sc):
        s.params["seed"] = 1000 + i
    return sc


def _compare_with_single(scenes, batch, ticks):
    sims = [sfm.Sim(s) for s in scenes]
    try:
        batch.compute_field()
        for s in sims:
            s.compute_field()
        for F_b, s in zip(batch.fields(), sims):
            np.testing.assert_array_equal(F_b, s.field())
        for t in range(ticks):
            batch.step(1)
            for s in sims:
                s.step(1)
            ch_b, won_b = batch.decisions()
            xy_b, h_b, a_b = batch.peds()
            F_b = batch.fields()
            for i, s in enumerate(sims):
                ch, won = s.decisions()
                xy, h, a = s.peds()
                np.testing.assert_array_equal(F_b[i], s.field(), err_msg=f"lattice {i} tick {t}")
                np.testing.assert_array_equal(ch_b[i], ch, err_msg=f"lattice {i} tick {t}")
                np.testing.assert_array_equal(won_b[i], won)
                np.testing.assert_array_equal(xy_b[i], xy)
                np.testing.assert_array_equal(h_b[i], h)
                np.testing.assert_array_equal(a_b[i], a)
        st = batch.stats()
        assert st["error_flags"] == 0 and st["max_registrants"] <= 8
        assert st["exited"] == sum(s.stats()["exited"] for s in sims)
    finally:
        for s in sims:
            s.close()


def test_batch_matches_independent_contexts_bitwise():
    scenes = _mixed_batch()
    with sfm.Batch(scenes) as b:
        np.testing.assert_array_equal(
            np.concatenate([g.ravel() for g in b.guidance()]),
            np.concatenate([O.guidance(O.model(s), s.cell).ravel() for s in scenes]))
        _compare_with_single(scenes, b, ticks=4)


def test_batch_autotuned_tiles_give_the_same_ticks():
    scenes = _mixed_batch()
    with sfm.Batch(scenes) as b:
        shapes = b.autotune()
        assert set(shapes.values()) <= {"16x16", "32x16"}
        _compare_with_single(scenes, b, ticks=3)


def test_batch_lattices_match_the_oracle():
    scenes = _mixed_batch()
    picks = [1, 3, 7]
    with sfm.Batch(scenes) as b:
        orcs = [OracleRun(scenes[i]) for i in picks]
        for t in range(3):
            b.step(1)
            F = b.fields()
            ch_b, _ = b.decisions()
            xy_b, h_b, a_b = b.peds()
            for k, i in enumerate(picks):
                orc = orcs[k]
                Fo, So = orc.field()
                assert_field(F[i], Fo, So, f"lattice {i} tick {t}")
                ch_o, E, T, adm = orc.decide(Ffull=Fo.ravel(), Sfull=So.ravel())
                flips = compare_choices(ch_b[i], ch_o, E, T, adm)
                orc.advance(ch_o)
                if flips == 0:
                    np.testing.assert_array_equal(xy_b[i], orc.st.xy)
                    np.testing.assert_array_equal(a_b[i], orc.st.alive)
                else:
                    # the runs part ways at a tie: restart the batch lattice from
                    # the oracle's state is not possible per lattice, so stop here
                    return


def test_bounded_barrier_gives_up_and_context_recovers():
    scenes = _mixed_batch()[:4]
    with sfm.Batch(scenes) as b, sfm.Batch(scenes) as ref:
        sfm.sfm_batch_test_missing_ctas(b.ctx, 1)
        t0 = time.time()
        with pytest.raises(sfm.SfmError) as e:
            b.step(1)
        assert e.value.status == sfm.SFM_ETIMEOUT
        assert time.time() - t0 < 30
        # the timed-out tick stopped at its first barrier (bins only): nobody moved
        for x, y in zip(b.peds()[0], [s.xy for s in scenes]):
            np.testing.assert_array_equal(x, y)
        b.step(2)
        ref.step(2)
        for x, y in zip(b.peds()[0], ref.peds()[0]):
            np.testing.assert_array_equal(x, y)
        assert b.stats()["error_flags"] == 0


def test_batch_placement_errors():
    scenes = _mixed_batch()[:3]
    with sfm.Batch(scenes, place=False) as b:
        with pytest.raises(sfm.SfmError) as e:
            b.step(1)
        assert e.value.status == sfm.SFM_ESTATE
        xys = [s.xy.copy() for s in scenes]
        xys[1][0] = xys[1][1]
        with pytest.raises(sfm.SfmError) as e:
            b.place(xys)
        assert e.value.status == sfm.SFM_ECONFLICT
        b.place([s.xy for s in scenes], [s.heading for s in scenes], [s.goal for s in scenes])
        b.step(1)
        assert b.stats()["error_flags"] == 0


def test_sparse_and_dense_lattices_in_one_batch():
    """Decide, vote and commit go by pedestrian below a pedestrian on every tenth
    su of the batch, by bins from there on: batches of sparse and dense lattices
    on either side of the line, against single contexts."""
    def scene(W, H, n, seed, px):
        return SG.random_scene(W, H, n, r=4, seed=seed, periodic_x=px, periodic_y=px, ring=not px,
                               exits=() if px else ("east",), goal_mode="fixed" if px else "mixed",
                               heading_mode="random")
    sparse = [scene(90, 70, 629, 1, 1), scene(33, 65, 3, 2, 0), scene(300, 200, 900, 3, 0)]
    dense = [scene(90, 70, 630, 4, 1), scene(64, 64, 1200, 5, 0), scene(31, 37, 1147 // 2, 6, 1)]
    for scenes in (sparse, dense, sparse[:2] + dense + sparse[2:]):
        with sfm.Batch(scenes) as b:
            singles = [sfm.Sim(s) for s in scenes]
            try:
                for _ in range(2):
                    for x in singles + [b]:
                        x.step(3)
                    for got, want in zip(zip(*b.peds()), (s.peds() for s in singles)):
                        for x, y in zip(got, want):
                            np.testing.assert_array_equal(x, y)
                    for got, want in zip(zip(*b.decisions()), (s.decisions() for s in singles)):
                        for x, y in zip(got, want):
                            np.testing.assert_array_equal(x, y)
                st, of = b.stats(), [s.stats() for s in singles]
                assert st["t"] == 6 and st["error_flags"] == 0
                for key in ("moved_total", "exited"):
                    assert st[key] == sum(s[key] for s in of)
                assert st["max_registrants"] == max(s["max_registrants"] for s in of)
                # the same lattices with everybody but one gone, then nobody
                sfm.sfm_batch_place(b.ctx, [1] + [0] * (len(scenes) - 1), scenes[0].xy[:1].copy())
                b.step(2)
                sfm.sfm_batch_place(b.ctx, [0] * len(scenes), np.zeros((0, 2), np.int32))
                b.step(2)
                assert b.stats()["t"] == 10
            finally:
                for s in singles:
                    s.close()
