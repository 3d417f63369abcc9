"""Crowded lattices (9 pedestrians on 20 su and more), whose field the
tensor-core product sums: against the FP64 oracle at the edges of its tiles,
radii and alignments, closed and periodic; closer to it than the gather; and
bit for bit the same in bands, in a batch and at the candidates only."""
import time

import numpy as np
import pytest

import paper_1803_04782_gb300 as sfm
import scenegen as SG
from paper_1803_04782_gb300 import build as B
from parity import OracleRun, assert_field

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()
    sfm.lib()


def _crowd(W, H, r, px=1, py=1, rho=0.5, seed=0, **kw):
    free = (W - (0 if px else 2)) * (H - (0 if py else 2))
    return SG.random_scene(W, H, int(rho * free), r=r, seed=300 + seed + r, periodic_x=px, periodic_y=py,
                           ring=not (px and py), exits=() if (px and py) else ("east",),
                           goal_mode="fixed" if (px and py) else "mixed", heading_mode="random", **kw)


@pytest.mark.parametrize("W,H,r,px,py", [(64, 256, 3, 1, 1), (65, 257, 3, 0, 0), (127, 255, 9, 1, 0),
                                         (130, 300, 20, 0, 1), (7, 300, 3, 1, 0), (89, 89, 44, 1, 1),
                                         (200, 130, 38, 0, 0), (33, 40, 1, 1, 1)])
def test_product_field_against_the_oracle_and_the_gather(W, H, r, px, py):
    sc = _crowd(W, H, r, px, py, rho=0.6)
    assert 20 * sc.n >= 9 * W * H
    orc = OracleRun(sc)
    Fo, So = orc.field()
    with sfm.Sim(sc) as a, sfm.Sim(sc) as b:
        b.set_field_rule("gather")
        for s in (a, b):
            s.compute_field()
        Fa, Fb = a.field(), b.field()
        assert_field(Fa, Fo, So)
        # the product's sums are exact (its entries are off by 2^-24 of the
        # law's largest, its result by one rounding): no further off than FP32 sums
        err = [np.linalg.norm(F - Fo) / np.linalg.norm(Fo) for F in (Fa, Fb)]
        assert err[0] <= max(err[1], 6e-8) and not np.array_equal(Fa, Fb)
        a.compute_field()
        np.testing.assert_array_equal(a.field(), Fa)  # the split tiles' sums are zero again
        # the rule holds for any crowd when it is asked for
        b.set_field_rule("product")
        b.place(sc.xy[:40], sc.heading[:40], sc.goal[:40])
        b.compute_field()
        assert_field(b.field(), *_field_of(sc, 40))
        with pytest.raises(sfm.SfmError) as e:
            sfm._check(a.ctx, sfm.lib().sfm_set_field_rule(a.ctx, 3))
        assert e.value.status == sfm.SFM_EINVAL


def _field_of(sc, n):
    part = sc.copy()
    part.xy, part.heading, part.goal = sc.xy[:n].copy(), sc.heading[:n].copy(), sc.goal[:n].copy()
    return OracleRun(part).field()


@pytest.mark.parametrize("px,py,r,rows", [(0, 0, 36, 64), (1, 1, 36, 96), (1, 0, 5, 32)])
def test_bands_batch_and_candidates_round_as_one_launch(px, py, r, rows):
    sc = _crowd(150, 256, r, px, py, rho=0.55, seed=7)
    budget = sfm.band_budget(sc.W, sc.H, rows, px, py)
    init = np.zeros(int(sfm.lib().sfm_surrogate_nparams()), np.float32)
    even = _crowd(144, 256, r, px, py, rho=0.55, seed=8)  # the candidates want a multiple of their cells
    with sfm.Sim(sc) as a, sfm.Sim(sc, hbm_budget_bytes=budget) as b, sfm.Batch([sc, even]) as c, \
            sfm.Sim(even) as d, sfm.Sim(even) as e, sfm.Surrogate(coarsen=4, params=init) as sur:
        assert b.stats()["bands"] > 1
        if r == 36:
            b.set_footprint("32x32r")  # with closed y: the ring of rows
        a.compute_field()
        np.testing.assert_array_equal(a.field(), b.field_banded())
        c.compute_field()
        np.testing.assert_array_equal(a.field(), c.fields()[0])
        for _ in range(4):
            for s in (a, b, c, d):
                s.step(1)
            sur.step(e, 1)
            for x, y, z in zip(a.peds(), b.peds(), c.peds()):
                np.testing.assert_array_equal(x, y)
                np.testing.assert_array_equal(x, z[0])
            for x, y, z in zip(d.peds(), e.peds(), c.peds()):
                np.testing.assert_array_equal(x, y)
                np.testing.assert_array_equal(x, z[1])
            np.testing.assert_array_equal(d.decisions()[0], e.decisions()[0])
        for s in (a, b, c, d, e):
            assert s.stats()["error_flags"] == 0


@pytest.mark.parametrize("W,H,r,product", [(20, 20, 38, False), (12, 16, 20, False), (300, 4, 20, False),
                                           (40, 40, 44, True), (64, 64, 38, True), (41, 45, 20, True)])
def test_lattices_smaller_than_the_window_take_the_faster_way(W, H, r, product):
    sc = _crowd(W, H, r, 0, 0, rho=0.95, seed=13)
    assert 20 * sc.n >= 9 * W * H
    assert sfm.sfm_crowded(sfm.Lattice(W, H, 0, 0), r, sc.n) == product
    fields = []
    with sfm.Sim(sc) as s, sfm.Batch([sc]) as b:
        for rule in ("auto", "gather", "product"):
            s.set_field_rule(rule)
            s.compute_field()
            fields.append(s.field())
        b.compute_field()
        np.testing.assert_array_equal(b.fields()[0], fields[0])
    np.testing.assert_array_equal(fields[0], fields[2 if product else 1])
    assert not np.array_equal(fields[1], fields[2])


@pytest.mark.parametrize("r,law", [(12, {}), (25, {}), (40, {}), (44, {}), (30, dict(aO=-1.0, aE=-0.7)),
                                   (16, dict(kO=3.7e4, aO=-0.25, kE=0.0))])
def test_a_wall_far_away_is_as_exact_as_fp32(r, law):
    """One WALL and one EXIT su, in reach of different su: an entry rounded to
    FP32 (2^-24 of itself) and the rounding of the sum."""
    W = H = 4 * r + 9
    cell = np.zeros((H, W), np.uint8)
    at = {1: (r + 2, r + 1), 2: (W - r - 3, H - r - 2)}  # (x, y)
    for kind, (x, y) in at.items():
        cell[y, x] = kind
    p = dict(kO=1.0, aO=-0.5, kE=-1.0, aE=-0.5)
    p.update(law)
    want, terms = np.zeros((H, W)), np.zeros((H, W))
    yy, xx = np.mgrid[:H, :W]
    for kind, (x, y) in at.items():
        dx, dy = xx - x, yy - y
        near = (np.maximum(abs(dx), abs(dy)) <= r) & ((dx != 0) | (dy != 0))
        k, a = (np.float32(p["kO"]), np.float32(p["aO"])) if kind == 1 else (np.float32(p["kE"]), np.float32(p["aE"]))
        d = np.hypot(dx, dy)
        d[y, x] = 1.0
        v = np.where(near, float(k) * d ** float(a), 0.0)
        want += v
        terms += abs(v)
    with sfm.Sim(W=W, H=H, cell=cell, r=r, **p) as s:
        got = s.static_field().astype(np.float64)
    assert (np.abs(got - want) <= 2.0 ** -24 * (terms + np.abs(want)) * 1.0001).all()


@pytest.mark.parametrize("r,law", [(3, {}), (12, {}), (40, {}), (44, {}), (20, dict(aP=-1.0)), (40, dict(aP=-1.0))])
def test_a_pedestrian_far_away_keeps_its_digits(r, law):
    """One pedestrian by the product, or by the gather where the law is refused."""
    aP = np.float64(law.get("aP", -0.5))
    S = 2 * r + 3
    yy, xx = np.mgrid[:S, :S]
    dx, dy = xx - r - 1.0, yy - r - 1.0
    d = np.hypot(dx, dy)
    d[r + 1, r + 1] = 1.0
    with sfm.Sim(W=S, H=S, cell=np.zeros((S, S), np.uint8), r=r, **law) as s:
        s.set_field_rule("product")
        for h, (ux, uy) in enumerate([(0, 0), (1, 0), (1, 1), (0, 1), (-1, 1), (-1, 0), (-1, -1), (0, -1), (1, -1)]):
            s.place(np.array([[r + 1, r + 1]], np.int32), np.array([h], np.uint8))
            s.compute_field()
            u = max(1.0, np.hypot(ux, uy))
            base = np.where(np.maximum(abs(dx), abs(dy)) <= r, d ** aP, 0.0)
            base[r + 1, r + 1] = 0.0
            want = base * (1 + 0.5 * (ux * dx + uy * dy) / (u * d))
            off = np.abs(s.field() - want)
            assert (off <= (2.2e-7 if r <= 40 and not law else 2.0 ** -21) * base + 2.0 ** -24 * np.abs(want) * 1.001).all()


def test_autotuning_a_crowded_lattice_keeps_its_footprint():
    sc = _crowd(150, 256, 20, 1, 1, rho=0.55, seed=12)
    with sfm.Sim(sc) as s:
        for shape in sfm.FOOTPRINTS * 3:
            s.set_footprint(shape)
            assert s.autotune() == shape
    few = sc.copy()
    few.xy, few.heading, few.goal = (a[:sc.n // 10].copy() for a in (sc.xy, sc.heading, sc.goal))
    with sfm.Batch([few]) as b:
        was = b.autotune()
        b.place([sc.xy], [sc.heading], [sc.goal])
        for _ in range(8):
            assert b.autotune() == was
        with sfm.Sim(sc) as s:
            for x in (s, b):
                x.step(2)
            np.testing.assert_array_equal(s.peds()[0], b.peds()[0][0])


@pytest.mark.parametrize("n,sized,rows", [(900, False, 0), (0, False, 0), (0, False, 64), (0, True, 0)])
def test_nobody_moves_on_a_field_whose_wait_ran_out(n, sized, rows):
    """n: a crowd small enough for the stages in one block; rows: of a band."""
    sc = _crowd(40 if n else 96, 40 if n else 256, 12, 0, 0, rho=0.7, seed=11)
    n = n or sc.n
    assert 20 * n >= 9 * sc.W * sc.H
    xy, heading, goal = sc.xy[:n], sc.heading[:n], sc.goal[:n]
    kw = dict(hbm_budget_bytes=sfm.band_budget(sc.W, sc.H, rows, 0, 0)) if rows else {}
    sim = sfm.Sim(W=sc.W, H=sc.H, cell=sc.cell, r=12, **kw)
    ones = np.ones(n, np.uint8)

    def place():
        if sized:
            sim.place_sized(xy, heading, goal, ones, ones, ones)
        else:
            sim.place(xy, heading, goal)
    with sim, sfm.Sim(W=sc.W, H=sc.H, cell=sc.cell, r=12) as ref:
        place()
        sfm.sfm_test_wait_out(sim.ctx, 0)
        t0 = time.time()
        sim.step(3)
        with pytest.raises(sfm.SfmError) as e:
            sim.sync()
        assert e.value.status == sfm.SFM_ETIMEOUT and time.time() - t0 < 30
        st = sim.stats()
        assert (st["moved_total"], st["exited"], st["t"]) == (0, 0, 0)
        where = np.zeros((n, 2), np.int32), np.zeros(n, np.uint8), np.zeros(n, np.uint8)
        assert sfm.lib().sfm_read_peds(sim.ctx, *(a.ctypes.data for a in where), 0) == sfm.SFM_ETIMEOUT
        for got, want in zip(where, (xy, heading, ones)):
            np.testing.assert_array_equal(got, want)
        # placed anew it goes on, the split tiles' sums and all
        place()
        ref.place(xy, heading, goal)
        for s in (sim, ref):
            s.set_time(0)
            s.step(3)
            s.sync()
        for got, want in zip(sim.peds(), ref.peds()):
            np.testing.assert_array_equal(got, want)
        assert ref.stats()["moved_total"] > 0


def test_two_row_bands_round_as_the_whole_lattice():
    """The stepper of a row-band decomposition sums its field as the whole
    lattice does, whatever its own rows hold."""
    from paper_1803_04782_gb300 import bands as BD
    sc = _crowd(96, 320, 12, 1, 0, rho=0.5, seed=9)
    sc.xy = sc.xy[np.argsort(sc.xy[:, 1], kind="stable")]  # then thin the upper half out
    keep = np.flatnonzero((sc.xy[:, 1] < 160) | (np.arange(sc.n) % 10 != 0))
    sc.xy, sc.heading, sc.goal = sc.xy[keep], sc.heading[keep], sc.goal[keep]
    assert 20 * sc.n >= 9 * sc.W * sc.H
    L = BD.BandLayout(sc.H, 0, 12, 2)
    peds = BD.Peds(np.arange(sc.n, dtype=np.int32), sc.xy, sc.heading, sc.goal)
    with sfm.Sim(sc) as whole:
        D = whole.guidance()
        owned = [BD.own_of(L, k, peds) for k in range(2)]
        steps = [BD.sim_stepper(L, k, sc.W, 1, sc.cell, D, sc.params) for k in range(2)]
        for t in range(3):
            sends = [BD.sends_of(L, k, owned[k]) for k in range(2)]

            class Comm:
                def __init__(self, k):
                    self.k = k

                def exchange(self, mine):
                    return {j: sends[j][self.k].pack() for j in mine}
            owned = [BD.band_tick(L, k, Comm(k), steps[k][0], owned[k], t)[0] for k in range(2)]
        whole.step(3)
        xy, hd, al = whole.peds()
        for _, sim in steps:
            sim.close()
    ids = np.concatenate([o.ids for o in owned])
    order = np.argsort(ids)
    live = np.flatnonzero(al)
    np.testing.assert_array_equal(ids[order], live)
    np.testing.assert_array_equal(np.concatenate([o.xy for o in owned])[order], xy[live])
    np.testing.assert_array_equal(np.concatenate([o.heading for o in owned])[order], hd[live])


def test_the_rule_of_row_bands_is_the_whole_lattices_throughout():
    """Bands resumed from per-rank sets (no own_of), with the whole lattice's
    crowd given; and a look at a part of the crowd changes no stepper's rule."""
    from paper_1803_04782_gb300 import bands as BD
    sc = _crowd(96, 320, 12, 1, 0, rho=0.5, seed=10)
    assert 20 * sc.n >= 9 * sc.W * sc.H
    peds = BD.Peds(np.arange(sc.n, dtype=np.int32), sc.xy, sc.heading, sc.goal)
    with sfm.Sim(sc) as whole:
        D = whole.guidance()
        whole.compute_field()
        F = whole.field()
        whole.step(2)
        xy, hd, al = whole.peds()
    for given in (True, False):
        L = BD.BandLayout(sc.H, 0, 12, 2)
        who = L.owner(peds.xy[:, 1])
        owned = [peds.take(who == k) for k in range(2)]
        if not given:
            owned = [BD.own_of(L, k, peds) for k in range(2)]
        steps = [BD.sim_stepper(L, k, sc.W, 1, sc.cell, D, sc.params, crowd=sc.n if given else None)
                 for k in range(2)]
        try:
            for t in range(2):
                BD.own_of(L, 0, owned[0].take(np.arange(owned[0].n) < 10))
                sends = [BD.sends_of(L, k, owned[k]) for k in range(2)]

                class Comm:
                    def __init__(self, k):
                        self.k = k

                    def exchange(self, mine):
                        return {j: sends[j][self.k].pack() for j in mine}
                owned = [BD.band_tick(L, k, Comm(k), steps[k][0], owned[k], t)[0] for k in range(2)]
                for k in range(2 if t == 0 else 0):  # the product's bits, not the gather's
                    y = np.arange(L.y0[k], L.y1[k])
                    np.testing.assert_array_equal(steps[k][1].field()[L.local_row(k, y)], F[y])
        finally:
            for _, sim in steps:
                sim.close()
        ids = np.concatenate([o.ids for o in owned])
        order, live = np.argsort(ids), np.flatnonzero(al)
        np.testing.assert_array_equal(ids[order], live)
        np.testing.assert_array_equal(np.concatenate([o.xy for o in owned])[order], xy[live])
