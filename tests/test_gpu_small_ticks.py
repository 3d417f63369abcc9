"""The short launch sequences of small lattices against the long ones: bins
from the class grid in one launch (64 bins), two (4096) or three and more, the
pedestrian list's bins, and decide, vote and commit in one block or three
launches; and those stages bin by bin against
pedestrian by pedestrian; and the gather of few footprints against the
others.  All leave the same bits."""
import numpy as np
import pytest

import paper_1803_04782_gb300 as sfm
import scenegen as SG
from paper_1803_04782_gb300 import build as B
from parity import OracleRun, compare_choices, rect_cells

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()
    sfm.lib()


def _sim(W, H, n, periodic, walk, r=5):
    rng = np.random.default_rng(W + H + n)
    cell = np.zeros((H, W), np.uint8)
    cell[:, W // 2] = 1
    cell[H // 3:H // 2, W // 2] = 0
    cell[0, W // 4:W // 2] = 2
    s = sfm.Sim(W=W, H=H, cell=cell, periodic_x=periodic, periodic_y=periodic, r=r)
    at = rng.choice(np.flatnonzero(cell.ravel() == 0), n, replace=False)
    s.place(np.stack([at % W, at // W], 1).astype(np.int32), rng.integers(0, 9, n).astype(np.uint8),
            rng.integers(0, 9, n).astype(np.uint8), (rng.random(n) < 0.9).astype(np.uint8))
    if walk:
        period = rng.integers(1, 4, n).astype(np.uint8)
        s.set_walk_periods(period, (rng.integers(0, 4, n) % period).astype(np.uint8))
    return s


def _run(s, ticks=3):
    s.step(ticks)
    s.sync()
    st = s.stats()
    return [*s.peds(), *s.decisions(), s.field()], {
        k: st[k] for k in ("t", "alive", "exited", "moved_total", "max_registrants", "decided", "near_ties")}


@pytest.mark.parametrize("W,H,n,periodic,walk", [
    (7, 5, 1, 0, False), (33, 31, 300, 1, False), (100, 100, 1024, 0, True), (100, 100, 1025, 1, True),
    (256, 256, 1000, 0, False), (257, 256, 1023, 0, False), (2048, 2048, 70000, 1, False),
    (2049, 2048, 70000, 0, False)])
def test_short_and_long_launch_sequences_agree(W, H, n, periodic, walk):
    got = []
    for timing in (False, True):  # a timed tick runs stage by stage
        for binning in ("grid", "peds", "auto"):
            with _sim(W, H, n, periodic, walk) as s:
                s.set_binning(binning)
                s.set_timing(timing)
                got.append(_run(s))
    for arrays, stats in got[1:]:
        assert stats == got[0][1]
        for a, b in zip(arrays, got[0][0]):
            np.testing.assert_array_equal(a, b)


# decide, vote and commit in one block up to 384 pedestrians, 768 on at most
# 128 x 128 su, 1024 on 64 x 64, 192 beyond radius 33
@pytest.mark.parametrize("W,H,r,n", [(64, 64, 5, 1024), (64, 64, 5, 1025), (65, 64, 5, 768), (128, 128, 33, 769),
                                     (129, 128, 33, 384), (300, 300, 5, 385), (90, 80, 34, 192), (90, 80, 34, 193)])
def test_one_block_or_three_launches(W, H, r, n):
    got = []
    for timing in (False, True):  # a timed tick runs stage by stage
        with _sim(W, H, n, 1, True, r) as s:
            s.set_timing(timing)
            before = s.stats()["kernel_launches"]
            got.append(_run(s, 1))
            got[-1][1]["launches"] = s.stats()["kernel_launches"] - before
    one = n <= (192 if r > 33 else 384 if W * H > 128 * 128 else 768 if W * H > 64 * 64 else 1024)
    assert got[1][1].pop("launches") - got[0][1].pop("launches") == (2 if one else 0)
    assert got[0][1] == got[1][1]
    for a, b in zip(got[0][0], got[1][0]):
        np.testing.assert_array_equal(a, b)


# Lattices whose last bins are ragged; 512 threads a bin up to twice the SMs in
# bins, else 128.  The crowd is a dense clump across the (periodic) border.
@pytest.mark.parametrize("W,H,periodic", [(121, 131, 0), (129, 127, 1), (40, 397, 1), (601, 581, 0),
                                          (609, 577, 1)])
@pytest.mark.parametrize("numbered", [False, True])
def test_stages_by_bins_agree_with_stages_by_pedestrian(W, H, periodic, numbered):
    """The per-bin stages run from a pedestrian slot per ten su on: the same
    crowd without and with enough slots that are not alive."""
    rng = np.random.default_rng(W * H)
    n, slots = W * H // 12, W * H // 9
    cell = np.zeros((H, W), np.uint8)
    cell[H // 2, :] = 1
    cell[:, 5] = 2
    free = np.flatnonzero(cell.ravel() == 0)
    x, y = free % W, free // W
    edge = np.minimum(x, W - 1 - x) + np.minimum(y, H - 1 - y)
    at = rng.permutation(free[np.argsort(edge, kind="stable")][:n * 5 // 4])[:n]
    xy = np.stack([at % W, at // W], 1).astype(np.int32)
    heading, goal = (rng.integers(0, 9, slots).astype(np.uint8) for _ in range(2))
    period = rng.integers(1, 4, slots).astype(np.uint8)
    phase = (rng.integers(0, 4, slots) % period).astype(np.uint8)
    ids = rng.permutation(slots).astype(np.int32)
    out = []
    for m in (n, slots):
        with sfm.Sim(W=W, H=H, cell=cell, periodic_x=periodic, periodic_y=periodic, r=4) as s:
            pad = np.zeros((m - n, 2), np.int32)
            s.place(np.concatenate([xy, pad]), heading[:m], goal[:m], (np.arange(m) < n).astype(np.uint8))
            s.set_walk_periods(period[:m], phase[:m])
            if numbered:
                s.set_ids(ids[:m])
            arrays, stats = _run(s, 4)
            assert not np.any(arrays[2][n:]) and not np.any(arrays[3][n:]) and not np.any(arrays[4][n:])
            out.append(([a if a.shape == (H, W) else a[:n] for a in arrays], stats))
    assert out[0][1] == out[1][1] and out[0][1]["max_registrants"] > 2 and out[0][1]["exited"] > 0
    for a, b in zip(*(o[0] for o in out)):
        np.testing.assert_array_equal(a, b)


# 16 x 16 footprints: up to 16 an SM (2432 on 152 SMs; 784^2 has 2401, 800^2
# 2500) four pedestrians are gathered at a time; full bins (over 32 records) are
# cut to the rows in reach.  One radius of each table stride the gather has.
@pytest.mark.parametrize("W,H,rho,r,periodic", [
    (3, 3, 0.4, 1, 1), (31, 33, 0.4, 1, 0), (83, 85, 0.4, 41, 1), (50, 70, 0.03, 9, 0), (97, 130, 0.3, 17, 1),
    (784, 784, 0.3, 25, 0), (800, 800, 0.3, 25, 1), (784, 784, 0.01, 33, 1), (300, 200, 0.2, 40, 0),
    (300, 200, 0.2, 45, 0)])
def test_footprints_agree_on_either_side_of_the_few(W, H, rho, r, periodic):
    rng = np.random.default_rng(r)
    n = max(1, int(rho * W * H))
    at = rng.choice(W * H, n, replace=False)
    fields = []
    with sfm.Sim(W=W, H=H, cell=np.zeros((H, W), np.uint8), periodic_x=periodic, periodic_y=periodic, r=r) as s:
        s.place(np.stack([at % W, at // W], 1).astype(np.int32), rng.integers(0, 9, n).astype(np.uint8),
                np.zeros(n, np.uint8))
        for shape in ("16x16", "32x16", "32x32r"):
            s.set_footprint(shape)
            s.compute_field()
            fields.append(s.field())
    for f in fields[1:]:
        np.testing.assert_array_equal(f, fields[0])


# Rectangles, also long ones (a side is shared by four lanes, or by a lane that
# reads three su at a time), for one block's slots and for more.
@pytest.mark.parametrize("W,H,n,periodic", [(90, 70, 700, 0), (200, 190, 3500, 1)])
def test_rectangles_follow_the_oracle(W, H, n, periodic):
    sc = SG.random_scene(W, H, n, r=5, seed=7, obstacles=0 if periodic else 2, periodic_x=periodic,
                         periodic_y=periodic, ring=not periodic, exits=() if periodic else ("east",),
                         exit_len=12, heading_mode="random")
    rng = np.random.default_rng(3)
    kinds = np.array([(1, 1), (1, 5), (7, 3), (9, 1), (3, 3)], np.uint8)
    size = kinds[rng.choice(len(kinds), n, p=[0.5, 0.15, 0.1, 0.1, 0.15])]
    keep, taken = [], set()
    for p in range(n):
        rc = rect_cells(W, H, periodic, periodic, *sc.xy[p], *size[p])
        if rc is None or rc & taken or any(sc.cell[v, u] != SG.FREE for u, v in rc):
            continue
        keep.append(p)
        taken |= rc
    assert (len(keep) > 1024) == (W == 200)
    sub = SG.Scene("rectangles", W, H, periodic, periodic, sc.cell, sc.xy[keep].copy(),
                   sc.heading[keep].copy(), sc.goal[keep].copy(), sc.params)
    w, h = (np.ascontiguousarray(size[keep, i]) for i in (0, 1))
    orc = OracleRun(sub)
    orc.st.w, orc.st.h = w, h
    with sfm.Sim(sub, place=False) as sim:
        sim.place_sized(sub.xy, sub.heading, sub.goal, np.ones(sub.n, np.uint8), w, h)
        for _ in range(8):
            sim.step(1)
            Fo, So = orc.field()
            ch_o, E, T, adm = orc.decide(Ffull=Fo.ravel(), Sfull=So.ravel())
            ch_g, won_g = sim.decisions()
            flips = compare_choices(ch_g, ch_o, E, T, adm)  # ties only
            won_o, most = orc.advance(np.asarray(ch_g, np.uint8) if flips else ch_o)
            np.testing.assert_array_equal(won_g, won_o)
            for x, y in zip(sim.peds(), (orc.st.xy, orc.st.heading, orc.st.alive)):
                np.testing.assert_array_equal(x, y)
        assert sim.stats()["max_registrants"] >= 2 and sim.stats()["error_flags"] == 0


# The allocation-free field on either side of 16 footprints of 32 x 32 su an SM
# (2432 on 152 SMs; 1568 x 1600 has 2450, 1568 x 1568 2401): each gather with its own table layout, several sizes in a
# row over the same scratch.  Its bins are in order of arrival: equal up to the
# rounding of an FP32 sum of at most a window's terms (1e-5 of it).
def test_allocation_free_field_takes_the_contexts_gather():
    torch = pytest.importorskip("torch")
    for W, H, n, r in [(1700, 1650, 9000, 3), (1700, 1620, 30000, 20), (40, 50, 300, 8), (1700, 1650, 0, 40),
                       (1700, 1650, 30000, 40), (1700, 1650, 30000, 45), (1568, 1600, 30000, 20),
                       (1568, 1568, 30000, 20)]:
        rng = np.random.default_rng(r)
        at = rng.choice(W * H, n, replace=False)
        xy = np.stack([at % W, at // W], 1).astype(np.int32)
        heading = rng.integers(0, 9, n).astype(np.uint8)
        with sfm.Sim(W=W, H=H, cell=np.zeros((H, W), np.uint8), r=r) as s:
            s.place(xy, heading, np.zeros(n, np.uint8))
            s.compute_field()
            want = s.field()
        base = torch.zeros((H, W), dtype=torch.float32, device="cuda")
        out = torch.full_like(base, float("nan"))
        assert sfm.sfm_field_noalloc(sfm.Lattice(W, H, 0, 0), sfm.make_params(r=r),
                                     torch.from_numpy(xy).cuda(), torch.from_numpy(heading).cuda(), None,
                                     base, out) == sfm.SFM_OK
        got = out.cpu().numpy()
        assert np.abs(got - want).max() <= 1e-5 * max(np.abs(want).max(), 1e-30)


@pytest.mark.parametrize("W,H,rows,r,periodic", [(2100, 2400, 1216, 5, 0), (2100, 2400, 1120, 5, 0),
                                                 (520, 640, 160, 33, 1), (520, 640, 160, 33, 0)])
def test_bands_take_the_footprint_of_their_own_rows(W, H, rows, r, periodic):
    """The default footprint goes by the footprints of one launch; whatever it
    is, the bands' fields and moves are the whole lattice's."""
    rng = np.random.default_rng(W + rows)
    n = W * H // 30
    at = rng.choice(W * H, n, replace=False)
    xy = np.stack([at % W, at // W], 1).astype(np.int32)
    heading, goal = (rng.integers(0, 9, n).astype(np.uint8) for _ in range(2))
    budget = sfm.band_budget(W, H, rows, periodic, periodic)
    kw = dict(W=W, H=H, cell=np.zeros((H, W), np.uint8), periodic_x=periodic, periodic_y=periodic, r=r)
    with sfm.Sim(**kw) as whole, sfm.Sim(hbm_budget_bytes=budget, **kw) as bands:
        assert bands.stats()["bands"] == -(-H // rows)
        for s in (whole, bands):
            s.place(xy, heading, goal)
            s.compute_field() if s is whole else None
        np.testing.assert_array_equal(bands.field_banded(), whole.field())
        for s in (whole, bands):
            s.step(3)
        for a, b in zip(whole.peds(), bands.peds()):
            np.testing.assert_array_equal(a, b)
