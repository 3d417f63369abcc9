"""Guidance distances of lattices of few tiles, set up again and again, against
the oracle's Dijkstra: the kernel's CTAs then take every tile from the queue
many times, in an order that differs from run to run."""
import time

import numpy as np
import pytest

import oracle as O
import paper_1803_04782_gb300 as sfm
import scenegen as SG
from paper_1803_04782_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()
    O.build()
    sfm.lib()


def _maze(W, H, px, py, seed):
    """Walls every few rows with a gap at alternating ends; exits in two corners."""
    sc = SG.random_scene(W, H, 1, r=1, seed=seed, periodic_x=px, periodic_y=py, ring=False, exits=())
    cell = np.zeros((H, W), np.uint8)
    for k, y in enumerate(range(3 + seed % 3, H - 1, 4)):
        cell[y, :] = 1
        cell[y, (1 if k % 2 else W - 2)] = 0
    cell[0, 0] = cell[H - 1, W - 1] = 2
    sc.cell = cell
    return sc


@pytest.mark.parametrize("W,H,px,py", [(33, 32, 0, 0), (64, 32, 1, 0), (65, 33, 1, 1), (96, 33, 0, 1),
                                       (40, 130, 0, 0), (96, 96, 1, 1), (90, 77, 0, 0)])
def test_few_tiles_again_and_again(W, H, px, py):
    for seed in range(3):
        sc = _maze(W, H, px, py, seed)
        want = O.guidance(O.model(sc), sc.cell)
        for _ in range(12):
            with sfm.Sim(W=W, H=H, cell=sc.cell, periodic_x=px, periodic_y=py, r=1) as s:
                np.testing.assert_array_equal(s.guidance(), want)


def test_a_tile_that_is_never_finished_ends_the_wait():
    sc = _maze(200, 150, 0, 0, 0)
    with sfm.Sim(W=200, H=150, cell=sc.cell, r=1) as s:
        before = s.guidance()
        t0 = time.time()
        with pytest.raises(sfm.SfmError) as e:
            sfm.sfm_test_wait_out(s.ctx, 1)
        assert e.value.status == sfm.SFM_ETIMEOUT and time.time() - t0 < 10
        np.testing.assert_array_equal(s.guidance(), before)
        s.sync()
