"""Contexts side by side: launches that need different amounts of shared memory
of one kernel do not take each other's limit away, whether they come from
several host threads or from contexts made one after the other."""
import threading

import numpy as np
import pytest

import paper_1803_04782_gb300 as sfm
import scenegen as SG
from paper_1803_04782_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build()
    sfm.lib()


def _scene(r, rho, seed):
    return SG.random_scene(96, 96, int(rho * 96 * 96), r=r, seed=seed, periodic_x=1, periodic_y=1, ring=False,
                           exits=(), goal_mode="fixed", heading_mode="random")


# the product of crowded lattices, the 16 x 16 gather (two radii of one table
# stride), the scene's own static field
@pytest.mark.parametrize("rho,radii", [(0.5, (3, 40)), (0.2, (33, 40)), (0.2, (42, 47))])
def test_host_threads_with_contexts_of_their_own(rho, radii):
    want, errors = {}, []
    scenes = {r: _scene(r, rho, 40 + r) for r in radii}
    for r, sc in scenes.items():
        with sfm.Sim(sc) as s:
            s.compute_field()
            want[r] = s.field()
    go = threading.Barrier(len(radii))

    def work(r):
        try:
            with sfm.Sim(scenes[r]) as s:
                go.wait()
                for k in range(400):
                    s.compute_field()
                    if k % 100 == 0:
                        np.testing.assert_array_equal(s.field(), want[r])
                s.sync()
        except BaseException as e:  # noqa: BLE001 - reported below
            errors.append(f"r = {r}: {e}")
    threads = [threading.Thread(target=work, args=(r,)) for r in radii]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_a_batch_steps_after_a_smaller_one_was_made():
    big, small = [_scene(45, 0.2, 1)], [_scene(3, 0.2, 2)]
    with sfm.Batch(big) as alone:
        alone.step(2)
        want = [np.asarray(a[0]).copy() for a in alone.peds()]
    with sfm.Batch(big) as a, sfm.Batch(small) as b:
        a.step(2)
        b.step(2)
        for x, y in zip(want, a.peds()):
            np.testing.assert_array_equal(x, y[0])


@pytest.mark.parametrize("batch", [False, True])
def test_a_placement_that_does_not_fit_leaves_nobody_placed(batch):
    """The arrays of the crowd before are gone by then: a step must refuse, and
    a smaller placement work as in a new context."""
    torch = pytest.importorskip("torch")
    sc, n = _scene(5, 0.2, 3), 40_000_000  # 44 bytes a pedestrian of a context, 23 of a batch's
    big = np.zeros((n, 2), np.int32)
    make = (lambda: sfm.Batch([sc])) if batch else (lambda: sfm.Sim(sc))
    with make() as s, make() as ref:
        s.step(2)
        s.sync()
        free, _ = torch.cuda.mem_get_info()
        hold = torch.empty(free - (600 << 20), dtype=torch.uint8, device="cuda")
        with pytest.raises(sfm.SfmError) as e:
            if batch:
                sfm.sfm_batch_place(s.ctx, [n], big, None, None)
            else:
                s.place(big)
        assert e.value.status == sfm.SFM_ENOMEM
        del hold
        torch.cuda.empty_cache()
        with pytest.raises(sfm.SfmError) as e:
            s.step(1)
        assert e.value.status == sfm.SFM_ESTATE and s.stats()["n"] == 0
        for x in (s, ref):
            if batch:
                sfm.sfm_batch_place(x.ctx, [sc.n], sc.xy, sc.heading, sc.goal)
            else:
                x.place(sc.xy, sc.heading, sc.goal)
            sfm.sfm_set_time(x.ctx, 0)
            x.step(3)
        for a, b in zip(s.peds(), ref.peds()):
            np.testing.assert_array_equal(np.asarray(a), np.asarray(b))


def test_an_image_that_does_not_fit_leaves_none():
    """A surrogate whose buffers could not be grown: the size before works again."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(5)
    X, T = rng.random((3, 60, 70), np.float32), rng.random((50, 60), np.float32)
    flat = rng.normal(0, 0.1, int(sfm.lib().sfm_surrogate_nparams())).astype(np.float32)
    big = np.zeros((3, 2058, 2058), np.float32)  # activations of 2.4 GB
    with sfm.Surrogate(params=flat) as sur:
        loss, grads = sur.grad(X, T)
        free, _ = torch.cuda.mem_get_info()
        hold = torch.empty(free - (600 << 20), dtype=torch.uint8, device="cuda")
        with pytest.raises(sfm.SfmError) as e:
            sur.grad(big, np.zeros((2048, 2048), np.float32))
        assert e.value.status == sfm.SFM_ENOMEM
        del hold
        torch.cuda.empty_cache()
        again = sur.grad(X, T)
        assert again[0] == loss
        np.testing.assert_array_equal(again[1], grads)
