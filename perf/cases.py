"""The work that users of this library have it do, as cases that can be timed
and compared: episodes of a crowd in one lattice (room, counter-flow corridor,
large floor, periodic torus), the place / tick / read loop over host buffers,
multi-su pedestrians with walk periods, a batch of uneven rooms, the set-up of
a scene, ticks with the field at the candidates only, the allocation-free
field, and the surrogate's loss and gradients.

Every case goes through the public entry points of `paper_1803_04782_gb300`.
Sizes are those of the repository's own workloads (`scenegen`, `bench.py`, the
tests) or generic; scenes are drawn on the GPU from the seed alone, shaped like
`scenegen`'s.  Model constants are the library's defaults (k = 1, alpha = -0.5,
gamma = 0.5, beta = 1) throughout.
"""
import math

import numpy as np
import torch

import paper_1803_04782_gb300 as sfm

FREE, WALL, EXIT = 0, 1, 2
DIRS = ((0, 0), (1, 0), (1, 1), (0, 1), (-1, 1), (-1, 0), (-1, -1), (0, -1), (1, -1))


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call in earnest: the 100 x 100 room with 200 exit-seekers
        # and one exit, whole 50-tick run (launches and latency count)
        dict(name="room_run", kind="run", scene="room", W=100, H=100, n=200, r=10, ticks=50, bands=1,
             field=True),
        # the counter-flow corridor: few su, but dense thirds that jam
        dict(name="corridor_run", kind="run", scene="corridor", W=1000, H=200, n=20000, r=20, ticks=8,
             bands=1, field=False),
        # the benchmark's floor: a large sparse lattice in 4 row bands (the largest case)
        dict(name="floor_run", kind="run", scene="floor", W=16384, H=16384, n=1000000, r=40, ticks=4,
             bands=4, field=False),
        # the control loop of a host program: place from pinned host memory,
        # one tick, pedestrians back to the host, field left on the GPU
        dict(name="floor_loop", kind="loop", scene="floor", W=4096, H=4096, n=62500, r=40),
        # the paper's own experiments: periodic 1000 x 1000, half of it occupied,
        # 8 flows, the smallest and the largest field window (7 x 7 and 77 x 77)
        dict(name="torus_7x7", kind="run", scene="torus", W=1000, H=1000, n=500000, r=3, ticks=4,
             bands=1, field=False),
        dict(name="torus_77x77", kind="run", scene="torus", W=1000, H=1000, n=500000, r=38, ticks=1,
             bands=1, field=True),
        # 3 x 3 pedestrians with walk periods up to 5 (field window 21 x 21)
        dict(name="sized_walk", kind="sized", W=1000, H=1000, g=3, density=0.5, p_max=5, ticks=4),
        # a batch of uneven rooms, placed and stepped together
        dict(name="batch_rooms", kind="batch", scenes=32, side_lo=64, side_hi=1024, rho_lo=0.05,
             rho_hi=0.4, r_lo=5, r_hi=30, ticks=4),
        # setting up a scene: static field and guidance distances of a new floor
        dict(name="scene_setup", kind="setup", scene="floor", W=2048, H=2048, r=40),
        # ticks that compute the exact field at each pedestrian's candidates only
        dict(name="floor_candidates", kind="candidates", W=8192, H=8192, n=250000, r=40, ticks=4),
        # the allocation-free field of a crowd held in the caller's own buffers
        dict(name="field_noalloc", kind="noalloc", W=2048, H=2048, n=100000, r=20, periodic=0),
        # one loss and gradient of the field surrogate on a 512 x 512 coarse image
        dict(name="surrogate_grad", kind="grad", H=522, W=522),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; odd and ragged sizes throughout."""
    kind = rng.choice(["room", "corridor", "floor", "loop", "torus", "torus", "sized", "batch", "setup",
                       "candidates", "noalloc", "grad"])
    if kind == "room":
        W, H = _log_int(rng, 40, 400), _log_int(rng, 40, 400)
        return dict(kind="run", scene="room", W=W, H=H, n=max(1, int(rng.uniform(0.005, 0.1) * (W - 2) * (H - 2))),
                    r=rng.randint(3, 15), ticks=rng.choice([1, 10, 50]), bands=1, field=True)
    if kind == "corridor":
        W, H = _log_int(rng, 300, 3000), _log_int(rng, 60, 400)
        return dict(kind="run", scene="corridor", W=W, H=H, n=int(rng.uniform(0.02, 0.2) * W * (H - 2)),
                    r=rng.randint(8, 30), ticks=rng.choice([1, 4, 8]), bands=1, field=False)
    if kind == "floor":
        W = H = _log_int(rng, 1500, 12000)
        bands = rng.choice([1, 4])
        return dict(kind="run", scene="floor", W=W, H=H, n=W * H // 268, r=rng.randint(20, 40),
                    ticks=rng.choice([1, 4]), bands=bands, field=bands == 1)
    if kind == "loop":
        W = H = _log_int(rng, 700, 6000)
        return dict(kind="loop", scene="floor", W=W, H=H, n=int(W * H * rng.uniform(0.002, 0.01)),
                    r=rng.randint(20, 40))
    if kind == "torus":
        s = rng.randint(100, 1000)
        return dict(kind="run", scene="torus", W=s, H=s, n=int(s * s * rng.uniform(0.1, 0.9)),
                    r=rng.choice([3, 10, 17, 24, 31, 38]), ticks=1, bands=1, field=True)
    if kind == "sized":
        g = rng.choice([3, 5, 7])
        return dict(kind="sized", W=rng.randint(300, 1000), H=rng.randint(300, 1000), g=g,
                    density=round(rng.uniform(0.2, 0.6), 3), p_max=rng.choice([1, 3, 11]), ticks=4)
    if kind == "batch":
        return dict(kind="batch", scenes=rng.randint(4, 48), side_lo=64, side_hi=_log_int(rng, 128, 900),
                    rho_lo=0.05, rho_hi=0.4, r_lo=5, r_hi=30, ticks=rng.choice([1, 4]))
    if kind == "setup":
        W, H = _log_int(rng, 256, 4096), _log_int(rng, 256, 4096)
        return dict(kind="setup", scene="floor", W=W, H=H, r=rng.randint(3, 40))
    if kind == "candidates":
        W = H = 8 * _log_int(rng, 64, 1024)
        return dict(kind="candidates", W=W, H=H, n=W * H // 268, r=rng.randint(10, 40), ticks=4)
    if kind == "noalloc":
        W, H = _log_int(rng, 200, 4096), _log_int(rng, 200, 4096)
        return dict(kind="noalloc", W=W, H=H, n=min(1 << 20, int(W * H * rng.uniform(0.004, 0.2))),
                    r=rng.randint(3, 40), periodic=rng.choice([0, 1]))
    return dict(kind="grad", H=10 + _log_int(rng, 20, 520), W=10 + _log_int(rng, 20, 520))


# --------------------------------------------------------------------- scenes
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _ring(W, H):
    cell = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    cell[0, :] = WALL
    cell[-1, :] = WALL
    cell[:, 0] = WALL
    cell[:, -1] = WALL
    return cell


def _exit(cell, side, length):
    H, W = cell.shape
    span = H if side in ("east", "west") else W
    lo = max(1, span // 2 - length // 2)
    hi = min(span - 1, lo + length)
    if side == "east":
        cell[lo:hi, W - 1] = EXIT
    elif side == "west":
        cell[lo:hi, 0] = EXIT
    elif side == "north":
        cell[H - 1, lo:hi] = EXIT
    else:
        cell[0, lo:hi] = EXIT


def _pick(g, mask, n):
    """n distinct su of `mask`, uniform, as (x, y) int32 pairs on the GPU."""
    W = mask.shape[1]
    flat = mask.reshape(-1)
    if flat.numel() <= 1 << 22 or 8 * n > flat.numel():
        free = torch.nonzero(flat).reshape(-1)
        idx = free[torch.randperm(free.numel(), generator=g, device="cuda")[:n]]
    else:
        c = torch.randint(flat.numel(), (int(1.5 * n) + 4096,), generator=g, device="cuda")
        c = torch.unique(c[flat[c]])
        idx = c[torch.randperm(c.numel(), generator=g, device="cuda")[:n]]
    assert idx.numel() == n, "not enough free su"
    return torch.stack([idx % W, idx // W], dim=1).to(torch.int32).contiguous()


def _scene(c, seed):
    """cell, xy, heading, goal (CUDA tensors) and the periodic flags."""
    g, W, H, n = _gen(seed), c["W"], c["H"], c.get("n", 0)
    zeros = torch.zeros(n, dtype=torch.uint8, device="cuda")
    if c["scene"] == "room":
        cell = _ring(W, H)
        _exit(cell, "east", max(2, H // 10))
        return cell, _pick(g, cell == FREE, n), zeros, zeros.clone(), 0, 0
    if c["scene"] == "corridor":
        cell = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
        cell[0, :] = WALL
        cell[-1, :] = WALL
        west, east = cell == FREE, cell == FREE
        west[:, W // 3:] = False
        east[:, : W - W // 3] = False
        a = n // 2
        xy = torch.cat([_pick(g, west, a), _pick(g, east, n - a)])
        goal = torch.full((n,), 5, dtype=torch.uint8, device="cuda")
        goal[:a] = 1
        return cell, xy, goal.clone(), goal, 1, 0
    if c["scene"] == "floor":
        # rectangles of 5..200 su a side until a tenth of the area is wall
        cell = _ring(W, H)
        rng = np.random.default_rng(seed)
        top = min(200, max(6, min(W, H) // 8))
        k = max(1, int(0.11 * W * H / ((5 + top) / 2) ** 2))
        for x0, y0, w, h in zip(rng.integers(1, W - 1, k), rng.integers(1, H - 1, k),
                                rng.integers(5, top + 1, k), rng.integers(5, top + 1, k)):
            cell[y0:min(H - 1, y0 + h), x0:min(W - 1, x0 + w)] = WALL
        for side in ("east", "west", "north", "south"):
            _exit(cell, side, max(4, min(W, H) // 64))
        return cell, _pick(g, cell == FREE, n), zeros, zeros.clone(), 0, 0
    # torus: no walls, walkers of 8 flows headed their way
    cell = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    goal = (1 + torch.arange(n, device="cuda") % 8).to(torch.uint8)
    goal = goal[torch.randperm(n, generator=g, device="cuda")].contiguous()
    return cell, _pick(g, cell == FREE, n), goal.clone(), goal, 1, 1


def _budget(c, px, py):
    if c.get("bands", 1) <= 1:
        return 0
    rows = -(-c["H"] // c["bands"])
    return sfm.band_budget(c["W"], c["H"], -(-rows // 32) * 32, px, py) + 4096


def _sim(c, seed):
    cell, xy, heading, goal, px, py = _scene(c, seed)
    sim = sfm.Sim(W=c["W"], H=c["H"], cell=cell, periodic_x=px, periodic_y=py, r=c["r"], seed=seed,
                  hbm_budget_bytes=_budget(c, px, py))
    return dict(case=c, sim=sim, cell=cell, xy=xy, heading=heading, goal=goal, px=px, py=py)


class _Room:
    """What sfm.Batch takes: one lattice with its crowd and parameters."""

    def __init__(self, side, cell, xy, r, seed):
        self.W = self.H = side
        self.periodic_x = self.periodic_y = 0
        self.cell, self.xy = cell, xy
        self.heading = np.zeros(len(xy), np.uint8)
        self.goal = np.zeros(len(xy), np.uint8)
        self.params = dict(r=r, seed=seed)


def _rooms(c, seed):
    rng, g, rooms = np.random.default_rng(c["scenes"]), _gen(seed), []
    # sides, densities, radii and exits cover their ranges the same way
    # whatever the seed, which places the crowds
    sides = np.linspace(c["side_lo"], c["side_hi"], c["scenes"]).astype(int)
    rhos = rng.permutation(np.linspace(c["rho_lo"], c["rho_hi"], c["scenes"]))
    rs = rng.permutation(np.linspace(c["r_lo"], c["r_hi"], c["scenes"])).astype(int)
    for i, (s, rho, r) in enumerate(zip(sides, rhos, rs)):
        cell = _ring(int(s), int(s))
        for side in rng.permutation(["east", "west", "north", "south"])[: 1 + i % 4]:
            _exit(cell, str(side), max(4, int(s) // 16))
        free = cell == FREE
        xy = _pick(g, free, int(rho * int(free.sum())))
        rooms.append(_Room(int(s), cell.cpu().numpy(), xy.cpu().numpy(), int(r), seed * 1000 + i))
    return rooms


# -------------------------------------------------------------------- prepare
def prepare(case, seed):
    c, kind = dict(case), case["kind"]
    dev = dict(device="cuda")
    if kind == "run":
        s = _sim(c, seed)
        n = c["n"]
        s["out"] = dict(xy=torch.empty((n, 2), dtype=torch.int32, **dev),
                        heading=torch.empty(n, dtype=torch.uint8, **dev),
                        alive=torch.empty(n, dtype=torch.uint8, **dev))
        if c["field"]:
            s["out"]["field"] = torch.empty((c["H"], c["W"]), dtype=torch.float32, **dev)
        sfm.sfm_place(s["sim"].ctx, s["xy"], s["heading"], s["goal"])
        return s
    if kind == "loop":
        s = _sim(c, seed)
        n = c["n"]
        s["host"] = [t.cpu().pin_memory() for t in (s["xy"], s["heading"], s["goal"])]
        s["out"] = dict(xy=torch.empty((n, 2), dtype=torch.int32).pin_memory(),
                        heading=torch.empty(n, dtype=torch.uint8).pin_memory(),
                        alive=torch.empty(n, dtype=torch.uint8).pin_memory(),
                        field=torch.empty((c["H"], c["W"]), dtype=torch.float32, **dev))
        sfm.sfm_place(s["sim"].ctx, *s["host"])
        return s
    if kind == "sized":
        # g x g rectangles in randomly chosen cells of a g x g tiling, so none overlap
        W, H, gs = c["W"], c["H"], c["g"]
        rng = np.random.default_rng(seed)
        nbx, nby = W // gs, H // gs
        n = min(nbx * nby, int(round(c["density"] * W * H / gs ** 2)))
        pick = rng.choice(nbx * nby, size=n, replace=False)
        xy = np.stack([(pick % nbx) * gs + gs // 2, (pick // nbx) * gs + gs // 2], 1).astype(np.int32)
        goal = (1 + np.arange(n) % 8).astype(np.uint8)
        rng.shuffle(goal)
        side = np.full(n, gs, np.uint8)
        period = rng.integers(1, c["p_max"] + 1, size=n).astype(np.uint8)
        phase = (rng.integers(0, 1 << 16, size=n) % period).astype(np.uint8)
        sim = sfm.Sim(W=W, H=H, cell=np.zeros((H, W), np.uint8), periodic_x=1, periodic_y=1,
                      r=(7 * gs - 1) // 2, seed=seed)
        sim.place_sized(xy, goal, goal, np.ones(n, np.uint8), side, side)
        sim.set_walk_periods(period, phase)
        out = dict(xy=torch.empty((n, 2), dtype=torch.int32, **dev),
                   heading=torch.empty(n, dtype=torch.uint8, **dev))
        return dict(case=c, sim=sim, out=out)
    if kind == "batch":
        b = sfm.Batch(_rooms(c, seed))
        n = int(b.ped_off[-1])
        crowd = dict(counts=[len(s.xy) for s in b.scenes],
                     xy=torch.from_numpy(np.concatenate([s.xy for s in b.scenes])).cuda(),
                     heading=torch.zeros(n, dtype=torch.uint8, **dev),
                     goal=torch.zeros(n, dtype=torch.uint8, **dev))
        out = dict(xy=torch.empty((n, 2), dtype=torch.int32, **dev),
                   heading=torch.empty(n, dtype=torch.uint8, **dev),
                   alive=torch.empty(n, dtype=torch.uint8, **dev))
        if c["ticks"] == 1:
            out["field"] = torch.empty(int(b.su_off[-1]), dtype=torch.float32, **dev)
        return dict(case=c, batch=b, crowd=crowd, out=out)
    if kind == "setup":
        cell = _scene(dict(c, n=1), seed)[0]
        out = dict(static=torch.empty((c["H"], c["W"]), dtype=torch.float32, **dev),
                   guidance=torch.empty((c["H"], c["W"]), dtype=torch.int32, **dev))
        return dict(case=c, cell=cell, out=out, seed=seed)
    if kind == "candidates":
        s = _sim(dict(c, scene="floor"), seed)
        n = c["n"]
        s["case"] = c
        s["sur"] = sfm.Surrogate(coarsen=8, near_radius=3)  # delta = +inf: the exact field at the candidates
        s["out"] = dict(xy=torch.empty((n, 2), dtype=torch.int32, **dev),
                        heading=torch.empty(n, dtype=torch.uint8, **dev),
                        alive=torch.empty(n, dtype=torch.uint8, **dev))
        sfm.sfm_place(s["sim"].ctx, s["xy"], s["heading"], s["goal"])
        return s
    if kind == "noalloc":
        g = _gen(seed)
        W, H, n = c["W"], c["H"], c["n"]
        p = c["periodic"] if min(W, H) >= 2 * c["r"] + 1 else 0
        return dict(case=c, lat=sfm.Lattice(W, H, p, p), prm=sfm.make_params(r=c["r"]),
                    xy=_pick(g, torch.ones((H, W), dtype=torch.bool, **dev), n),
                    heading=torch.randint(0, 9, (n,), generator=g, dtype=torch.uint8, **dev),
                    alive=torch.ones(n, dtype=torch.uint8, **dev),
                    base=torch.rand((H, W), generator=g, **dev),
                    field=torch.empty((H, W), dtype=torch.float32, **dev))
    # grad: per-cell counts and heading sums of a crowd (64 su a cell), and
    # targets of the size that the far field has in training
    params, X, T = _network(c, seed)
    flat = sfm.flatten_params(params)
    return dict(case=c, sur=sfm.Surrogate(params=flat), X=X, T=T)


def _bf16(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(torch.bfloat16).float().numpy()


def _network(c, seed):
    rng = np.random.default_rng(seed)
    params = []
    for cin, cout, k in ((3, 32, 5), (32, 32, 3), (32, 32, 3), (32, 1, 3)):
        W = rng.normal(0.0, math.sqrt(2.0 / (cin * k * k)), (cout, cin, k, k))
        params.append((_bf16(W), _bf16(rng.normal(0.0, 0.05, cout))))
    n = rng.poisson(4.0, (c["H"], c["W"])).astype(np.float32)
    ang = rng.uniform(0.0, 2.0 * math.pi, n.shape)
    mag = np.sqrt(n) * rng.random(n.shape)
    X = _bf16(np.stack([n, mag * np.cos(ang), mag * np.sin(ang)]) / 64.0)
    T = rng.normal(0.5, 0.5, (c["H"] - 10, c["W"] - 10)).astype(np.float32)
    return params, X, T


# ------------------------------------------------------------------------ run
def run(s):
    c, kind = s["case"], s["case"]["kind"]
    o = s.get("out")
    if kind == "run":
        # an episode from the crowd at hand: place it, run, read it back
        ctx = s["sim"].ctx
        sfm.sfm_place(ctx, s["xy"], s["heading"], s["goal"])
        sfm.sfm_set_time(ctx, 0)
        sfm.sfm_step(ctx, c["ticks"])
        if c["field"]:
            sfm.sfm_read_field(ctx, o["field"])
        sfm.sfm_read_peds(ctx, o["xy"], o["heading"], o["alive"])
        return o
    if kind == "loop":
        ctx = s["sim"].ctx
        sfm.sfm_place(ctx, *s["host"])
        sfm.sfm_step(ctx, 1)
        sfm.sfm_read_field(ctx, o["field"])
        sfm.sfm_read_peds(ctx, o["xy"], o["heading"], o["alive"])
        return o
    if kind == "sized":
        # a run that goes on (nobody leaves a torus): the next ticks
        sfm.sfm_step(s["sim"].ctx, c["ticks"])
        sfm.sfm_read_peds(s["sim"].ctx, o["xy"], o["heading"])
        return o
    if kind == "batch":
        ctx, w = s["batch"].ctx, s["crowd"]
        sfm.sfm_batch_place(ctx, w["counts"], w["xy"], w["heading"], w["goal"])
        sfm.sfm_set_time(ctx, 0)
        sfm.sfm_step(ctx, c["ticks"])
        if "field" in o:
            sfm.sfm_read_field(ctx, o["field"])
        sfm.sfm_read_peds(ctx, o["xy"], o["heading"], o["alive"])
        return o
    if kind == "setup":
        sim = sfm.Sim(W=c["W"], H=c["H"], cell=s["cell"], r=c["r"], seed=s["seed"])
        sfm.sfm_read_static_field(sim.ctx, o["static"])
        sfm.sfm_read_guidance(sim.ctx, o["guidance"])
        sim.close()
        return o
    if kind == "candidates":
        ctx = s["sim"].ctx
        sfm.sfm_place(ctx, s["xy"], s["heading"], s["goal"])
        sfm.sfm_set_time(ctx, 0)
        s["sur"].step(s["sim"], c["ticks"])
        sfm.sfm_read_peds(ctx, o["xy"], o["heading"], o["alive"])
        return o
    if kind == "noalloc":
        st = sfm.sfm_field_noalloc(s["lat"], s["prm"], s["xy"], s["heading"], s["alive"], s["base"],
                                   s["field"])
        return dict(status=st, field=s["field"])
    loss, grads = s["sur"].grad(s["X"], s["T"])
    return dict(loss=loss, grads=grads)


# ----------------------------------------------------------------------- work
def _tick_work(W, H, n, r, ticks):
    # a tick: the static field read, the field written (4 bytes a su each), 64
    # bytes a pedestrian (state, records, candidates, moves); one addition a
    # pair of a su and a pedestrian within reach
    return ticks * (8.0 * W * H + 64.0 * n), ticks * float(n) * (2 * r + 1) ** 2


def work(case):
    c, kind = case, case["kind"]
    if kind in ("run", "loop"):
        b, f = _tick_work(c["W"], c["H"], c["n"], c["r"], c.get("ticks", 1))
        b += 20.0 * c["n"] + (4.0 * c["W"] * c["H"] if c.get("field", True) else 0.0)
    elif kind == "sized":
        n = c["density"] * c["W"] * c["H"] / c["g"] ** 2
        b, f = _tick_work(c["W"], c["H"], n, (7 * c["g"] - 1) // 2, c["ticks"])
        b += 9.0 * n
    elif kind == "batch":
        side = (c["side_lo"] ** 2 + c["side_lo"] * c["side_hi"] + c["side_hi"] ** 2) / 3.0
        n = 0.5 * (c["rho_lo"] + c["rho_hi"]) * side
        b, f = _tick_work(side, 1.0, n, 0.5 * (c["r_lo"] + c["r_hi"]), c["ticks"])
        b, f = c["scenes"] * (b + 20.0 * n), c["scenes"] * f
    elif kind == "setup":
        # cells read, static field and distances written and read back; one
        # addition for each wall su (a tenth of the area) within reach of a su
        b = 17.0 * c["W"] * c["H"]
        f = 0.1 * c["W"] * c["H"] * (2 * c["r"] + 1) ** 2
    elif kind == "candidates":
        # no lattice field: the static field at 9 su a pedestrian, and the
        # pairs of those 9 su
        b = c["ticks"] * 136.0 * c["n"] + 20.0 * c["n"]
        f = c["ticks"] * 9.0 * c["n"] * c["n"] * (2 * c["r"] + 1) ** 2 / (c["W"] * c["H"])
    elif kind == "noalloc":
        b = 8.0 * c["W"] * c["H"] + 10.0 * c["n"]
        f = float(c["n"]) * (2 * c["r"] + 1) ** 2
    else:
        px = float((c["H"] - 10) * (c["W"] - 10))
        per = 2.0 * (75 * 32 + 2 * 288 * 32 + 288)  # forward multiply-adds of a pixel, as flops
        b, f = 20.0 * px, 3.0 * per * px - 2.0 * 75 * 32 * px
    return dict(bytes=b, flops=f)


# ------------------------------------------------------------------ tolerance
def tolerance(case):
    kind = case["kind"]
    if kind == "grad":
        # BF16 activations between FP32-accumulated layers: another order of
        # the sums moves single activations by one BF16 rounding (the present
        # gradients are 1e-4 off 64 bits on the listed image, 6e-4 on a small one)
        return dict(rel=2e-3, max=2e-2)
    if kind == "noalloc":
        return dict(rel=2e-6, max=2e-5)
    if kind == "setup":
        return dict(rel=1e-6, max=1e-5, differ=0.0)
    # 32-bit sums of the field (up to 9e-7 off 64 bits for a dense crowd); a
    # decision between two energies that agree to their rounding may fall
    # either way and moves one pedestrian, and its neighbours on the ticks
    # after.  With the kernels' constants scaled by 1 + 2^-22, about what such
    # sums are off by, up to 8e-4 of the values differ (batch, 4 ticks).
    return dict(rel=2e-6, max=2e-5, differ=4e-3)


# ---------------------------------------------------------------------- exact
def _kernels(r, gamma):
    ax = torch.arange(-r, r + 1, dtype=torch.float64, device="cuda")
    dy, dx = torch.meshgrid(ax, ax, indexing="ij")
    d = torch.sqrt(dx * dx + dy * dy)
    d[r, r] = 1.0
    base = d ** -0.5
    base[r, r] = 0.0
    out = []
    for hx, hy in DIRS:
        m = math.hypot(hx, hy) or 1.0
        out.append(base * (1.0 + gamma * (hx / m * dx + hy / m * dy) / d))
    return base, out


def _convolve(planes, kernels, r, px, py):
    """sum_i planes[i] (H x W) convolved with kernels[i] ((2r+1)^2), in 64 bits."""
    H, W = planes[0].shape
    Hp, Wp = H if py else H + 2 * r, W if px else W + 2 * r
    acc = None
    for p, k in zip(planes, kernels):
        K = torch.zeros((Hp, Wp), dtype=torch.float64, device="cuda")
        K[: 2 * r + 1, : 2 * r + 1] = k
        K = torch.roll(K, (-r, -r), (0, 1))
        P = torch.zeros((Hp, Wp), dtype=torch.float64, device="cuda")
        P[:H, :W] = p
        z = torch.fft.rfft2(P) * torch.fft.rfft2(K)
        acc = z if acc is None else acc + z
    return torch.fft.irfft2(acc, s=(Hp, Wp))[:H, :W]


def _crowd_field(W, H, xy, heading, r, px, py, gamma=0.5):
    _, ks = _kernels(r, gamma)
    planes = []
    idx = xy[:, 1].long() * W + xy[:, 0].long()
    for h in range(9):
        p = torch.zeros(H * W, dtype=torch.float64, device="cuda")
        p[idx[heading == h]] = 1.0
        planes.append(p.view(H, W))
    return _convolve(planes, ks, r, px, py)


def _static_field(cell, r, px, py):
    base, _ = _kernels(r, 0.0)
    return _convolve([(cell == WALL).double(), (cell == EXIT).double()], [base, -base], r, px, py)


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind in ("run", "loop"):
        if kind == "run" and not (c["field"] and c["ticks"] == 1):
            return None  # what the ticks leave behind are whole numbers
        cell, xy, heading, _, px, py = _scene(c, seed)
        F = _crowd_field(c["W"], c["H"], xy, heading, c["r"], px, py)
        F += _static_field(cell, c["r"], px, py)
        return dict(xy=None, heading=None, alive=None, field=F)
    if kind == "batch":
        if c["ticks"] != 1:
            return None
        F = []
        for s in _rooms(c, seed):
            xy, cell = torch.from_numpy(s.xy).cuda(), torch.from_numpy(s.cell).cuda()
            h = torch.zeros(len(s.xy), dtype=torch.uint8, device="cuda")
            f = _crowd_field(s.W, s.H, xy, h, s.params["r"], 0, 0)
            F.append((f + _static_field(cell, s.params["r"], 0, 0)).reshape(-1))
        return dict(xy=None, heading=None, alive=None, field=torch.cat(F))
    if kind == "setup":
        cell = _scene(dict(c, n=1), seed)[0]
        return dict(static=_static_field(cell, c["r"], 0, 0), guidance=None)
    if kind == "noalloc":
        s = prepare(c, seed)
        F = _crowd_field(c["W"], c["H"], s["xy"], s["heading"], c["r"], s["lat"].periodic_x,
                         s["lat"].periodic_y)
        return dict(status=None, field=F + s["base"].double())
    if kind == "grad":
        params, X, T = _network(c, seed)
        ws = [(torch.tensor(W, dtype=torch.float64, device="cuda", requires_grad=True),
               torch.tensor(b, dtype=torch.float64, device="cuda", requires_grad=True))
              for W, b in params]
        x = torch.tensor(X, dtype=torch.float64, device="cuda")[None]
        for i, (W, b) in enumerate(ws):
            cols = x.unfold(2, W.shape[2], 1).unfold(3, W.shape[3], 1)
            x = torch.einsum("ncyxij,ocij->noyx", cols, W) + b[None, :, None, None]
            if i < 3:
                x = torch.relu(x)
        loss = 0.5 * torch.mean((x[0, 0] - torch.tensor(T, dtype=torch.float64, device="cuda")) ** 2)
        loss.backward()
        g = torch.cat([t.grad.reshape(-1) for wb in ws for t in wb])
        return dict(loss=float(loss), grads=g)
    return None
