"""The crowded lattice's field product, on CPU: its limb tables, operand
addresses and sums, restated in NumPy from their description (sfm_product.cu),
give the window sums of the class-table law for every radius class, and no
entry, sum or address leaves its range."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

TW, TH, MAXR, SMEM = 64, 256, 44, 227 * 1024


def chunks(r):
    return (2 * r + 8 + 15) // 16


def pitch(r):
    return (TW - 8 + 16 * chunks(r)) * 2


@pytest.fixture(scope="module")
def chosen(tmp_path_factory):
    """The library's own choice of scales (None: refused)."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("limbs") / "scales")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_1803_04782_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "limb_scales_host.cpp"), "-o", exe], check=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, check=True).stdout
        return None if out.startswith("refused") else tuple(float(v) for v in out.split())
    return run


def limb16(v):
    return np.where(np.abs(v) > 2048, v.astype(np.float16).astype(np.float64), np.rint(v))


def split(v, s0, s1):
    hi = limb16(v * s0)
    return hi, limb16((v * s0 - hi) * s1)


def law(r, ch, k=1.0, a=-0.5, g=0.5):
    ax = np.arange(-r, r + 1, dtype=np.float64)
    dy, dx = np.meshgrid(ax, ax, indexing="ij")
    d = np.hypot(dx, dy)
    d[r, r] = 1.0
    q = math.sqrt(0.5)
    v = k * d ** a * (1.0, g * dx / d, g * dy / d, g * q * (dx + dy) / d, g * q * (dy - dx) / d)[ch]
    v[r, r] = 0.0
    return v


def partial_sums(first, axes):
    """Largest magnitude that a sum of a limb can reach over full windows: the
    planes one after the other, presence first, a su with one heading at most."""
    m = np.max(np.abs(axes), axis=0)
    return max(np.maximum(0, first + m).sum(), np.maximum(0, m - first).sum(), m.sum())


def crowd_limbs(r, s, k, a, g):
    limbs = [split(law(r, ch, k, a, g), *s) for ch in range(5)]
    for hi, lo in limbs:
        for limb in (hi, lo):  # integers that FP16 holds
            assert (limb == limb.astype(np.float16).astype(np.float64)).all() and (limb == np.rint(limb)).all()
    return limbs


@pytest.mark.parametrize("r", [1, 2, 3, 7, 12, 20, 31, 32, 36, 37, 40, 44])
def test_limbs_are_exact_and_their_sums_fit(chosen, r):
    s = chosen("crowd", r, 1.0, -0.5, 0.5)
    limbs = crowd_limbs(r, s, 1.0, -0.5, 0.5)
    for i in range(2):
        assert partial_sums(limbs[0][i], [l[i] for l in limbs[1:]]) < 2 ** 24   # exact in FP32
    # what the second limb's rounding leaves, for one pedestrian
    err = [np.abs(hi / s[0] + lo / (s[0] * s[1]) - law(r, ch)) for ch, (hi, lo) in enumerate(limbs)]
    assert (err[0] + np.max(err[1:], axis=0) <= (2.2e-7 if r <= 40 else 2.0 ** -21) * law(r, 0)).all()


def test_sums_fit_for_flat_rising_and_steep_laws(chosen):
    """Every law that the library takes, over exponents, heading weights and
    magnitudes: flat ones just above a power of two have large second limbs
    all over the window."""
    taken = 0
    for r in (3, 17, 28, 31, 44):
        for a in (-2.0, -1.0, -0.3, -0.05, 0.0, 0.05, 0.5, 1.0):
            for g in (0.0, 0.5, 1.0, 1.7, 2.0):
                for k in (1.0, 0.51, 2049.0 / 2048.0, 4095.5 / 4096.0, -3.3e4):
                    s = chosen("crowd", r, k, a, g)
                    if s is None:
                        continue
                    taken += 1
                    limbs = crowd_limbs(r, s, k, a, g)
                    err = [np.abs(hi / s[0] + lo / (s[0] * s[1]) - law(r, ch, k, a, g))
                           for ch, (hi, lo) in enumerate(limbs)]
                    assert (err[0] + np.max(err[1:], axis=0) <= 2.0 ** -20.999 * np.abs(law(r, 0, k, a, g))).all()
                    for i in range(2):
                        assert partial_sums(limbs[0][i], [l[i] for l in limbs[1:]]) < 2 ** 24, (r, a, g, k)
    assert taken > 300


def test_sums_of_walls_and_exits_fit_and_no_entry_is_further_off_than_fp32s(chosen):
    """The second limb is any integer up to 65504, in two tables."""
    taken = 0
    assert all(chosen("cells", r, 1.0, -0.5, -1.0, -0.5) for r in range(12, 41))  # the default laws
    for r in (12, 28, 40, 44):
        for k0, a0, k1, a1 in ((1.0, -0.5, -1.0, -0.5), (1.0, 0.0, -1.0, 0.0), (0.51, 0.0, 0.0, 0.0),
                               (2049.0 / 2048.0, 0.01, -0.75, -0.01), (1.0, -0.2, -1.5, -0.4), (0.0, 0.0, 0.3, 0.1)):
            s = chosen("cells", r, k0, a0, k1, a1)
            if s is None:
                continue
            taken += 1
            two = []
            for k, a in ((k0, a0), (k1, a1)):
                v = law(r, 0, k, a)
                hi = limb16(v * s[0])
                lo = np.rint((v * s[0] - hi) * s[1])
                most = limb16(lo)
                for limb in (hi, most, lo - most):
                    assert (limb == limb.astype(np.float16).astype(np.float64)).all()
                assert (np.abs(hi / s[0] + lo / (s[0] * s[1]) - v) <= 2.0 ** -24 * np.abs(v)).all()
                two.append((hi, most, np.abs(lo - most)))
            for i in range(2):  # a partial sum has some of the small tables' entries
                extra = i * np.maximum(two[0][2], two[1][2])
                up = (np.maximum(np.maximum(two[0][i], two[1][i]), 0) + extra).sum()
                down = (np.maximum(np.maximum(-two[0][i], -two[1][i]), 0) + extra).sum()
                assert max(up, down) < 2 ** 24, (r, k0, a0, k1, a1)
    assert taken > 10


@pytest.mark.parametrize("r", range(1, MAXR + 1))
def test_operand_addresses_stay_in_their_buffers(r):
    C, P, K = chunks(r), pitch(r), 2 * r + 16
    assert P % 16 == 0 and 16 * C >= 2 * r + 8
    rows, stage = TH + 2 * r, (2 * r + 31) * 512
    # A: row group b (16 lattice rows down), window row ky, chunk c, half h, 8 x 16 bytes
    assert (15 * 16 + K - 1) * P + (C - 1) * 32 + 16 + 128 <= rows * P
    # B: window row ky starts at j = 2r + 15 - ky; 32 groups (su row, limb) of 256 bytes
    assert 0 <= (K - 1 - (K - 1)) and (K - 1) * 512 + 31 * 256 + 256 <= stage
    plane = -(-rows * P // 128) * 128
    assert 256 + plane + 2 * stage <= SMEM


@pytest.mark.parametrize("r", [1, 3, 5, 9])
def test_tile_product_equals_the_window_sums(chosen, r):
    """One tile through the tables and addresses, in integers, against the
    direct window sum of the same fixed-point law."""
    rng = np.random.default_rng(r)
    C, K, J = chunks(r), 2 * r + 16, 2 * r + 31
    s0, s1 = chosen("crowd", r, 1.0, -0.5, 0.5)
    width = TW - 8 + 16 * C
    for ch in (0, 3):
        v = law(r, ch)
        limbs = split(v, s0, s1)
        plane = rng.integers(-1, 2, (TH + 2 * r, width)).astype(np.float64)
        tab = np.zeros((C, J, 2, 8, 16))
        for j in range(J):
            for nx in range(8):
                for k in range(16 * C):
                    dy, dx = j - r - 15, nx - k + r
                    if abs(dx) <= r and abs(dy) <= r:
                        for limb in range(2):
                            tab[k // 16, j, limb, nx, k % 16] = limbs[limb][dy + r, dx + r]
        for by, bx in ((0, 0), (7, 3), (15, 7)):
            D = np.zeros((16, 2, 8))
            for c in range(C):
                for ky in range(K):
                    a = plane[16 * by + ky, 8 * bx + 16 * c: 8 * bx + 16 * c + 16]
                    for ny in range(16):
                        D[ny] += tab[c, ny - ky + 2 * r + 15] @ a
            for ny, nx in ((0, 0), (5, 7), (15, 2)):
                win = plane[16 * by + ny: 16 * by + ny + 2 * r + 1, 8 * bx + nx: 8 * bx + nx + 2 * r + 1]
                for limb in range(2):
                    assert D[ny, limb, nx] == (win * limbs[limb][::-1, ::-1]).sum()
