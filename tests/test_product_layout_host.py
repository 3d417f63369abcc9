"""The crowded lattice's field product, on CPU: its limb tables, operand
addresses and sums, restated in NumPy from their description (sfm_product.cu),
give the window sums of the class-table law for every radius class, and no
entry, sum or address leaves its range."""
import math

import numpy as np
import pytest

TW, TH, MAXR, SMEM = 64, 256, 44, 227 * 1024


def chunks(r):
    return (2 * r + 8 + 15) // 16


def pitch(r):
    return (TW - 8 + 16 * chunks(r)) * 2


def scales(r, k=1.0, a=-0.5, g=0.5):
    v = np.abs(law(r, 0, k, a, g))
    n = (2 * r + 1) ** 2 + 60
    s0 = 2.0 ** math.floor(math.log2(4096.0 / (v.max() * max(1.0, abs(g)))))
    while v.sum() * (1 + abs(g)) * s0 + 2 * n > 2 ** 24 - 1:
        s0 /= 2
    s1 = 4096.0
    while n * 2 * s1 / 2 > 2 ** 24 - 1:
        s1 /= 2
    return s0, s1


def split(v, s0, s1):
    hi = np.where(np.abs(v * s0) > 2048, (v * s0).astype(np.float16).astype(np.float64), np.rint(v * s0))
    return hi, np.rint((v * s0 - hi) * s1).astype(np.float16).astype(np.float64)


def law(r, ch, k=1.0, a=-0.5, g=0.5):
    ax = np.arange(-r, r + 1, dtype=np.float64)
    dy, dx = np.meshgrid(ax, ax, indexing="ij")
    d = np.hypot(dx, dy)
    d[r, r] = 1.0
    q = math.sqrt(0.5)
    v = k * d ** a * (1.0, g * dx / d, g * dy / d, g * q * (dx + dy) / d, g * q * (dy - dx) / d)[ch]
    v[r, r] = 0.0
    return v


@pytest.mark.parametrize("r", [1, 2, 3, 7, 12, 20, 31, 32, 36, 37, 40, 44])
def test_limbs_are_exact_and_their_sums_fit(r):
    s0, s1 = scales(r)
    hi_all = lo_all = np.zeros((2 * r + 1, 2 * r + 1))
    for ch in range(5):
        v = law(r, ch)
        hi, lo = split(v, s0, s1)
        for limb in (hi, lo):
            assert np.abs(limb).max() <= 4096 and (limb == np.rint(limb)).all()
        # a su is in the occupancy plane and at most one heading plane
        if ch == 0:
            hi0, lo0 = np.abs(hi), np.abs(lo)
        else:
            hi_all = np.maximum(hi_all, np.abs(hi))
            lo_all = np.maximum(lo_all, np.abs(lo))
        # what the second limb's rounding leaves: 2^-23 of the law's largest
        # entry and less, and far below its smallest
        err = np.abs(hi / s0 + lo / (s0 * s1) - v).max()
        assert err <= 2.0 ** -23 and 2 * err <= 5.0e-6 * np.abs(law(r, 0))[0, 0]
    assert (hi0 + hi_all).sum() < 2 ** 24 and (lo0 + lo_all).sum() < 2 ** 24   # exact in FP32


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
def test_tile_product_equals_the_window_sums(r):
    """One tile through the tables and addresses, in integers, against the
    direct window sum of the same fixed-point law."""
    rng = np.random.default_rng(r)
    C, K, J = chunks(r), 2 * r + 16, 2 * r + 31
    s0, s1 = scales(r)
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
