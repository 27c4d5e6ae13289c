"""The plan's back-projection constants, from the built library (CPU only).

* tile_bins: the staged bins and most candidates per view that the other test of the
  staged bins emulates are the library's own;
* stack_candidates: the lanes and rounds a slice stack gives a view's candidate bins
  hold all of them, counted with the kernels' float32 expressions.
"""
import ctypes
import math
import random

import numpy as np
import pytest

import test_back_tile_bins as staged

f32 = np.float32


def _lib():
    from paper_2106_03172_gb300 import build
    return ctypes.CDLL(build.build())


def _call(name, pixel, binw, nb, nx, ny):
    fn = getattr(_lib(), name)
    fn.restype = None
    a, b = ctypes.c_int(), ctypes.c_int()
    fn(ctypes.c_double(pixel), ctypes.c_double(binw), nb, nx, ny, ctypes.byref(a), ctypes.byref(b))
    return a.value, b.value


def test_staged_bins_are_the_emulated_ones():
    rng = random.Random(1)
    for _ in range(300):
        nx, ny = (int(math.exp(rng.uniform(0, 9.7))) for _ in range(2))
        pixel, binw = rng.uniform(0.5, 4.0), math.exp(rng.uniform(-7, 3))
        nb = int(math.exp(rng.uniform(0, 14.5)))
        bw, cand = _call("_ZN5petvr9tile_binsEddiiiRiS0_", pixel, binw, nb, nx, ny)
        assert bw == staged._tile_bins(pixel, binw, nb, nx, ny)
        eps = 1e-3 + 4e-7 * (nb + nx + ny)
        if nb < 1 << 20 and pixel / binw <= staged.STAGE_BINS:
            assert cand == max(2, math.floor(1.41422 * pixel / binw + 2 * eps) + 1)
        else:
            assert bw > staged.STAGE_BINS


@pytest.mark.parametrize("nx,ny,na,nb,pixel,binw", [
    (24, 24, 18, 35, 2.0, 1.4), (64, 60, 84, 138, 2.0, 0.08), (64, 60, 31, 500, 2.0, 0.02), (200, 180, 12, 300, 2.0, 2.0),
    (48, 48, 64, 40, 2.0, 5.0), (16, 16, 40, 900, 2.0, 0.05), (500, 40, 24, 700, 1.0, 0.7), (33, 31, 1024, 47, 2.0, 2.0)])
def test_stack_lanes_hold_every_candidate(nx, ny, na, nb, pixel, binw):
    cands, rounds = _call("_ZN5petvr16stack_candidatesEddiiiRiS0_", pixel, binw, nb, nx, ny)
    assert 1 <= cands <= 32 and (rounds == 1 or cands == 32)
    for i in range(0, na, max(1, na // 64)):
        col, cm, cn, n_minor, n_major = staged._view(nx, ny, na, nb, pixel, binw, i)
        du, inv_k = f32(-cn / cm), f32(cm * pixel / binw)
        uc0 = f32(-0.5 * (nb - 1) * binw / (cm * pixel) + (0.5 if n_minor % 2 else 0.0))
        kc = (np.arange(n_major) - 0.5 * n_major).astype(f32)[:, None]
        m = (np.arange(n_minor) - (n_minor >> 1)).astype(f32)[None, :]
        base = staged._fma(kc, du, uc0)
        e1 = (((m - max(du, f32(0))) - base - f32(1e-3)) * inv_k).astype(f32)
        e2 = (((m + f32(1) - min(du, f32(0))) - base + f32(1e-3)) * inv_k).astype(f32)
        jlo = np.maximum(0, np.ceil(np.minimum(e1, e2)).astype(np.int64))
        jhi = np.minimum(nb - 1, np.floor(np.maximum(e1, e2)).astype(np.int64))
        assert (jhi - jlo + 1).max() <= cands * rounds, i
