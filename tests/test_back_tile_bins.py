"""The bins a back-projection tile stages, emulated in float32 on the CPU.

A tile stages, per view, `bw` bins from the smallest first candidate of its
corners on, and every pixel reads its candidate bins from there unchecked.
For every tile and view of several geometries (square, odd, ragged, bins finer
and coarser than pixels) this checks that each pixel's candidates lie inside
the staged range, and that they include every ray that meets the pixel (from
the FP64 positions of all rays).  The expressions are the kernels' own, with
fused multiply-adds as FP64 products rounded once to FP32.
"""
import math

import numpy as np
import pytest

f32 = np.float32
TILE, STAGE_BINS = 16, 1024


def _fma(a, b, c):
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(f32)


def _snap(x):
    return float(round(x)) if abs(x - round(x)) < 1e-12 else x


def _tile_bins(pixel, binw, nb, nx, ny):
    ratio = pixel / binw
    eps = 1e-3 + 4e-7 * (nb + nx + ny)
    if nb >= 1 << 20 or ratio > STAGE_BINS:
        return STAGE_BINS + 1
    return min(STAGE_BINS + 1, math.ceil((TILE - 1) * 1.41422 * ratio)
               + max(2, math.floor(1.41422 * ratio + 2 * eps) + 1) + 4)


def _view(nx, ny, na, nb, pixel, binw, i):
    c, s = _snap(math.cos(i * math.pi / na)), _snap(math.sin(i * math.pi / na))
    col = abs(c) < abs(s)
    cm, cn = (s, c) if col else (c, s)
    n_minor, n_major = (ny, nx) if col else (nx, ny)
    return col, cm, cn, n_minor, n_major


@pytest.mark.parametrize("nx,ny,na,nb,pixel,binw", [
    (64, 64, 60, 91, 2.0, 2.0), (37, 29, 23, 41, 1.7, 1.3), (40, 53, 31, 200, 2.0, 0.5), (33, 48, 24, 20, 2.0, 5.0),
    (256, 256, 12, 367, 2.0, 2.0), (201, 147, 19, 250, 1.7, 1.4), (512, 512, 7, 733, 2.0, 2.0), (16, 16, 9, 450, 2.0, 0.1),
    (1, 1, 5, 3, 2.0, 2.0), (1000, 17, 5, 1500, 1.0, 1.0)])
def test_candidates_are_staged_and_complete(nx, ny, na, nb, pixel, binw):
    bw = _tile_bins(pixel, binw, nb, nx, ny)
    assert bw <= STAGE_BINS
    for i in range(na):
        col, cm, cn, n_minor, n_major = _view(nx, ny, na, nb, pixel, binw, i)
        du64 = -cn / cm
        du, du_lo = f32(du64), f32(du64 - float(f32(du64)))
        inv_k = f32(cm * pixel / binw)
        adu = abs(du)
        eps = f32(f32(1e-3) + f32(4e-7) * f32(nb + nx + ny))
        off = f32(0.5 if n_minor % 2 else 0.0)
        first = f32(-adu if inv_k > 0 else 1.0)
        cst = f32(_fma(f32(first - off), inv_k, f32(0.5) * f32(nb - 1)) + f32(f32(1.0) - eps))
        nc = int(math.floor(_fma(f32(1.0) + adu, abs(inv_k), f32(2.0) * eps))) + 1
        cand = max(2, math.floor(1.41422 * pixel / binw + 2e-3 + 8e-7 * (nb + nx + ny)) + 1)
        assert nc <= cand
        read = cand if cand <= 3 else nc
        k_off = f32(1.0 if du < 0 else 0.0)
        # every pixel's first candidate
        m = (np.arange(n_minor) - (n_minor >> 1)).astype(f32)
        kc = (np.arange(n_major) - 0.5 * n_major).astype(f32) + k_off
        band = _fma(-(kc * du).astype(f32), inv_k, cst)
        j = np.floor(_fma(m[:, None], inv_k, band[None, :]).astype(np.float64)).astype(np.int64)
        # the tiles' staged ranges (pixels of a ragged tile past the image read their bins too)
        for tm in range(0, n_minor, TILE):
            for tk in range(0, n_major, TILE):
                m0 = f32(tm - (n_minor >> 1))
                k0 = f32(f32(tk) - f32(0.5) * f32(n_major) + k_off)
                ma = min(f32(m0 * inv_k), f32(f32(m0 + f32(15)) * inv_k))
                slope = f32(f32(-du) * inv_k)
                p = min(f32(slope * k0), f32(slope * f32(k0 + f32(15))))
                j0 = int(math.floor(f32(f32(ma + p) + cst))) - 1
                part = j[tm:tm + TILE, tk:tk + TILE]
                assert part.min() >= j0 and part.max() + read <= j0 + bw, (i, tm, tk)
        # every ray that meets the pixel is a candidate (the exact offsets, all rays)
        u = ((np.arange(nb) - 0.5 * (nb - 1)) * binw) / (cm * pixel) + float(off)
        for ki in np.unique(np.linspace(0, n_major - 1, 6).astype(int)):
            x = u[None, :] + (ki - 0.5 * n_major + float(k_off)) * du64 - m[:, None].astype(np.float64)
            hit = (x > -abs(du64) + 1e-9) & (x < 1.0 - 1e-9)
            jj = np.arange(nb)[None, :]
            inside = (jj >= j[:, ki][:, None]) & (jj < j[:, ki][:, None] + nc)
            assert not np.any(hit & ~inside), (i, ki)
