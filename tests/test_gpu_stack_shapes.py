"""Slice stacks of more than 16 slices where their lists take another turn.

Back projection: more than 32 candidate bins a view (several rounds of lanes); forward:
band chunks longer than one list holds (images longer than 512 pixels).  Tolerances
per element against the oracle: the FP32 sum of at most n nonnegative terms is within
n 2^-24 of its exact value, n the longest row or column of the oracle's matrix; the
weights are within 2e-5 of the exact ones, plus 2e-6 of the largest value (the
projection tolerance of the parity tests).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import em
from paper_2106_03172_gb300.phantoms import Geometry

pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float32).ravel()).cuda()


def _close(got, want, terms):
    got = got.double().cpu().numpy().reshape(want.shape)
    tol = (terms * 2.0 ** -24 + 2e-5) * np.abs(want) + 2e-6 * np.abs(want).max()
    assert np.all(np.abs(got - want) <= tol), (np.abs(got - want) / tol).max()


@pytest.mark.parametrize("nx,ny,views,bins,pixel,binw,nz", [
    (14, 12, 9, 500, 2.0, 0.08, 20),        # 25 bins a pixel: 36 candidates, two rounds
    (14, 12, 9, 900, 2.0, 0.03, 47),        # 67 bins a pixel: 95 candidates, three rounds
    (520, 8, 10, 40, 2.0, 9.0, 20),         # chunks of 130 bands
])
def test_stack_projections(nx, ny, views, bins, pixel, binw, nz):
    from paper_2106_03172_gb300 import petvr as pv
    geom = Geometry(nx, ny, views, bins, pixel_mm=pixel, bin_mm=binw, nz=nz)
    prob = em.build_problem(geom, np.ones((views * bins, nz)), 0.5, 2, 0.01)
    plan = pv.Plan(geom, 2)
    rng = np.random.default_rng(3)
    y = rng.uniform(0.5, 1.5, (prob.M, nz)).astype(np.float32)
    f = rng.uniform(0.5, 1.5, (prob.N, nz)).astype(np.float32)
    img, sino = torch.empty(prob.N * nz, device="cuda"), torch.empty(prob.M * nz, device="cuda")
    column = np.diff(prob.A.tocsc().indptr).max()
    row = np.diff(prob.A.tocsr().indptr).max()
    pv.pet_back(plan.handle, _cuda(y), -1, img)
    pv.pet_forward(plan.handle, _cuda(f), None, 0.0, -1, sino)
    _close(img, prob.A.T @ y.astype(np.float64), column)
    _close(sino, prob.A @ f.astype(np.float64), row)
    rows = prob.subsets[1]
    sub = torch.empty(len(rows) * nz, device="cuda")
    pv.pet_back(plan.handle, _cuda(y[rows]), 1, img)
    pv.pet_forward(plan.handle, _cuda(f), None, 0.0, 1, sub)
    _close(img, prob.At[1].T @ y[rows].astype(np.float64), column)
    _close(sub, prob.At[1] @ f.astype(np.float64), row)
