"""Single-slice back projections in every launch shape, against the oracle.

Plain back projections choose their block by the number of 16 x 16 tiles (one or
two per SM, three, more) and of views (8, 64); 152 SMs.  Images are long or large
enough for each rule and the bins few, so that the oracle's matrix stays small.

Tolerance per element: the FP32 sum of at most n nonnegative terms is within
n 2^-24 of its exact value, n the largest column count of the oracle's matrix; the
weights are within 2e-5 of the exact ones, plus 2e-6 of the image's largest value
(the projection tolerance of the parity tests).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import em
from paper_2106_03172_gb300.phantoms import Geometry

pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float32).ravel()).cuda()


def _host(t):
    torch.cuda.synchronize()
    return t.double().cpu().numpy()


def _close(got, want, prob):
    rtol = np.diff(prob.A.tocsc().indptr).max() * 2.0 ** -24 + 2e-5
    tol = rtol * np.abs(want) + 2e-6 * np.abs(want).max()
    assert np.all(np.abs(got - want) <= tol), (np.abs(got - want) / tol).max()


# tiles: 9, 9, 160, 312, 480, 480 (views at the rules' edges: 8, 64, a pass of 16 or 32)
@pytest.mark.parametrize("nx,ny,views,bins", [
    (41, 37, 64, 31), (41, 37, 65, 31), (41, 37, 97, 31), (160, 250, 17, 29), (160, 250, 65, 29), (200, 370, 16, 23),
    (200, 370, 17, 23), (241, 465, 8, 19), (241, 465, 9, 19), (241, 465, 1, 19)])
def test_plain_back_projection_shapes(nx, ny, views, bins):
    from paper_2106_03172_gb300 import petvr as pv
    geom = Geometry(nx, ny, views, bins, pixel_mm=2.0, bin_mm=5.3)
    prob = em.build_problem(geom, np.ones(views * bins), 0.5, 1, 0.01)
    plan = pv.Plan(geom, 1)
    y = np.random.default_rng(4).uniform(0.5, 1.5, prob.M).astype(np.float32)
    img = torch.empty(prob.N, device="cuda")
    pv.pet_back(plan.handle, _cuda(y), -1, img)
    _close(_host(img), prob.A.T @ y.astype(np.float64), prob)
