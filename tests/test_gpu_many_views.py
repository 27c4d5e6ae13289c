"""Volume back projections with as many views as a plan takes (1024).

The slice-stack and multi-ring kernels keep the views of their subset in shared
memory; with one subset, and in all-view passes (pet_back of -1, SEM's first
statistic), those are all views of the plan.

Tolerance of a back projection, per element: the FP32 sum of at most n
nonnegative terms is within n 2^-24 of its exact value, n the largest column
count of the oracle's matrix, and the weights within 2e-5 (the projection
tolerance of the parity tests).  SEM's first update: relative L2 1e-5.
"""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from cases import rel_l2
from oracle import em
from paper_2106_03172_gb300.phantoms import Geometry

pytestmark = pytest.mark.gpu

VIEWS = 1024


def _rings(nz):
    return Geometry(9, 8, VIEWS, 11, nz=nz, n_rings=2, ring_mm=3.0, radius_mm=30.0, slice_mm=2.0)


GEOMETRIES = {
    "stack5": Geometry(9, 8, VIEWS, 11, nz=5), "stack20": Geometry(9, 8, VIEWS, 11, nz=20),
    "stack47": Geometry(9, 8, VIEWS, 11, nz=47), "ring3": _rings(3), "ring6": _rings(6), "ring10": _rings(10),
}


@functools.lru_cache(maxsize=None)
def _case(name, n_subsets):
    geom = GEOMETRIES[name]
    inner = 1 if geom.n_rings else geom.nz
    lines = geom.n_angles * geom.n_bins * max(1, geom.n_rings) ** 2
    g = np.random.default_rng(5).poisson(4.0, (lines, inner)).astype(np.float64)
    return geom, em.build_problem(geom, g, 0.5, n_subsets, 0.01)


def _cuda(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float32).ravel()).cuda()


def _host(t):
    torch.cuda.synchronize()
    return t.double().cpu().numpy()


def _close(got, want, prob):
    rtol = np.diff(prob.A.tocsc().indptr).max() * 2.0 ** -24 + 2e-5
    assert np.all(np.abs(got - want) <= rtol * np.abs(want)), np.max(np.abs(got - want) / np.abs(want))


@pytest.mark.parametrize("n_subsets", [1, 3])
@pytest.mark.parametrize("name", list(GEOMETRIES))
def test_back_projection_of_all_views(name, n_subsets):
    from paper_2106_03172_gb300 import petvr as pv
    geom, prob = _case(name, n_subsets)
    plan = pv.Plan(geom, n_subsets)
    y = np.random.default_rng(6).uniform(0.5, 1.5, (prob.M, prob.nz)).astype(np.float32)
    img = torch.empty(prob.N * prob.nz, device="cuda")
    pv.pet_back(plan.handle, _cuda(y), -1, img)
    _close(_host(img).reshape(-1, prob.nz), prob.A.T @ y.astype(np.float64), prob)
    sens = torch.empty(prob.N, device="cuda")
    for t in range(n_subsets):
        pv.pet_plan_sensitivity(plan.handle, t, sens)
        _close(_host(sens), prob.sens_t[t][:, 0], prob)


@pytest.mark.parametrize("name", list(GEOMETRIES))
def test_sem_statistic_of_all_views(name):
    from paper_2106_03172_gb300 import petvr as pv
    geom, prob = _case(name, 1)
    plan = pv.Plan(geom, 1)
    gp = pv.Problem(plan, _cuda(prob.g), None, 0.5, prob.beta)
    f0 = np.random.default_rng(7).uniform(0.5, 1.5, (prob.N, prob.nz)).astype(np.float32).astype(np.float64)
    img = _cuda(f0)
    pv.State(gp, "sem", img).epoch([0], alpha=0.5)
    want = em.SEM(prob, f0, schedule=lambda k: 0.5).step(0)
    assert rel_l2(_host(img), want) <= 1e-5
