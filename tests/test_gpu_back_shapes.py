"""Single-slice back projections in every launch shape, against the oracle.

Plain back projections choose their block by the number of 16 x 16 tiles (one or
two per SM, three, more) and of views (8, 64); 152 SMs.  Images are long or large
enough for each rule and the bins few, so that the oracle's matrix stays small.
Subset updates take staged bins (two, three or more candidates, or bins read in
place where they are too many to stage) or runs, by the bins per pixel, the views
and the tiles; a batch's members take theirs by another rule, with the same bits.

Tolerance per element: the FP32 sum of at most n nonnegative terms is within
n 2^-24 of its exact value, n the largest column count of the oracle's matrix; the
weights are within 2e-5 of the exact ones, plus 2e-6 of the image's largest value
(the projection tolerance of the parity tests).  Updates: relative L2 1e-5.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from cases import rel_l2
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


def _update_problem(nx, ny, per_subset, fineness, subsets=2):
    # at 30 bins a pixel and 5 views a field of 260 bins leaves three pixels 0.025 mm of a subset's
    # rays, whose FP32 rounding alone moves the image by 1.2e-5: there the field covers the image
    wide = fineness == 30.0 and per_subset == 5
    bins = int(1.43 * max(nx, ny) * fineness) + 1
    if not wide:
        bins = min(bins, 260)
    geom = Geometry(nx, ny, per_subset * subsets, bins, pixel_mm=2.0, bin_mm=2.0 / fineness)
    g = np.random.default_rng(2).poisson(4.0, geom.n_rays).astype(np.float32)
    return geom, g


# bins per pixel 1 and 0.77: two candidates; 1.6 and 2: three; 2.2, 4 and 30: more; 60: in place.
# Views either side of the rule's lines (48 tiles and more: another line)
@pytest.mark.parametrize("nx,ny,per_subset,fineness", [
    (40, 37, 7, 1.0), (40, 37, 33, 1.0), (40, 37, 10, 0.77), (40, 37, 11, 0.77), (40, 37, 35, 0.3),
    (40, 37, 8, 1.6), (40, 37, 9, 1.6), (40, 37, 10, 1.6), (40, 37, 16, 2.0), (40, 37, 20, 2.0), (40, 37, 5, 2.2), (40, 37, 6, 2.2), (40, 37, 3, 4.0),
    (40, 37, 18, 4.0), (40, 37, 5, 30.0), (40, 37, 6, 30.0), (40, 37, 5, 60.0), (40, 37, 2, 60.0), (40, 37, 6, 60.0),
    (120, 90, 12, 1.6), (120, 90, 13, 1.6), (120, 90, 8, 4.0), (120, 90, 9, 4.0)])
def test_update_shapes(nx, ny, per_subset, fineness):
    from paper_2106_03172_gb300 import petvr as pv
    geom, g = _update_problem(nx, ny, per_subset, fineness)
    prob = em.build_problem(geom, g.astype(np.float64), 0.5, 2, 0.01)
    plan = pv.Plan(geom, 2)
    gp = pv.Problem(plan, _cuda(g), None, 0.5, 0.01)
    f0 = np.random.default_rng(3).uniform(0.5, 1.5, (prob.N, 1)).astype(np.float32).astype(np.float64)
    for method, alg in (("osem", None), ("svrem", em.SVREM(prob, f0, 0.7, 1)), ("saga", em.SAGA(prob, f0, 1.0))):
        img = _cuda(f0)
        state = pv.State(gp, method, img)
        f = f0
        for t in (1, 0, 1):
            state.epoch([t], alpha=0.7 if method == "svrem" else 1.0)
            f = em.osem_step(prob, f, t) if alg is None else alg.step(t)
            assert rel_l2(_host(img), f) <= 1e-5, (method, t)


# 9, 48, 160, 300, 620 and 520 tiles: images that are one tile high but for the first two
@pytest.mark.parametrize("mode", ["phases", "dataflow"])
@pytest.mark.parametrize("nx,ny,per_subset,fineness", [
    (40, 37, 6, 4.0), (120, 90, 9, 4.0), (120, 90, 9, 60.0), (120, 90, 13, 1.6), (120, 90, 11, 0.77), (2560, 7, 12, 1.0),
    (2560, 7, 13, 1.0), (4800, 5, 17, 1.0), (4800, 5, 14, 1.0), (4800, 5, 11, 0.6), (9920, 5, 6, 1.0), (9920, 5, 9, 0.6),
    (9920, 5, 9, 2.2), (8320, 5, 6, 1.0), (8320, 5, 7, 1.0), (8320, 5, 9, 0.6), (8320, 5, 9, 2.2), (8320, 5, 9, 4.0)])
def test_update_shapes_have_the_same_bits(mode, nx, ny, per_subset, fineness):
    """A state's own updates (runs or staged bins by its rule) and a batch's."""
    from paper_2106_03172_gb300 import petvr as pv
    geom, g = _update_problem(nx, ny, per_subset, fineness)
    plan = pv.Plan(geom, 2)
    gp = pv.Problem(plan, _cuda(g), None, 0.5, 0.01)
    f0 = np.random.default_rng(3).uniform(0.5, 1.5, nx * ny)
    for method, alpha in (("osem", 1.0), ("saga", 1.0), ("svrem", 0.7)):
        alone, batched = _cuda(f0), _cuda(f0)
        pv.State(gp, method, alone).epoch([1, 0, 1], alpha=alpha)
        state = pv.State(gp, method, batched)
        batch = pv.Batch([state])
        batch.set_mode(mode)
        batch.epoch([[1, 0, 1]], [alpha], [1])
        batch.sync()
        assert torch.equal(alone, batched), method


# launches whose subset is given by the host: the warm start's updates and SEM's statistic of all views
@pytest.mark.parametrize("nx,ny,per_subset,fineness", [
    (40, 37, 7, 1.0), (40, 37, 11, 0.77), (40, 37, 6, 4.0), (120, 90, 13, 1.6), (120, 90, 9, 4.0)])
def test_warm_start_and_sem_shapes(nx, ny, per_subset, fineness):
    from paper_2106_03172_gb300 import petvr as pv
    geom, g = _update_problem(nx, ny, per_subset, fineness)
    prob = em.build_problem(geom, g.astype(np.float64), 0.5, 2, 0.01)
    plan = pv.Plan(geom, 2)
    gp = pv.Problem(plan, _cuda(g), None, 0.5, 0.01)
    img = torch.empty(prob.N, device="cuda")
    pv.pet_warm_start(gp.handle, img)
    f0 = _host(img).reshape(-1, 1)
    assert rel_l2(f0, prob.initial_image()) <= 1e-5
    pv.State(gp, "sem", img).epoch([1], alpha=0.5)
    assert rel_l2(_host(img), em.SEM(prob, f0, schedule=lambda k: 0.5).step(1)) <= 1e-5
