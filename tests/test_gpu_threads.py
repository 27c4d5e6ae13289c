"""Host threads that run different plans at the same time.

Two threads issue the updates of one method directly (no graphs: every update
launches) on a 64^2 plan and on a 256^2 plan, whose launches ask for different
amounts of shared memory from the same kernel.  No call may be refused, and both
images have the bits of the same updates issued by one thread.
"""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = r"""
import sys, threading
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
from paper_2106_03172_gb300 import petvr as pv
from paper_2106_03172_gb300.phantoms import Geometry

EPOCHS = 150

def setup(n, views, bins, seed):
    rng = np.random.default_rng(seed)
    plan = pv.Plan(Geometry(n, n, views, bins), 6)
    g = torch.from_numpy(rng.poisson(5.0, views * bins).astype(np.float32)).cuda()
    prob = pv.Problem(plan, g, None, 0.5, 0.01)
    img = torch.from_numpy(rng.uniform(0.5, 1.5, n * n).astype(np.float32)).cuda()
    torch.cuda.synchronize()
    return pv.State(prob, sys.argv[2], img), img, torch.cuda.Stream()

def work(job, errors):
    state, img, stream = job
    try:
        for e in range(EPOCHS):
            state.epoch([(e + i) % 6 for i in range(6)], alpha=0.5, stream=stream)
        stream.synchronize()
    except Exception as ex:
        errors.append(repr(ex))

PLANS = [(64, 60, 91, 1), (256, 36, 367, 2)]
images = []
for threads in (False, True):
    jobs, errors = [setup(*p) for p in PLANS], []
    if threads:
        ts = [threading.Thread(target=work, args=(j, errors)) for j in jobs]
        [t.start() for t in ts]
        [t.join() for t in ts]
    else:
        [work(j, errors) for j in jobs]
    assert not errors, errors
    images.append([j[1].cpu().numpy() for j in jobs])
for a, b in zip(*images):
    np.testing.assert_array_equal(a, b)
"""


@pytest.mark.parametrize("method", ["osem", "saga"])
def test_two_threads_two_plan_sizes(method):
    env = dict(os.environ, PETVR_NO_GRAPHS="1")
    res = subprocess.run([sys.executable, "-c", CODE, ROOT, method], capture_output=True, text=True, env=env, cwd=ROOT,
                         timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
