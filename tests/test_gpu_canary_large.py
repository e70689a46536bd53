"""The guard regions and NaN padding of test_gpu_canary around lattices large enough for the kernels that
small ones do not reach: two steps per launch (FP32, a million nodes) and the split step (FP16)."""
import numpy as np
import pytest

from paper_1710_10569_gb300 import workloads as W
from test_gpu_canary import GUARD, PATTERN, clb, guarded_lattice, padding_views  # noqa: F401 (clb: the fixture)

pytestmark = pytest.mark.gpu

F32, F16 = W.STORAGE_F32, W.STORAGE_F16DEV
P, D, A, WET = W.WALL_PERIODIC, W.WALL_DIRICHLET, W.WALL_ADIABATIC, W.WALL_WET
CASES = [(F32, (1011, 1013), (P, P, P, P)), (F32, (1011, 1013), (D, A, A, D)), (F32, (59, 17201), (P, P, D, D)), (F32, (113, 10090), (A, D, D, A)), (F32, (53, 20011), (D, D, A, A)),
         (F32, (20011, 53), (A, D, P, P)), (F16, (801, 603), (D, D, A, A)), (F16, (801, 603), (WET, WET, WET, WET)),
         (F16, (641, 640), (P, P, P, P)), (F16, (130001, 4), (P, P, D, D))]


@pytest.mark.parametrize("storage,shape,walls", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_large_lattices_leave_guards_and_padding(clb, storage, shape, walls):  # noqa: F811
    import torch
    prob = W.random_problem(*shape, seed=5, storage=storage, walls=walls, moving=WET not in walls)
    scale = 0.02 if min(shape) < 8 else 0.3
    prob.T, prob.ux, prob.uy = scale * prob.T, scale * prob.ux, scale * prob.uy
    lat = guarded_lattice(clb, prob)
    assert lat.steps_per_launch() == (2 if storage == F32 else 1)
    views, _ = padding_views(clb, lat, storage)
    for v in views:
        v.fill_(float("nan"))
    before = [v.clone() for v in views]
    lat.step(37)  # a graph, pairs of steps and an odd step
    lat.run(0.0, 20, 10)
    got = lat.fields()
    torch.cuda.synchronize()
    g = lat._mem
    assert bool((g[:GUARD] == PATTERN).all()) and bool((g[GUARD + lat.footprint:] == PATTERN).all())
    for v, b in zip(views, before):
        assert torch.equal(v.contiguous().view(-1).view(torch.uint8), b.contiguous().view(-1).view(torch.uint8)), "padding was written"
    lat.close()
    ref = clb.Batch([prob])
    ref.set_steps_per_launch(1)
    ref.step(57)
    for a, b in zip(got, ref.fields(0)):
        assert np.isfinite(a).all() and np.array_equal(a, b)
    ref.close()
