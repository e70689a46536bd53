"""The FP16 step of large lattices, split into a kernel for the interior warps and one for the edge warps
(rows next to y walls, columns next to x walls or holding a ragged row end) that run side by side,
against the batched step, one kernel that holds every path: bitwise the same fields. Sizes from the
first lattice that is split on: odd and even rows, rows of one warp column and of thousands, few rows
and tens of thousands; every wall layout, fixed, moving and wet, both kinds of rates, 1, 2 and 4 nodes
per thread."""
import numpy as np
import pytest

from paper_1710_10569_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P, D, A, WET = W.WALL_PERIODIC, W.WALL_DIRICHLET, W.WALL_ADIABATIC, W.WALL_WET
LAYOUTS = {"periodic": (P, P, P, P), "layer": (P, P, D, D), "box": (D, A, A, D), "cavity": (D, D, A, A), "sides": (A, D, P, P),
           "wet_y": (P, P, WET, WET), "wet_x": (WET, WET, P, P), "wet_box": (WET, WET, WET, WET)}
# of 400,000 nodes or more: ragged rows, rows of whole warp columns, one warp column, few rows, many rows
SHAPES = [(801, 603), (640, 640), (1283, 313), (133337, 3), (7, 60001), (131, 3067), (256, 1600)]


@pytest.fixture(scope="module")
def clb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1710_10569_gb300 import clb as c
    return c


def problem(shape, layout, rates, moving):
    w = LAYOUTS[layout]
    prob = W.random_problem(*shape, seed=shape[0] % 97, storage=W.STORAGE_F16DEV, walls=w, moving=moving and WET not in w)
    if rates == 1.0:
        prob.params.update(s_3=1.0, s_4=1.0, lambda2=1.0)
    scale = 0.02 if min(shape) < 8 else 0.3  # thin extents: gentle fields
    prob.T, prob.ux, prob.uy = scale * prob.T, scale * prob.ux, scale * prob.uy
    return prob


@pytest.mark.parametrize("layout", sorted(LAYOUTS))
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[0]}x{s[1]}")
def test_split_step_equals_the_batched_step(clb, shape, layout):
    assert shape[0] * shape[1] >= 400000
    for rates in (1.0, 1.2):
        prob = problem(shape, layout, rates, moving=rates != 1.0)
        b = clb.Batch([prob])
        b.step(5)
        ref = b.fields(0)
        b.close()
        assert all(np.isfinite(x).all() for x in ref)
        for npt in (0, 4, 2, 1):
            lat = clb.Lattice.from_problem(prob)
            if npt:
                lat.set_launch(32 if npt == 4 else 128, 2 if npt != 2 else 1, npt)
            lat.step(5)
            for x, y in zip(lat.fields(), ref):
                assert np.array_equal(x, y), (rates, npt)
            lat.close()


@pytest.mark.parametrize("layout", ["cavity", "wet_box"])
def test_split_step_in_graphs(clb, layout):
    """The fork and join of the two kernels inside a captured chunk of steps, and the diagnostics after it."""
    prob = problem((801, 603), layout, 1.2, moving=False)
    b = clb.Batch([prob])
    lat = clb.Lattice.from_problem(prob)
    for n in (37, 64):
        b.step(n)
        lat.step(n)
        nu, er = b.diagnostics()
        assert lat.check(prob.nu_axis) == (nu[0], er[0])
    for x, y in zip(lat.fields(), b.fields(0)):
        assert np.isfinite(x).all() and np.array_equal(x, y)
    lat.close()
    b.close()
