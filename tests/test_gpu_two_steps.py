"""The kernels that take several steps per launch (large lattices) against one step per launch.

The FP32 kernel that takes two steps per launch against the one-step kernel, which
an explicit launch shape selects: every population bitwise, over windows and rows of every kind (one
and several windows per row, odd rows, a last window of one column, rows that end in mid-window,
segments of every remainder), every wall layout, fixed and moving, both collision forms, and even
and odd numbers of steps."""
import numpy as np
import pytest

from paper_1710_10569_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P, D, A = W.WALL_PERIODIC, W.WALL_DIRICHLET, W.WALL_ADIABATIC
LAYOUTS = {"periodic": (P, P, P, P), "layer": (P, P, D, D), "box": (D, A, A, D), "cavity": (D, D, A, A), "sides": (A, D, P, P)}


@pytest.fixture(scope="module")
def clb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1710_10569_gb300 import clb as c
    return c


@pytest.mark.parametrize("shape,steps", [((53, 19001), 2), ((60, 17003), 7), ((59, 17200), 4), ((118, 8701), 3), ((121, 9002), 5),
                                         ((1001, 1003), 7), ((2048, 517), 34), ((30011, 41), 6)],
                         ids=lambda v: f"{v[0]}x{v[1]}" if isinstance(v, tuple) else f"{v}")
@pytest.mark.parametrize("layout", sorted(LAYOUTS))
def test_two_steps_per_launch_equal_one(clb, layout, shape, steps):
    one = (shape[0] + steps) % 2 == 0
    prob = W.random_problem(*shape, seed=shape[0] + steps, storage=W.STORAGE_F32, walls=LAYOUTS[layout], moving=not one)
    if one:
        prob.params.update(s_3=1.0, s_4=1.0, lambda2=1.0)
    got = []
    for shape_set in (False, True):
        lat = clb.Lattice.from_problem(prob)
        if shape_set:
            lat.set_launch(128, 1, 2)
        lat.step(steps)
        got.append(lat.populations())
        assert lat.steps == steps
        lat.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.array_equal(a, b)


# The autotuner's choice is kept by storage form and size: a lattice of that size with wet walls, which the
# two-step kernel does not know, steps as under an explicit shape whatever another lattice's tuning chose.
def test_wet_walls_after_tuning_the_same_size(clb):
    prob = W.random_problem(2048, 600, seed=5, storage=W.STORAGE_F32, walls=LAYOUTS["layer"])
    lat = clb.Lattice.from_problem(prob)
    lat.autotune()
    lat.close()
    prob.params.update(wall=(P, P, W.WALL_WET, W.WALL_WET))
    got = []
    for shape_set in (False, True):
        lat = clb.Lattice.from_problem(prob)
        if shape_set:
            lat.set_launch(128, 1, 2)
        lat.step(6)
        got.append(lat.populations())
        lat.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.array_equal(a, b)


# The temperature equation alone: four steps per launch against the same number of calls of one step.
@pytest.mark.parametrize("shape", [(8193, 49), (4096, 101), (1121, 358), (112, 3601), (55, 7301), (703, 702)],
                         ids=lambda v: f"{v[0]}x{v[1]}")
@pytest.mark.parametrize("layout", sorted(LAYOUTS))
def test_four_thermal_steps_per_launch_equal_one(clb, layout, shape):
    nx, ny = shape
    storage = W.STORAGE_F32 if (nx + ny) % 2 == 0 else W.STORAGE_F16DEV
    rng = np.random.default_rng(nx)
    p = W.default_params(nu=0.05, kappa=0.03, storage=storage, wall=LAYOUTS[layout], T_wall=(0.3, -0.2, 0.5, -0.4),
                         lambda2=1.0 if ny % 3 else 1.3, u_wall=((0, 0.02), (0, 0.01), (0.02, 0.03), (0.01, -0.02)))
    T, ux, uy = rng.uniform(-0.5, 0.5, (ny, nx)), rng.uniform(-0.1, 0.1, (ny, nx)), rng.uniform(-0.1, 0.1, (ny, nx))
    got = []
    for calls in ([9], [1] * 9):
        h = clb.Thermal(nx, ny, p)
        h.init(T, ux, uy)
        for n in calls:
            h.step(n)
        got.append(h.populations())
        h.close()
    assert np.isfinite(got[0]).all() and np.array_equal(*got)


# Batches: pairs of steps in one launch against one step per launch (an explicit tile shape).
@pytest.mark.parametrize("sizes", [[(512, 512), (61, 70), (333, 129), (64, 64), (2, 3), (120, 900)], [(700, 700)],
                                   [(60, 35)] * 230, [(1025, 31)] * 15 + [(59, 300)] * 9], ids=["mixed", "one", "many", "wide"])
@pytest.mark.parametrize("rates", [1.0, 1.2])
def test_two_steps_per_batched_launch_equal_one(clb, sizes, rates):
    layouts = list(LAYOUTS.values())
    probs = [W.random_problem(nx, ny, seed=k, storage=W.STORAGE_F32, walls=layouts[k % len(layouts)], moving=rates != 1.0)
             for k, (nx, ny) in enumerate(sizes)]
    for p in probs:
        p.params.update(s_3=rates, s_4=rates, lambda2=rates)
        if min(p.nx, p.ny) < 4:
            p.T, p.ux, p.uy = 0.01 * p.T, 0.01 * p.ux, 0.01 * p.uy
    got = []
    for tile in (None, (64, 2, 2)):
        b = clb.Batch(probs)
        if tile:
            b.set_tile(*tile)
        b.step(39)
        got.append([b.fields(k) for k in range(len(probs))])
        assert set(b.status()[2]) == {39}
        b.close()
    for k, (x, y) in enumerate(zip(*got)):
        for a, b in zip(x, y):
            assert np.isfinite(a).all() and np.array_equal(a, b), k
