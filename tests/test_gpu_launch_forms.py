"""Which launch form a handle uses (one, two or four steps per launch; chains of launches per 3-D box),
and the calls that report, change and restore it."""
import numpy as np
import pytest

from paper_1710_10569_gb300 import workloads as W

pytestmark = pytest.mark.gpu

F64, F32, F16 = W.STORAGE_F64, W.STORAGE_F32, W.STORAGE_F16DEV
P, D, A, WET = W.WALL_PERIODIC, W.WALL_DIRICHLET, W.WALL_ADIABATIC, W.WALL_WET
LAYOUTS = {"periodic": (P, P, P, P), "layer": (P, P, D, D), "box": (D, A, A, D), "cavity": (D, D, A, A), "sides": (A, D, P, P)}


@pytest.fixture(scope="module")
def clb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1710_10569_gb300 import clb as c
    return c


# Odd rows of two windows, which take two steps per launch: bitwise equal to one.
@pytest.mark.parametrize("layout", sorted(LAYOUTS))
def test_two_steps_on_odd_rows_of_two_windows(clb, layout):
    for rates in (1.0, 1.2):
        prob = W.random_problem(113, 10091, seed=3, storage=F32, walls=LAYOUTS[layout], moving=rates != 1.0)
        prob.params.update(s_3=rates, s_4=rates, lambda2=rates)
        got = []
        for steps in (2, 1):
            lat = clb.Lattice.from_problem(prob)
            if steps == 1:
                lat.set_steps_per_launch(1)
            assert lat.steps_per_launch() == steps
            lat.step(5)
            got.append(lat.populations())
            lat.close()
        for a, b in zip(*got):
            assert np.isfinite(a).all() and np.array_equal(a, b)


def step_us(handle, n=320):
    """Time of a step, the least of five runs of n steps each, after as many untimed ones."""
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    handle.step(n)
    best = 1e30
    for _ in range(5):
        torch.cuda.synchronize()
        e0.record()
        handle.step(n)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 1e3 / n)
    return best


# The sizes at which test_gpu_two_steps compares several steps per launch with one: the default arm
# does take them, and an explicit shape does not.
@pytest.mark.parametrize("layout", sorted(LAYOUTS))
def test_sizes_compared_elsewhere_take_several_steps(clb, layout):
    for nx, ny in [(53, 19001), (60, 17003), (59, 17200), (118, 8701), (1001, 1003), (2048, 517), (30011, 41)]:
        lat = clb.Lattice(nx, ny, W.default_params(storage=F32, wall=LAYOUTS[layout]))
        assert lat.steps_per_launch() == 2, (nx, ny)
        lat.set_launch(128, 1, 2)
        assert lat.steps_per_launch() == 1, (nx, ny)
        lat.close()
    # (wide rows between x walls and most odd ones take four steps from more nodes on: see the next test)
    for nx, ny in ([(4096, 101)] if LAYOUTS[layout][0] == P else []) + [(112, 3601), (55, 7301)]:
        h = clb.Thermal(nx, ny, W.default_params(storage=F32 if (nx + ny) % 2 == 0 else F16, wall=LAYOUTS[layout]))
        assert h.steps_per_launch() == 4, (nx, ny)
        h.set_steps_per_launch(1)
        assert h.steps_per_launch() == 1
        h.set_steps_per_launch(0)
        assert h.steps_per_launch() == 4
        with pytest.raises(clb.CLBError):
            h.set_steps_per_launch(2)
        h.close()


def thermal(clb, nx, ny, storage, walls, lambda2):
    p = W.default_params(nu=0.05, kappa=0.03, storage=storage, wall=LAYOUTS[walls], T_wall=(0.3, -0.2, 0.5, -0.4), lambda2=lambda2,
                         u_wall=((0, 0.02), (0, 0.01), (0.02, 0.03), (0.01, -0.02)))
    rng = np.random.default_rng(nx)
    h = clb.Thermal(nx, ny, p)
    h.init(*(a * (rng.random((ny, nx)) - 0.5) for a in (1.0, 0.2, 0.2)))
    return h


@pytest.mark.parametrize("storage", [F32, F16])
@pytest.mark.parametrize("walls", sorted(LAYOUTS))
@pytest.mark.parametrize("lambda2", [1.0, 1.3])
def test_four_thermal_steps_on_odd_rows(clb, walls, lambda2, storage):
    """Odd rows of many windows, of a size from which every layout takes four steps per launch: bitwise
    equal to one step per launch."""
    got = []
    for steps in (4, 1):
        h = thermal(clb, 2451, 1701, storage, walls, lambda2)
        if steps == 1:
            h.set_steps_per_launch(1)
        assert h.steps_per_launch() == steps
        h.step(9)
        got.append(h.populations())
        h.close()
    assert np.isfinite(got[0]).all() and np.array_equal(*got)


# Four steps per launch between x walls took up to 1.18 times as long as one on lattices of 0.4 to 2 million
# nodes (5% for the timing and the sizes next to the line).
@pytest.mark.parametrize("storage", [F32, F16])
@pytest.mark.parametrize("lambda2", [1.0, 1.3])
@pytest.mark.parametrize("shape", [(640, 640), (1024, 1024), (1500, 1000), (100, 6000), (2048, 2048)], ids=lambda s: "%dx%d" % s)
def test_default_thermal_form_is_not_the_slower_one(clb, shape, lambda2, storage):
    h = thermal(clb, *shape, storage, "cavity", lambda2)
    us = step_us(h)
    h.set_steps_per_launch(1)
    assert us <= 1.05 * step_us(h)
    h.close()


# The same on odd rows and shapes next to the line (8%: the estimates are good to 5 and 10%).
@pytest.mark.parametrize("shape,walls,lambda2,storage",
                         [((727, 1495), "layer", 1.3, F16), ((2971, 220), "layer", 1.3, F16), ((2371, 177), "periodic", 1.0, F16),
                          ((2869, 537), "layer", 1.3, F32), ((377, 1648), "layer", 1.3, F32), ((489, 2588), "cavity", 1.0, F16),
                          ((1761, 539), "periodic", 1.3, F16), ((802, 829), "cavity", 1.0, F32), ((162, 5968), "cavity", 1.3, F16)])
def test_default_thermal_form_on_odd_rows(clb, shape, walls, lambda2, storage):
    h = thermal(clb, *shape, storage, walls, lambda2)
    us = step_us(h)
    h.set_steps_per_launch(1)
    assert us <= 1.08 * step_us(h)
    h.close()


MIXED = [(512, 512), (61, 70), (333, 129), (64, 64), (2, 3), (120, 900)]


@pytest.mark.parametrize("rates", [1.0, 1.2])
@pytest.mark.parametrize("sizes", [MIXED, [(700, 700)], [(60, 35)] * 230, [(1025, 31)] * 15 + [(59, 300)] * 9],
                         ids=["mixed", "one", "many", "wide"])
def test_batches_compared_elsewhere_take_two_steps(clb, sizes, rates):
    probs = [W.random_problem(nx, ny, seed=k, storage=F32) for k, (nx, ny) in enumerate(sizes)]
    for p in probs:
        p.params.update(s_3=rates, s_4=rates, lambda2=rates)
    b = clb.Batch(probs)
    if sizes is MIXED and rates != 1.0:  # too few nodes for general rates: see the next test
        assert b.steps_per_launch() == 1
        b.close()
        return
    assert b.steps_per_launch() == 2
    b.set_tile(*b.launch()["tile"])  # as it is: nothing changes
    assert b.steps_per_launch() == 2
    b.set_tile(64, 2, 2)
    assert b.steps_per_launch() == 1
    b.set_steps_per_launch(0)
    assert b.steps_per_launch() == 2 and b.launch()["tile"] == (64, 2, 2)
    b.set_steps_per_launch(1)
    assert b.steps_per_launch() == 1
    with pytest.raises(clb.CLBError):
        b.set_steps_per_launch(3)
    b.close()


def test_mixed_batch_with_general_rates(clb):
    """Two steps per launch bitwise equal to one on a batch of mixed sizes large enough to take them."""
    sizes = MIXED + [(601, 599)]
    probs = [W.random_problem(nx, ny, seed=k, storage=F32, walls=sorted(LAYOUTS.values())[k % 5], moving=True)
             for k, (nx, ny) in enumerate(sizes)]
    for p in probs:
        p.params.update(s_3=1.2, s_4=1.2, lambda2=1.2)
        if min(p.nx, p.ny) < 4:
            p.T, p.ux, p.uy = 0.01 * p.T, 0.01 * p.ux, 0.01 * p.uy
    got = []
    for steps in (2, 1):
        b = clb.Batch(probs)
        if steps == 1:
            b.set_steps_per_launch(1)
        assert b.steps_per_launch() == steps
        b.step(39)
        got.append([b.fields(k) for k in range(len(probs))])
        b.close()
    for k, (x, y) in enumerate(zip(*got)):
        for a, c in zip(x, y):
            assert np.isfinite(a).all() and np.array_equal(a, c), k


def test_forms_not_taken(clb):
    for nx, ny, storage, walls in [(1200, 1200, F64, LAYOUTS["layer"]), (1200, 1200, F16, LAYOUTS["layer"]), (64, 64, F32, LAYOUTS["layer"]),
                                   (1200, 1200, F32, (P, P, WET, WET)), (1200, 1200, F32, (WET, WET, P, P))]:
        lat = clb.Lattice(nx, ny, W.default_params(storage=storage, wall=walls))
        assert lat.steps_per_launch() == 1
        lat.set_steps_per_launch(0)
        assert lat.steps_per_launch() == 1
        lat.close()


def test_lattice_form_survives_calls_that_change_nothing(clb):
    prob = W.random_problem(1100, 1000, seed=3, storage=F32, walls=LAYOUTS["cavity"])
    lat = clb.Lattice.from_problem(prob)
    lat.set_launch()
    lat.set_launch(*lat.launch())
    lat.set_pipeline(*lat.pipeline())
    lat.set_pipeline(0)
    assert lat.steps_per_launch() == 2
    lat.step(35)
    ref = lat.fields()
    shape = lat.launch()
    lat.set_launch(128, 2, 2)
    assert lat.steps_per_launch() == 1 and lat.launch() == (128, 2, 2)
    lat.set_steps_per_launch(0)
    assert lat.steps_per_launch() == 2
    lat.set_launch(*shape)
    lat.set_steps_per_launch(1)
    lat.init_fields(*prob.fields())
    lat.step(35)
    assert lat.steps_per_launch() == 1
    for x, y in zip(lat.fields(), ref):
        assert np.array_equal(x, y)
    with pytest.raises(clb.CLBError):
        lat.set_steps_per_launch(2)
    lat.close()


def test_3d_batch_form_survives_the_present_tile(clb):
    b = clb.Batch3D([W.random_problem3d(24 + k, 22, 20, seed=k, storage=F32) for k in range(8)])
    assert b.chains()
    b.set_tile(*b.launch()["block"])
    assert b.chains()
    b.step(33)
    ref = [b.fields(k) for k in range(8)]
    b.set_tile(64, 2)
    assert not b.chains()
    for chains in (True, False):
        b.set_chains(chains)
        assert b.chains() == chains
        for k in range(8):
            b.init_fields(k, *b.problems[k].fields())
        b.step(33)
        for k in range(8):
            for x, y in zip(b.fields(k), ref[k]):
                assert np.array_equal(x, y), (chains, k)
    b.close()


# Batches whose buffers stay in L2 and whose rows fill the warps of one step per launch: two steps per
# launch took up to 1.5 times as long there (120 of 64 x 64: 14.4 against 9.6 us per step). The default is no
# slower than one step per launch, whichever it takes (5% for the timing).
@pytest.mark.parametrize("walls", ["cavity", "layer"])
@pytest.mark.parametrize("rates", [1.0, 1.2])
@pytest.mark.parametrize("size", [(120, 64, 64), (50, 125, 90), (8, 256, 256), (32, 128, 128), (12, 200, 200), (300, 40, 40)],
                         ids=lambda s: "%dx%dx%d" % s)
def test_default_batch_form_is_not_the_slower_one(clb, size, walls, rates):
    count, nx, ny = size
    probs = [W.random_problem(nx, ny, seed=k, storage=F32, walls=LAYOUTS[walls]) for k in range(count)]
    for p in probs:
        p.params.update(s_3=rates, s_4=rates, lambda2=rates)
        p.T, p.ux, p.uy = 0.1 * p.T, 0.1 * p.ux, 0.1 * p.uy
    b = clb.Batch(probs)
    assert b.steps_per_launch() == (2 if count in (12, 300) else 1)
    us = step_us(b)
    b.set_steps_per_launch(1)
    assert us <= 1.05 * step_us(b)
    b.close()


# Lattices just above the size at which two steps per launch begin: the default is not the slower form.
@pytest.mark.parametrize("rates", [1.0, 1.2])
@pytest.mark.parametrize("size,walls,steps", [((1024, 1024), "cavity", 1), ((1024, 1024), "layer", 2), ((2048, 512), "cavity", 2),
                                              ((60, 17003), "cavity", 2), ((1100, 1000), "cavity", 2), ((17003, 60), "cavity", 2),
                                              ((128, 9019), "cavity", 1), ((121, 9002), "layer", 1), ((121, 9002), "cavity", 1),
                                              ((305, 3700), "cavity", 2)])
def test_default_lattice_form_is_not_the_slower_one(clb, size, walls, steps, rates):
    prob = W.random_problem(*size, seed=1, storage=F32, walls=LAYOUTS[walls])
    prob.params.update(s_3=rates, s_4=rates, lambda2=rates)
    prob.T, prob.ux, prob.uy = 0.1 * prob.T, 0.1 * prob.ux, 0.1 * prob.uy
    lat = clb.Lattice.from_problem(prob)
    assert lat.steps_per_launch() == steps
    us = step_us(lat)
    lat.set_steps_per_launch(1)
    assert us <= 1.05 * step_us(lat)
    lat.close()


# Large FP32 lattices: blocks of two warps side by side only where the rows fill them (they took up to 1.11
# times as long elsewhere).
@pytest.mark.parametrize("size", [(200, 4000), (600, 700), (1000, 700), (701, 699), (1024, 950)], ids=lambda s: "%dx%d" % s)
def test_default_block_is_not_the_slower_one(clb, size):
    prob = W.random_problem(*size, seed=1, storage=F32, walls=LAYOUTS["layer"])
    prob.params.update(s_3=1.0, s_4=1.0, lambda2=1.0)
    prob.T, prob.ux, prob.uy = 0.1 * prob.T, 0.1 * prob.ux, 0.1 * prob.uy
    lat = clb.Lattice.from_problem(prob)
    assert lat.launch() == ((64, 1, 2) if size[0] % 128 == 0 else (32, 2, 2))
    us = step_us(lat)
    for shape in ((64, 1, 2), (32, 2, 2)):
        lat.set_launch(*shape)
        assert us <= 1.04 * step_us(lat), shape
    lat.close()


# The autotuner times the default it replaces, and two steps per launch at any width: what it picks is no
# slower than the untuned handle (it lacked the default blocks, and two steps on narrow lattices).
@pytest.mark.parametrize("size,storage", [((256, 256), F64), ((60, 17003), F32), ((90, 12000), F32), ((701, 699), F32), ((640, 640), F16),
                                          ((2048, 600), F32)], ids=str)
def test_tuned_shape_is_not_the_slower_one(clb, size, storage):
    prob = W.random_problem(*size, seed=1, storage=storage, walls=LAYOUTS["layer"])
    prob.T, prob.ux, prob.uy = 0.1 * prob.T, 0.1 * prob.ux, 0.1 * prob.uy
    lat = clb.Lattice.from_problem(prob)
    steps = lat.steps_per_launch()
    us = step_us(lat)
    shape = lat.autotune()
    assert lat.launch() == shape and lat.steps_per_launch() == steps
    assert step_us(lat) <= 1.04 * us
    lat.close()


# The tuner's choice for a lattice with wet walls, which the two-step kernel does not know, is not that of a
# lattice of the same size without them; nor is that of the other kind of rates.
def test_tuned_shapes_are_kept_by_walls_and_rates(clb):
    nx, ny = 2048, 604
    wet = clb.Lattice(nx, ny, W.default_params(storage=F32, wall=(P, P, WET, WET)))
    wet.autotune()
    wet.close()
    lat = clb.Lattice(nx, ny, W.default_params(storage=F32, wall=LAYOUTS["layer"]))
    assert lat.steps_per_launch() == 2
    shape = lat.autotune()
    assert lat.steps_per_launch() == 2
    lat.close()
    again = clb.Lattice(nx, ny, W.default_params(storage=F32, wall=LAYOUTS["layer"]))
    assert again.launch() == shape and again.steps_per_launch() == 2
    again.close()
    general = clb.Lattice(nx, ny, W.default_params(storage=F32, wall=LAYOUTS["layer"], s_3=1.2))
    assert general.launch() == (64, 1, 2) and general.steps_per_launch() == 2
    general.close()


# A lattice initialised again goes to the buffer the others are in: after an odd number of steps the graphs
# of chains stay as they are (they were made again, which took tens of steps' time, for every such call).
def test_reinitialised_box_keeps_the_graphs(clb):
    import time
    import torch
    probs = [W.random_problem3d(16, 15, 14, seed=k, storage=F32) for k in range(48)]
    for p in probs:
        p.ux, p.uy, p.uz, p.T = 0.1 * p.ux, 0.1 * p.uy, 0.1 * p.uz, 0.1 * p.T
    b = clb.Batch3D(probs)
    b.set_chains(True)
    b.step(65)

    def step_ms():
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        b.step(32)
        torch.cuda.synchronize()
        return (time.perf_counter() - t0) * 1e3

    before = min(step_ms() for _ in range(5))
    after = []
    for _ in range(5):
        b.step(1)  # the state changes buffers
        b.init_fields(7, *probs[7].fields())
        after.append(step_ms())
    assert min(after) <= 2 * before
    lat = clb.Lattice3D.from_problem(probs[7])
    lat.step(32)
    for x, y in zip(lat.populations(), b.member(7).populations()):
        assert np.isfinite(x).all() and np.array_equal(x, y)
    lat.close()
    b.close()


# Chains of launches per box: with steps left over, from either buffer and after one lattice was
# initialised again, bitwise the lattices alone.
@pytest.mark.parametrize("storage", [F64, F32, F16])
def test_chains_equal_single_boxes(clb, storage):
    shapes = [(9, 7, 5), (33, 20, 17), (5, 4, 3)]
    probs = [W.random_problem3d(*s, seed=k, storage=storage, moving=k == 1) for k, s in enumerate(shapes)]
    for p in probs:  # thin extents: gentle fields
        p.ux, p.uy, p.uz, p.T = 0.2 * p.ux, 0.2 * p.uy, 0.2 * p.uz, 0.2 * p.T
    b = clb.Batch3D(probs)
    b.set_chains(True)
    b.step(37)
    b.init_fields(1, *probs[1].fields())
    b.step(41)
    for k, p in enumerate(probs):
        lat = clb.Lattice3D.from_problem(p)
        lat.step(41 if k == 1 else 78)
        for x, y in zip(lat.populations(), b.member(k).populations()):
            assert np.isfinite(x).all() and np.array_equal(x, y), k
        lat.close()
    b.close()


# Chains were taken for every batch: 1,000 boxes of edge 8 stepped in 293 us instead of 121. The default is
# not the slower form (8% for the estimate).
@pytest.mark.parametrize("count,edge,storage", [(12, 8, F32), (6, 10, F32), (5, 14, F32), (16, 6, F16), (256, 8, F32), (1000, 8, F32), (48, 12, F32), (512, 12, F32), (800, 14, F32),
                                                (256, 16, F32), (12, 32, F32), (256, 8, F16), (100, 12, F16), (256, 8, F64)])
def test_default_3d_batch_form_is_not_the_slower_one(clb, count, edge, storage):
    b = clb.Batch3D([W.rayleigh_benard3d(edge, edge, edge, Ra=2e3, storage=storage)] * count)
    b.step(320)
    us = step_us(b, 128)
    chains = b.chains()
    b.set_chains(not chains)
    assert us <= 1.08 * step_us(b, 128), chains
    b.close()


# The first steps of a batch do not pay for graphs of thousands of launches (20 ms for 256 boxes, whose
# steps take 0.1 ms).
def test_first_steps_of_a_3d_batch(clb):
    import time
    import torch
    prob = W.rayleigh_benard3d(16, 16, 16, Ra=2e3, storage=F32)

    def first_ms(chains):
        b = clb.Batch3D([prob] * 256)
        if not chains:
            b.set_chains(False)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        b.step(64)
        torch.cuda.synchronize()
        ms = (time.perf_counter() - t0) * 1e3
        assert b.chains() == chains
        b.close()
        return ms

    first_ms(False)
    assert min(first_ms(True) for _ in range(3)) <= 1.3 * min(first_ms(False) for _ in range(3))


# The same for uneven batches near 400,000 nodes, some of odd widths.
@pytest.mark.parametrize("rates", [1.0, 1.2])
@pytest.mark.parametrize("sizes", [[(300, 300), (500, 400), (129, 1000), (64, 90)], [(513, 385), (301, 700)], [(257, 300)] * 6,
                                   [(91, 120)] * 40, [(180, 180)] * 13, [(101, 101)] * 40], ids=["uneven", "odd", "257", "91", "180", "101"])
def test_default_form_of_uneven_batches_is_not_the_slower_one(clb, sizes, rates):
    probs = [W.random_problem(nx, ny, seed=k, storage=F32, walls=sorted(LAYOUTS.values())[k % 5]) for k, (nx, ny) in enumerate(sizes)]
    for p in probs:
        p.params.update(s_3=rates, s_4=rates, lambda2=rates)
        p.T, p.ux, p.uy = 0.1 * p.T, 0.1 * p.ux, 0.1 * p.uy
    b = clb.Batch(probs)
    us = step_us(b)
    b.set_steps_per_launch(1)
    assert us <= 1.05 * step_us(b)
    b.close()


# Mid-sized FP32 lattices: blocks of four warps side by side where the rows fill them and the lattice is one
# round of resident warps (two rows of one warp took up to 1.2 times as long there).
@pytest.mark.parametrize("walls", ["cavity", "layer"])
@pytest.mark.parametrize("size,shape", [((232, 905), (128, 1, 2)), ((250, 800), (128, 1, 2)), ((500, 400), (128, 1, 2)), ((964, 192), (128, 1, 2)),
                                        ((408, 506), (32, 2, 2)), ((232, 1300), (32, 2, 2)), ((513, 385), (32, 2, 2)),
                                        ((300, 700), (32, 2, 2)), ((128, 1500), (32, 2, 2))])
def test_default_block_of_mid_sized_lattices(clb, size, shape, walls):
    prob = W.random_problem(*size, seed=1, storage=F32, walls=LAYOUTS[walls])
    prob.params.update(s_3=1.0, s_4=1.0, lambda2=1.0)
    prob.T, prob.ux, prob.uy = 0.1 * prob.T, 0.1 * prob.ux, 0.1 * prob.uy
    lat = clb.Lattice.from_problem(prob)
    assert lat.launch() == shape
    us = step_us(lat, 640)
    for other in ((32, 2, 2), (128, 1, 2)):
        if size != (232, 1300) or walls == "cavity":
            lat.set_launch(*other)
            assert us <= 1.04 * step_us(lat, 640), other
    lat.close()
