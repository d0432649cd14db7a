"""The multi-step kernel of small lattices against the one-step kernels (taken
while kernel timing is on): the same trajectory bit for bit, for every kind of
0D boundary, marching order, storage type, first layers of one to five chunks
of 256 cells, batches, per-step 0D input, and launches split at the step limit;
with a cluster of blocks per instance and with one grid over all instances.
"""
import numpy as np
import pytest

from workloads import batch, configs, geometry
from workloads.spec import BC_VELOCITY, Instance

pytestmark = pytest.mark.gpu


def _box():
    return Instance(node=geometry.closed_box(17, 9, 13), tau=0.7, name="box")


def _lv(radius, length):
    return batch.lv_tube_instance(batch.draw_params(np.random.default_rng(0), 1)[0], radius, length)


def _order(inst, order):
    for b in inst.boundaries:
        if len(b.params) == 4:
            b.params = list(b.params) + [float(order)]
    return inst


CASES = {
    "velocity": lambda: [configs.rigid_tube()],
    "lv": lambda: [configs.lv_tube(period=300)],
    "lv_order2": lambda: [_order(configs.lv_tube(period=300), 2)],
    "lv_order4": lambda: [_order(configs.lv_tube(period=300), 4)],
    "lv_along_x": lambda: [configs.lv_tube_x(31)],
    "pressure": lambda: [configs.pressure_tube(15, 15, 24, 5.2, 0.8, 2e-3, 0.0)],
    "box": lambda: [_box()],
    "two_chunks": lambda: [configs.rigid_tube(27, 27, 20, radius=10.3)],
    "five_chunks": lambda: [configs.rigid_tube(41, 41, 12, radius=18.3)],
    "batch": lambda: [configs.lv_tube(period=300), _box(), _lv(6.3, 41), configs.rigid_tube(16, 16, 24, radius=5.0)],
}
# sizes at which the rule takes one grid: a few blocks, all of them, instances of
# different sizes and relaxation times, no boundary at all
GRID = {
    "lv": lambda: [_lv(8.0, 131)],
    "lv_order4": lambda: [_order(_lv(13.0, 203), 4)],
    "velocity": lambda: [configs.rigid_tube(31, 31, 170, radius=11.4)],
    "pressure": lambda: [configs.pressure_tube(30, 30, 150, 12.6, 0.8, 2e-3, 0.0)],
    "two_passes": lambda: [_lv(16.2, 310)],
    "box": lambda: [Instance(node=geometry.closed_box(61, 47, 53), tau=0.7, name="box")],
    "uneven": lambda: [_lv(6.0, 128), Instance(node=geometry.closed_box(31, 17, 53), tau=0.7, name="box"),
                       _lv(12.0, 200), configs.rigid_tube()],
}
CASES.update({"grid_" + k: v for k, v in GRID.items()})


def _pair(insts, precision, steps):
    from paper_2112_05258_gb300 import Lattice
    a, b = (Lattice(insts, precision=precision) for _ in range(2))
    for q, inst in enumerate(insts):
        f = configs.random_populations(inst, seed=q, amp=2e-3)
        a.init_populations(q, f)
        b.init_populations(q, f)
    b.set_kernel_timing(True)
    for n in steps:
        a.step(n)
        b.step(n)
    a.sync()
    b.sync()
    return a, b


def _same(a, b, insts):
    for q, inst in enumerate(insts):
        assert np.array_equal(a.populations(q), b.populations(q))
        assert np.array_equal(a.waves(q), b.waves(q))
        for k in range(len(inst.boundaries)):
            assert np.array_equal(a.state_0d(q, k), b.state_0d(q, k))


@pytest.mark.parametrize("precision", ["f32", "f16"])
@pytest.mark.parametrize("name", list(CASES))
def test_multi_step_kernel_equals_one_step_kernels(name, precision):
    insts = CASES[name]()
    a, b = _pair(insts, precision, (1, 2, 350, 61))
    assert a.info().steps_per_launch > 0      # the case takes the multi-step kernel
    _same(a, b, insts)
    a.step(7)                                 # and goes on after a switch of the path
    b.set_kernel_timing(False)
    b.step(7)
    _same(a, b, insts)


@pytest.mark.parametrize("inst", [lambda: configs.lv_tube(period=300), lambda: configs.rigid_tube()])
def test_multi_step_kernel_fp64_and_long_calls(inst):
    insts = [inst()]
    a, b = _pair(insts, "f64", (4 * 300 + 1, 3001))   # the second call goes past the steps of one launch
    n = a.info().steps_per_launch
    a.step(n + 5)
    b.step(n + 5)
    _same(a, b, insts)


@pytest.mark.parametrize("inst", [lambda: configs.rigid_tube(), GRID["velocity"]])
def test_step_io_of_a_velocity_inlet_equals_per_step_calls(inst):
    import torch
    from paper_2112_05258_gb300 import Lattice
    inst = inst()
    inst = inst[0] if isinstance(inst, list) else inst
    n = 90
    omega = torch.tensor(2 * np.pi / (1000.0 + 5.0 * np.arange(n)).reshape(n, 1)).pin_memory()
    rows = torch.zeros((n, 16), dtype=torch.float64, pin_memory=True)
    want = torch.zeros((n, 16), dtype=torch.float64, pin_memory=True)
    a, b = (Lattice([inst], precision="f32") for _ in range(2))
    assert inst.boundaries[0].kind == BC_VELOCITY and a.info().steps_per_launch > 0
    a.step_io(0, 0, n, omega.data_ptr(), 1, rows.data_ptr())
    a.sync()
    b.set_kernel_timing(True)
    for k in range(n):
        b.set_0d_params(0, 0, omega[k].numpy())
        b.step(1)
        b.state_0d_async(0, want[k].data_ptr())
    b.sync()
    assert np.array_equal(rows.numpy(), want.numpy())
    _same(a, b, [inst])


def test_large_or_elastic_lattices_keep_the_step_graphs():
    from paper_2112_05258_gb300 import Lattice
    for inst in (configs.ib_tube(), _lv(13.0, 800)):
        assert Lattice([inst]).info().steps_per_launch == 0


WIDE = {
    "lv": lambda: _lv(13.0, 770),
    "lv_order4": lambda: _order(_lv(12.2, 881), 4),
    "velocity": lambda: configs.rigid_tube(31, 31, 1003, radius=11.4),
    "pressure": lambda: configs.pressure_tube(30, 30, 818, 12.6, 0.8, 2e-3, 0.0),
}


@pytest.mark.parametrize("precision", ["f32", "bf16"])
@pytest.mark.parametrize("name", list(WIDE))
def test_one_launch_boundary_equals_two_kernels(name, precision):
    # a tube too large for the multi-step kernel takes its boundary work in one
    # launch of clusters (started while stream-collide ends); many copies in one
    # lattice have too many boundary blocks for it and take the two kernels
    from paper_2112_05258_gb300 import Lattice
    inst = WIDE[name]()
    copies = 40
    one, many = Lattice([inst], precision=precision), Lattice([inst] * copies, precision=precision)
    assert one.info().steps_per_launch == 0 and one.info().launches_per_step == 2
    assert many.info().launches_per_step == 3
    f = configs.random_populations(inst, seed=5, amp=2e-3)
    one.init_populations(0, f)
    many.init_populations(7, f)
    for n in (1, 130, 71):
        one.step(n)
        many.step(n)
    assert np.array_equal(one.populations(0), many.populations(7))
    assert np.array_equal(one.waves(0), many.waves(7))
    for k in range(2):
        assert np.array_equal(one.state_0d(0, k), many.state_0d(7, k))


@pytest.mark.parametrize("name,bc,cols", [("lv", 1, 4), ("velocity", 0, 1)])
def test_step_io_in_the_one_launch_boundary(name, bc, cols):
    import torch
    from paper_2112_05258_gb300 import Lattice
    inst = WIDE[name]()
    n = 150
    base = np.array(inst.boundaries[bc].params[:cols], dtype=np.float64)
    par = torch.from_numpy(np.tile(base, (n, 1)) * (1.0 + 0.2 * np.sin(np.arange(n) / 9.0))[:, None]).pin_memory()
    par[:, 1:] = torch.from_numpy(base[1:])
    rows = torch.zeros((n, 16), dtype=torch.float64, pin_memory=True)
    want = torch.zeros((n, 16), dtype=torch.float64, pin_memory=True)
    a, b = (Lattice([inst], precision="f32") for _ in range(2))
    a.step(3)
    b.step(3)
    a.step_io(0, bc, n, par.data_ptr(), cols, rows.data_ptr())
    a.sync()
    for k in range(n):
        b.set_0d_params(0, bc, par[k].numpy())
        b.step(1)
        b.state_0d_async(0, want[k].data_ptr())
    b.sync()
    assert np.array_equal(rows.numpy(), want.numpy())
    assert np.array_equal(rows.numpy()[:, 0], np.arange(4, 154))
    assert np.array_equal(a.populations(0), b.populations(0))


PARTS = {
    "two": lambda: [_lv(13.0, 450), _lv(12.2, 443)],
    "one_launch": lambda: [Instance(node=geometry.closed_box(61, 47, 53), tau=0.7, name="box"), _lv(13.0, 203),
                           _lv(6.3, 41), configs.rigid_tube(31, 31, 170, radius=11.4), _lv(12.2, 301)],
    "two_kernels": lambda: [_lv(20.3, 171), _lv(6.0, 128), _order(_lv(12.0, 200), 4), _lv(17.7, 77), _lv(9.1, 333)],
}


@pytest.mark.parametrize("precision", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("name", list(PARTS))
def test_batch_in_parts_equals_whole_steps(name, precision):
    insts = PARTS[name]()
    a, b = _pair(insts, precision, (64, 1, 130, 63, 7))
    assert a.info().steps_per_launch == 0 and a.info().parts == min(4, len(insts))
    _same(a, b, insts)


@pytest.mark.parametrize("name", ["one_launch", "wide"])
def test_short_graphs_equal_single_steps(name):
    insts = PARTS["one_launch"]() if name == "one_launch" else [_lv(20.3, 171)]
    a, b = _pair(insts, "f32", (1, 45, 15, 24, 63))
    assert a.info().short_graph_steps == 8
    _same(a, b, insts)


def _solid():
    return Instance(node=np.ones((5, 6, 7), np.uint8), tau=0.8, name="solid")


# batches whose first, middle or last instances store no cells
HOLLOW = {
    "one_tube": lambda: [_solid(), _lv(13.0, 830)],
    "one_tube_last": lambda: [_lv(13.0, 830), _solid(), _solid()],
    "three_tubes": lambda: [_solid(), _lv(13.0, 450), configs.rigid_tube(31, 31, 170, radius=11.4), _lv(12.2, 443)],
    "half_of_the_cells": lambda: [_solid(), _solid(), _lv(13.0, 600), _lv(6.3, 41), _solid(), _lv(9.1, 333), _lv(6.0, 128)],
}


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("name", list(HOLLOW))
def test_batch_with_solid_instances_equals_whole_steps(name, precision):
    # whole graphs, single-step ones and graphs again: the step counter that the
    # inlet phase, the elastance and the waveform rows follow advances in all
    insts = HOLLOW[name]()
    a, b = _pair(insts, precision, (64, 3, 130, 63, 7))
    tubes = sum(bool((i.node == 0).any()) for i in insts)
    assert a.info().steps_per_launch == 0 and a.info().parts == min(4, tubes)
    _same(a, b, insts)


@pytest.mark.parametrize("name", ["lv", "velocity", "uneven"])
def test_grid_that_gives_up_waiting_is_reported(name):
    # one poll at each barrier: blocks give up while the others still work, each
    # returns, and the launch is reported as failed whatever its populations
    # came to; the next lattice is not touched by it
    from paper_2112_05258_gb300 import LBMError, Lattice
    insts = GRID[name]()
    a = Lattice(insts, precision="f32")
    for q, inst in enumerate(insts):
        a.init_populations(q, configs.random_populations(inst, seed=q, amp=2e-3))
    a.set_wait_limit(1)
    a.step(400)
    with pytest.raises(LBMError) as e:
        a.sync()
    assert e.value.status == -2 and "did not meet" in str(e.value)
    a.close()
    a, b = _pair(insts, "f32", (30,))
    _same(a, b, insts)


def test_a_launch_that_gave_up_is_not_called_unstable():
    from paper_2112_05258_gb300 import LBMError, Lattice
    inst = GRID["lv"]()[0]
    f = configs.random_populations(inst, seed=1, amp=0.0)
    f[5] += 0.4                               # |v| > 0.3 everywhere: both status bits are set
    a = Lattice([inst], precision="f32")
    a.init_populations(0, f)
    a.set_wait_limit(1)
    a.step(400)
    with pytest.raises(LBMError) as e:
        a.sync()
    assert e.value.status == -2
    with pytest.raises(LBMError):
        a.set_wait_limit(0)


@pytest.mark.parametrize("inst", [lambda: configs.lv_tube(period=300), lambda: GRID["lv"]()[0], lambda: _lv(13.0, 830)])
def test_steps_on_a_stream_that_is_captured(inst):
    # no lattice's steps can be captured (a replay would pass the step count on
    # the host by); a call of no steps enqueues nothing and is accepted
    import torch
    from paper_2112_05258_gb300 import LBMError, Lattice
    inst, s = inst(), torch.cuda.Stream()
    for n in (0, 1, 64):
        lat = Lattice([inst], precision="f32", stream=s.cuda_stream)
        lat.step(n + 1)
        lat.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(s):
            g.capture_begin(capture_error_mode="thread_local")
            try:
                lat.step(n)
                refused = False
            except LBMError:
                refused = True
            try:
                g.capture_end()
            except RuntimeError:                # a refused graph launch ends the capture
                assert refused
        assert refused == (n > 0) and lat.info().steps == n + 1
        lat.close()


# lattices whose single-step calls the layout of a multi-step launch does not
# repay: wide first layers, many cells, FP64 first layers, no boundary
SINGLE = {
    "flat": (lambda: [_lv(18.1, 12)], "f32"),
    "long": (lambda: [_lv(16.2, 310)], "f16"),
    "f64": (lambda: [configs.rigid_tube()], "f64"),
    "box": (lambda: [Instance(node=geometry.closed_box(31, 17, 53), tau=0.7, name="box")], "bf16"),
}


@pytest.mark.parametrize("name", list(SINGLE))
def test_single_step_calls_between_longer_ones(name):
    insts, precision = SINGLE[name][0](), SINGLE[name][1]
    a, b = _pair(insts, precision, (1, 1, 2, 1, 3, 40, 1, 2, 1))
    info = a.info()
    assert info.steps_per_launch > 0 and info.multi_step_from == (3 if name == "box" else 2)
    _same(a, b, insts)


def test_large_lattices_without_boundaries_keep_the_step_graphs():
    insts = [Instance(node=geometry.closed_box(80, 60, 50), tau=0.7, name="box")]
    a, b = _pair(insts, "f32", (64, 7))
    assert a.info().steps_per_launch == 0
    _same(a, b, insts)


@pytest.mark.parametrize("case", ["cluster", "grid", "batch"])
def test_without_multi_step_launches(case):
    # the caller's choice of step graphs (whole, short and single-step ones) for a
    # lattice that would take multi-step launches, and back
    import torch
    from paper_2112_05258_gb300 import Lattice
    insts = {"cluster": CASES["lv"], "grid": GRID["velocity"], "batch": GRID["uneven"]}[case]()
    a, b = (Lattice(insts, precision="f32") for _ in range(2))
    a.set_multi_step(False)
    assert a.info().steps_per_launch == 0 and a.info().short_graph_steps == 8 and b.info().steps_per_launch > 0
    params = torch.tensor(np.tile(insts[0].boundaries[1].params, (21, 1)), dtype=torch.float64).pin_memory()
    rows = [torch.zeros((21, 16), dtype=torch.float64, pin_memory=True) for _ in range(2)]
    for lat, r in zip((a, b), rows):
        for n in (150, 1, 31):
            lat.step(n)
        lat.step_io(0, 1, 21, params.data_ptr(), params.shape[1], r.data_ptr())
        lat.sync()
    assert np.array_equal(rows[0].numpy(), rows[1].numpy())
    _same(a, b, insts)
    a.set_multi_step(True)
    assert a.info().steps_per_launch == b.info().steps_per_launch
    for lat in (a, b):
        lat.step(9)
        lat.sync()
    _same(a, b, insts)


@pytest.mark.parametrize("name", ["lv", "velocity", "two_chunks", "grid_lv", "grid_two_passes", "grid_uneven"])
def test_multi_step_kernel_bf16(name):
    insts = CASES[name]()
    a, b = _pair(insts, "bf16", (1, 2, 150, 61))
    assert a.info().steps_per_launch > 0
    _same(a, b, insts)


def _io_against_calls(inst, precision, bc, n, start, **kw):
    """n steps with per-step 0D input and output in one call, and as calls of one
    step between a parameter update and a state read, which are only queued."""
    import torch
    from paper_2112_05258_gb300 import Lattice
    base = np.array(inst.boundaries[bc].params, dtype=np.float64)
    par = torch.from_numpy(np.tile(base, (n, 1)) * np.where(np.arange(base.size) == 0, 1.0 + 0.2 * np.sin(np.arange(n) / 9.0)[:, None], 1.0)).pin_memory()
    rows = [torch.zeros((n, 8 * len(inst.boundaries)), dtype=torch.float64, pin_memory=True) for _ in range(2)]
    a, b = (Lattice([inst], precision=precision, **kw) for _ in range(2))
    a.step(start)
    b.step(start)
    a.step_io(0, bc, n, par.data_ptr(), base.size, rows[0].data_ptr())
    a.sync()
    for k in range(n):
        b.set_0d_params(0, bc, par[k].numpy())
        b.step(1)
        b.state_0d_async(0, rows[1][k].data_ptr())
    b.sync()
    assert np.array_equal(rows[0].numpy(), rows[1].numpy())
    assert np.array_equal(rows[0].numpy()[:, 0], np.arange(start + 1, start + n + 1))
    _same(a, b, [inst])
    return a


@pytest.mark.parametrize("make,bc", [(lambda: CASES["lv"]()[0], 1), (lambda: CASES["lv_order4"]()[0], 1),
                                     (lambda: configs.rigid_tube(), 0),
                                     (lambda: configs.rigid_tube(27, 27, 251, radius=10.3), 0)])  # two chunks
def test_step_io_fp64_in_the_multi_step_kernel(make, bc):
    assert _io_against_calls(make(), "f64", bc, 90, 5).info().steps_per_launch > 0


# lattices without wall nodes whose boundary work is two kernels: FP64 beyond the
# multi-step sizes, and FP32 with more links than the clusters of one launch take
TWO_KERNELS = {
    "f64": (lambda: _lv(20.3, 351), "f64", 1),
    "f64_velocity": (lambda: configs.rigid_tube(41, 41, 405, radius=18.6), "f64", 0),
    "wide": (lambda: _lv(33.0, 40), "f32", 1),
}


@pytest.mark.parametrize("name", list(TWO_KERNELS))
def test_step_io_in_graphs_of_two_boundary_kernels(name):
    # two graphs of 64 steps and a rest of 22, from an odd step on
    make, precision, bc = TWO_KERNELS[name]
    info = _io_against_calls(make(), precision, bc, 150, 7).info()
    assert info.steps_per_launch == 0 and info.launches_per_step == 3


@pytest.mark.parametrize("name", ["f64", "wide"])
def test_queued_parameter_updates_between_step_graphs(name):
    # updates queued between graphs of 16 steps without waiting, and the same with a
    # wait after each call
    from paper_2112_05258_gb300 import Lattice
    make, precision, bc = TWO_KERNELS[name]
    inst = make()
    base = np.array(inst.boundaries[bc].params)
    a, b = (Lattice([inst], precision=precision, graph_steps=16) for _ in range(2))
    assert a.info().steps_per_launch == 0
    for k in range(12):
        p = base * np.where(np.arange(base.size) == 0, 1.0 + 0.05 * k, 1.0)
        for lat, wait in ((a, False), (b, True)):
            lat.set_0d_params(0, bc, p)
            lat.step(16 if k % 3 else 21)
            if wait:
                lat.sync()
    a.sync()
    _same(a, b, [inst])


def test_batch_of_wide_boundaries_takes_two_kernels():
    # 16 blocks of 512 threads a tube: fourteen tubes have more of them than SMs
    from paper_2112_05258_gb300 import Lattice
    few, many = ([_lv(13.0, 203 + q) for q in range(n)] for n in (5, 14))
    assert Lattice(few).info().launches_per_step == 2
    a, b = _pair(many, "f16", (64, 7))
    assert a.info().launches_per_step == 3
    _same(a, b, many)
