"""Axisymmetric lattice on the GPU (liblbm through include/lbm_axi.h) against
the axisymmetric CPU oracle on identical inputs.

FP64 instantiation: populations, fields, waveforms and 0D states agree to
rounding (1e-12 on f ~ 1/9) for a Womersley inlet with an RCR outlet, the
hybrid LV inlet through several valve cycles, and a stenosis with radial
velocities (links across the axis, mass source active), from rest and from
seeded random populations.  FP32: waveforms within 1e-4 of their peak.
"""
import numpy as np
import pytest

from oracle.axisym import AxiOracle
from workloads import axisym as axw
from workloads.spec import BC_PRESSURE, BC_RCR, BC_VELOCITY, Boundary

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Axi():
    from paper_2112_05258_gb300 import load
    from paper_2112_05258_gb300.axisym import AxiLattice
    load()
    return AxiLattice


def _stenosis_case(outlet="pressure"):
    node, _ = axw.stenosis(12, 40, 10.0, 4.0, 6.0)
    n_in = int((node[:, 0] == 2).sum())
    r = np.arange(n_in) + 0.5
    prof = np.zeros((n_in, 3))
    prof[:, 0] = 0.03 * (1 - (r / 10.0) ** 2)
    prof[:, 1] = 0.01
    out = Boundary(BC_PRESSURE, 0, -1, [1e-4]) if outlet == "pressure" else Boundary(BC_RCR, 0, -1, [0.05, 200.0, 1.0, 0.0])
    return axw.AxiInstance(node=node, tau=0.7, name="axi_stenosis",
                           boundaries=[Boundary(BC_VELOCITY, 0, +1, [2 * np.pi / 200], profile=prof), out])


def _compare(lat, o, atol_f=1e-12, atol_w=1e-12):
    fl = o.fluid
    fg, fo = lat.populations(), o.populations()
    assert np.abs(fg[:, fl] - fo[:, fl]).max() < atol_f
    for a, b in zip(lat.fields(), o.fields()):
        assert np.abs(a[fl] - b[fl]).max() < atol_f
    wg, wo = lat.waves(), o.waves()
    assert wg.shape == wo.shape
    assert np.array_equal(wg[:, 0], wo[:, 0])
    assert np.abs(wg[:, 1:] - wo[:, 1:]).max() < atol_w
    for k in range(len(o.bcs)):
        sg, so = lat.state_0d(k), o.state_0d(k)
        assert sg[6] == so["valve"]
        if o.bcs[k]["kind"] == 2:                       # LV: closure time
            assert sg[7] == so["Td"]
        assert abs(sg[2] - so["Qu"]) < atol_w and abs(sg[3] - (so["Pbar"] - 1 / 3)) < atol_w


def _run(Axi, inst, steps, f0=None, prec="f64", **kw):
    lat = Axi(inst, precision=prec, **kw)
    o = AxiOracle(inst.node, inst.tau, inst.boundaries, q_scale=inst.q_scale)
    if f0 is not None:
        lat.init_populations(f0)
        o.set_populations(f0)
    lat.step(steps)
    lat.sync()
    o.step(steps)
    return lat, o


def test_f64_womersley_rcr(Axi):
    lat, o = _run(Axi, axw.womersley_tube(), 300)
    _compare(lat, o)


def test_f64_lv_inlet_cycles(Axi):
    inst = axw.lv_tube(period=600)
    lat, o = _run(Axi, inst, 1500)
    w = o.waves()
    assert (np.diff(w[:, 4]) < 0).sum() >= 2
    _compare(lat, o, 1e-11, 1e-11)


def test_f64_stenosis_radial_flow(Axi):
    lat, o = _run(Axi, _stenosis_case(), 400)
    assert np.abs(o.fields()[2]).max() > 1e-4           # radial velocities present
    _compare(lat, o)


def test_f64_random_start(Axi):
    inst = _stenosis_case("rcr")
    rng = np.random.default_rng(5)
    f0 = (np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
          * (1 + 1e-2 * rng.standard_normal((9,) + inst.node.shape)))
    lat, o = _run(Axi, inst, 150, f0=f0)
    _compare(lat, o)


def test_graph_equals_direct(Axi):
    inst = axw.lv_tube(period=300)
    g = Axi(inst, precision="f64", graph_steps=8)
    g.step(203)
    d = Axi(inst, precision="f64", graph_steps=1000)
    d.step(203)
    assert np.array_equal(g.populations(), d.populations())
    assert np.array_equal(g.waves(), d.waves())


def test_graph_equals_direct_long_tube(Axi):
    # 1100 nodes along x: x-blocks 1 to 3 of 256 hold no first-layer node, so
    # inside the graphs their collide of the next step runs beside the boundary
    # kernels; bit for bit the same as the serial order of direct launches
    inst = axw.lv_tube(nx=1100, period=300)
    g = Axi(inst, precision="f64", graph_steps=8)
    g.step(203)
    d = Axi(inst, precision="f64", graph_steps=1000)
    d.step(203)
    assert np.array_equal(g.populations(), d.populations())
    assert np.array_equal(g.waves(), d.waves())


def test_f32_womersley_waveforms(Axi):
    inst = axw.womersley_tube()
    lat, o = _run(Axi, inst, 3000, prec="f32")
    wg, wo = lat.waves(), o.waves()
    for col in (1, 2, 5, 6):
        assert np.abs(wg[:, col] - wo[:, col]).max() < 1e-4 * np.abs(wo[:, col]).max() + 1e-9


def _wide(kind):
    """A grid small enough for the multi-step kernel whose first layers span
    two chunks of 256 nodes; LV and RCR ends, or a constant pressure."""
    inst = axw.lv_tube(nr=300, nx=12, radius=290.0, period=60)
    if kind == "order4":
        for b in inst.boundaries:
            b.params = list(b.params) + [4.0]
    if kind == "pressure":
        inst.boundaries[1] = Boundary(BC_PRESSURE, 0, -1, [1e-4])
    return inst


@pytest.mark.parametrize("kind", ["order1", "order4", "pressure"])
def test_wide_first_layers_match_oracle(Axi, kind):
    lat, o = _run(Axi, _wide(kind), 150)
    _compare(lat, o)


def test_step_calls_of_any_length_give_the_same_bits(Axi):
    # one call, many short calls and calls past the steps of one launch
    inst = axw.lv_tube(period=60)
    a, b = Axi(inst, precision="f32"), Axi(inst, precision="f32")
    a.step(4500)
    for n in (1, 2, 97, 4097, 303):
        b.step(n)
    a.sync()
    b.sync()
    assert np.array_equal(a.populations(), b.populations())
    assert np.array_equal(a.waves()[-200:], b.waves()[-200:])


def _layered(kind, radius):
    """A short grid with `radius` first-layer nodes at each end."""
    nr = radius + 10
    if kind == "velocity":
        inst = axw.womersley_tube(nr=nr, nx=12, radius=float(radius), period=200)
    else:
        inst = axw.lv_tube(nr=nr, nx=12, radius=float(radius), period=60)
    if kind == "order2":
        for b in inst.boundaries:
            b.params = list(b.params) + [2.0]
    if kind == "pressure":
        inst.boundaries[1] = Boundary(BC_PRESSURE, 0, -1, [1e-4])
    return inst


@pytest.mark.parametrize("prec,radius", [("f32", 6), ("f32", 256), ("f32", 257), ("f32", 513), ("f32", 690),
                                         ("f64", 6), ("f64", 130)])
@pytest.mark.parametrize("kind", ["order1", "order2", "pressure", "velocity"])
def test_multi_step_launches_equal_one_step_kernels(Axi, kind, prec, radius):
    # first layers of one to three chunks of 256 nodes, every kind of end: the same
    # bits as the one-step kernels, also after a change of path at an odd step
    inst = _layered(kind, radius)
    a, b = Axi(inst, precision=prec), Axi(inst, precision=prec)
    b.set_multi_step(False)
    assert a.info().steps_per_launch > 0 and b.info().steps_per_launch == 0
    for n in (1, 150, 32):
        a.step(n)
        b.step(n)
    a.set_multi_step(False)
    b.set_multi_step(True)
    for n in (66, 7):
        a.step(n)
        b.step(n)
    a.sync()
    b.sync()
    assert np.array_equal(a.populations(), b.populations())
    assert np.array_equal(a.waves(), b.waves())
    for k in range(2):
        assert np.array_equal(a.state_0d(k), b.state_0d(k))


@pytest.mark.parametrize("prec,nr", [("f64", 20), ("f32", 140)])
def test_graph_equals_direct_on_one_step_kernels(Axi, prec, nr):
    # too large for the multi-step launches; of the five x-blocks of a row 1 to 3
    # hold no first-layer node, so that inside the graphs their next collision
    # runs beside the boundary kernels
    inst = axw.lv_tube(nr=nr, nx=1100, radius=nr - 2.0, period=300)
    g, d = Axi(inst, precision=prec, graph_steps=8), Axi(inst, precision=prec, graph_steps=1000)
    assert g.info().steps_per_launch == 0 and g.info().overlapped_blocks == 3
    for lat in (g, d):
        lat.step(203)
        lat.sync()
    assert np.array_equal(g.populations(), d.populations())
    assert np.array_equal(g.waves(), d.waves())


def test_grid_beyond_the_l2(Axi):
    # the collision that fetches its populations ahead: graphs equal direct
    # launches bit for bit, and 12 steps from white noise follow the FP64 lattice.
    # Deviations stay below 0.03 = 4/9 of 1 % times 6.7; a step rounds each about 16
    # times at 2^-24 (3e-8), 12 steps add up to 3.4e-7, and 1e-6 leaves a factor
    # three for the terms in 1/r next to the axis.
    inst = axw.lv_tube(nr=320, nx=12000, radius=318.0, period=300)
    rng = np.random.default_rng(2)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    f0 = w * (1 + 1e-2 * rng.standard_normal((9,) + inst.node.shape).clip(-6, 6))
    g, d, e = (Axi(inst, precision=p, graph_steps=n) for p, n in (("f32", 4), ("f32", 1000), ("f64", 4)))
    assert g.info().fetched_ahead == 1 and e.info().fetched_ahead == 0 and g.info().steps_per_launch == 0
    for lat in (g, d, e):
        lat.init_populations(f0)
        lat.step(12)
        lat.sync()
    fg = g.populations()
    assert np.array_equal(fg, d.populations())
    assert np.abs(fg - e.populations()).max() < 1e-6


@pytest.mark.parametrize("prec,nx,nr", [("f32", 12, 1100), ("f32", 62, 1000), ("f64", 330, 41)])
def test_grids_whose_blocks_take_longer_than_one_step_kernels(Axi, prec, nx, nr):
    # wide first layers, and FP64 bulk blocks of many nodes: graphs of one-step
    # kernels, though the grid would fit the multi-step launch
    inst = axw.lv_tube(nr=nr, nx=nx, radius=nr - 1.0, period=60)
    assert Axi(inst, precision=prec).info().steps_per_launch == 0
