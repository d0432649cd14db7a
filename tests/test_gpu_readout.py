"""FP32 device read-out (lbm_read_fields_device) against FP64 sums of the
populations the library reads out, over storage types, odd boxes, output
arrays at any 4-byte address, and non-finite populations.

Tolerance: the result is an FP32 rounding (2^-24 relative) of a sum that is
exact to 2^-44 of its terms' magnitudes; 2^-23 and 2^-40 leave a factor two
and more.
"""
import numpy as np
import pytest

from workloads import batch, configs

pytestmark = pytest.mark.gpu


def _device_fields(lat, inst, q, shift=0):
    import torch
    n = inst.node.size
    bufs = [torch.full((n + 8,), float("nan"), dtype=torch.float32, device="cuda") for _ in range(4)]
    torch.cuda.synchronize()        # the lattice has its own stream
    lat.fields_device(q, *[b.data_ptr() + 4 * shift for b in bufs])
    lat.sync()
    return [b[shift:shift + n].cpu().numpy() for b in bufs]


@pytest.mark.parametrize("precision", ["f32", "f16", "bf16", "f64"])
def test_device_fields_are_the_rounded_sums(d3q19, precision):
    from paper_2112_05258_gb300 import Lattice
    insts = [configs.lv_tube(period=300), batch.tube_batch(3, 11)[0][2], configs.ib_tube(19, 21, 17, radius=4.3),
             configs.lv_tube_x(31)]
    lat = Lattice(insts, precision=precision)
    for q, inst in enumerate(insts):
        lat.init_populations(q, configs.random_populations(inst, seed=q, amp=0.02))
    lat.step(21)
    lat.sync()
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    for q, inst in enumerate(insts):
        f = lat.populations(q)
        fl = inst.node.reshape(-1) == 0
        s = np.where(fl, f - w[:, None], 0.0)
        mag = np.abs(s).sum(0)
        want = [np.where(fl, f.sum(0) / 3, 0.0)] + [d3q19[:, a] @ s for a in range(3)]
        got = _device_fields(lat, inst, q, shift=q)
        for g, e in zip(got, want):
            assert (np.abs(g - e) <= 2.0 ** -23 * np.abs(e) + 2.0 ** -40 * mag).all()
            assert (g[~fl] == 0).all()


def test_device_fields_keep_infinities_and_nan():
    from paper_2112_05258_gb300 import Lattice
    inst = configs.lv_tube(period=300)
    lat = Lattice([inst], precision="f32")
    f = configs.random_populations(inst, seed=3)
    cells = np.flatnonzero(inst.node.reshape(-1) == 0)[[5, 400, 1200]]
    f[0, cells[0]] = np.inf
    f[7, cells[1]] = -np.inf
    f[3, cells[2]] = np.nan
    lat.init_populations(0, f)
    got = _device_fields(lat, inst, 0)
    want = lat.fields(0)
    for g, e in zip(got, want):
        assert np.array_equal(np.isnan(g), np.isnan(e)) and np.array_equal(np.isinf(g), np.isinf(e))
        at = np.isinf(e)
        assert np.array_equal(g[at], e[at].astype(np.float32))

