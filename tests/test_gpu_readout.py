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



def _cancelling(node, seed, precision):
    """Deviations s (19 x cells, exact in the storage type) whose sums cancel over
    many binades: in every cell one of 1 + sum s, jx, jy, jz adds a small term, a
    middle one and a large one (2^-22, 2^0, 2^10; FP16: 2^-12) before the large
    and the middle one are taken away again, so that what the large one pushed
    out of an FP32 sum decides."""
    rng = np.random.default_rng(seed)
    n = node.size
    e = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
                  (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
                  (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])

    def stored(v):
        v = v.astype(np.float32)
        if precision == "f16":
            return v.astype(np.float16).astype(np.float32)
        return (v.view(np.uint32) & 0xffff0000).view(np.float32) if precision == "bf16" else v

    def some(k):                            # +-[1/2, 1) 2^k
        return stored(rng.uniform(0.5, 1.0, n) * rng.choice([-1.0, 1.0], n) * 2.0 ** k)

    up = 10 if precision == "f16" else 0
    s = np.zeros((19, n), np.float32)
    kind = rng.integers(0, 4, n)
    for a in range(4):
        terms = [(i, 1) for i in range(1, 19)] if a == 0 else [(i, e[i, a - 1]) for i in range(19) if e[i, a - 1]]
        m, A = some(0), some(10)
        values = [some(up - 22), some(up - 21), m, some(up - 25), A, -A, some(up - 24), -m, some(up - 23), some(up - 26)]
        for (i, sign), v in zip(terms, values):
            s[i] = np.where(kind == a, sign * v, s[i])
    s[0] = np.where(kind == 0, stored(np.float32(-1.0) + some(-12)), s[0])
    return s, e


@pytest.mark.parametrize("precision", ["f32", "f16", "bf16"])
def test_device_fields_lose_no_more_than_fp64_sums(precision):
    # the error against exact sums: half an FP32 unit in the last place of the
    # result and 2^-53, the unit of FP64, of the terms' magnitudes (sequential
    # FP64 sums of these terms stay below it: at most three additions are rounded,
    # at a quarter of that each)
    import math
    from paper_2112_05258_gb300 import Lattice
    inst = configs.rigid_tube()
    s, e = _cancelling(inst.node, 9, precision)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    lat = Lattice([inst], precision=precision)
    f = s.astype(np.float64) + w[:, None]
    assert np.array_equal((f - w[:, None]).astype(np.float32), s)
    lat.init_populations(0, f)
    got = _device_fields(lat, inst, 0)
    for a, g in enumerate(got):
        terms = [s[i].astype(np.float64) * (1 if a == 0 else e[i, a - 1]) for i in range(19)] + [np.full(s.shape[1], float(a == 0))]
        T = np.array(terms)
        for c in np.flatnonzero(inst.node.reshape(-1) == 0):
            exact, mag = math.fsum(T[:, c]), np.abs(T[:, c]).sum()
            if a == 0:
                exact, mag = exact / 3, mag / 3
            assert abs(g[c] - exact) <= 2.0 ** -24 * (1 + 2.0 ** -20) * abs(exact) + 2.0 ** -53 * mag, (a, c)
