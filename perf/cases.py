"""Performance cases: the work that a user of this framework has it do.

A case advances a coupled lattice (or trains the warm-start network) through
the public Python entry points and returns what the program reads afterwards:
pressure and momentum fields, 0D state rows, trained parameters, predictions.
The kinds, with the program each stands for:

* ``tubes``     rigid tubes with 0D ends: one small tube (parity and
                development runs, latency bound), the same with a 0D input and
                a state row per step (coupling to an outside 0D model), sweeps
                of one tube (training data of the warm start) and batches of
                uneven tubes (parameter studies);
* ``membrane``  a straight elastic tube, wall nodes with springs or filaments;
* ``aorta``     the curved elastic vessel with branches, LV inlet and three
                Windkessel outlets;
* ``axi``       the axisymmetric lattice at the resolutions of the convergence
                study and at the large grid of the throughput measurement;
* ``train``     Adam steps of the warm-start network, then a prediction.

``exact`` restates the same discrete equations in plain FP64 torch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2112_05258_gb300 import Lattice
from paper_2112_05258_gb300.axisym import AxiLattice
from paper_2112_05258_gb300.mlp import MLP
from workloads import aorta, axisym, batch, configs
from workloads.spec import BC_LV, BC_PRESSURE, BC_RCR, BC_VELOCITY

CS2 = 1.0 / 3.0
POP_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
MAX_CELLS = 17.5e6      # fluid cells of the largest batch (listed and drawn)


def listed():
    tubes = dict(kind="tubes", n=1, inlet="lv", r_min=6.0, r_max=6.0, l_min=128, l_max=128, io=False)
    return [
        # the 24x24x64 tube with Womersley inlet and Windkessel outlet that parity runs use
        dict(tubes, name="tube_f32", inlet="womersley", r_min=8.0, r_max=8.0, l_min=64, l_max=64,
             precision="f32", steps=100),
        # the smallest LV tube, in the precision of the parity runs; odd step count
        dict(tubes, name="lv_tube_f64", r_min=5.0, r_max=5.0, l_min=32, l_max=32, precision="f64", steps=37),
        # one patient-sized tube driven by an outside 0D model: parameters in and states out each step
        dict(tubes, name="tube_io_f32", r_min=13.3, r_max=13.3, l_min=321, l_max=321, precision="f32",
             steps=150, io=True),
        # training data of the warm start: many copies of one small tube
        dict(tubes, name="sweep_f32", n=64, precision="f32", steps=100),
        # a parameter study over uneven tubes, FP32 and mixed precision
        dict(tubes, name="batch_f32", n=96, r_max=20.0, l_max=512, precision="f32", steps=100),
        dict(tubes, name="batch_f16", n=96, r_max=20.0, l_max=512, precision="f16", steps=100),
        # the straight elastic tube whose wall is 151 filaments
        dict(kind="membrane", name="membrane_f32", n_xy=64, nz=512, radius=24.0, filaments=True, precision="f32",
             steps=64),
        # the elastic aorta between two snapshots, FP32 and mixed precision
        dict(kind="aorta", name="aorta_f32", nz=1024, precision="f32", steps=64),
        dict(kind="aorta", name="aorta_f16", nz=1024, precision="f16", steps=64),
        # the axisymmetric convergence study, and its large grid
        dict(kind="axi", name="axi_d64", workload="conv", n_d=64, precision="f32", steps=200),
        dict(kind="axi", name="axi_d1024", workload="aorta", n_d=1024, precision="f32", steps=512),
        # two epochs of the warm-start training, then a prediction of one batch
        dict(kind="train", name="train_512", n_in=8, hidden=256, n_hidden=3, batch=512, steps=16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["tubes", "tubes", "tubes", "membrane", "aorta", "axi", "axi", "train"])
    steps = int(_log(rng, 20, 100))
    precision = rng.choice(["f32", "f32", "f16", "bf16", "f64"])
    if kind == "tubes":
        r_min = rng.uniform(4.0, 12.0)
        r_max = rng.uniform(r_min, 20.0)
        l_min = int(_log(rng, 24, 256))
        l_max = int(rng.uniform(l_min, 512))
        most = max(1.0, min(96.0, MAX_CELLS * (0.5 if precision == "f64" else 1.0) / (math.pi * r_max ** 2 * l_max)))
        n = int(_log(rng, 1.0, most + 0.999))
        return dict(kind=kind, n=n, inlet=rng.choice(["lv", "lv", "womersley"]), r_min=round(r_min, 2),
                    r_max=round(r_max, 2), l_min=l_min, l_max=l_max, io=rng.random() < 0.2,
                    precision=precision, steps=steps)
    if kind == "membrane":
        radius = rng.uniform(5.0, 26.0)
        return dict(kind=kind, n_xy=int(2 * radius + 8 + rng.randrange(4)), nz=int(_log(rng, 24, 512)),
                    radius=round(radius, 2), filaments=rng.random() < 0.4,
                    precision=precision, steps=steps)
    if kind == "aorta":
        return dict(kind=kind, nz=int(_log(rng, 256, 1024)), precision=rng.choice(["f32", "f16", "bf16"]),
                    steps=min(steps, 64))
    if kind == "axi":
        workload = rng.choice(["conv", "aorta"])
        return dict(kind=kind, workload=workload, n_d=int(_log(rng, 20, 1024)),
                    precision=rng.choice(["f32", "f32", "f64"]), steps=4 * steps)
    return dict(kind=kind, n_in=rng.choice([6, 8]), hidden=64 * rng.randrange(1, 7), n_hidden=rng.randrange(1, 5),
                batch=16 * int(_log(rng, 4, 128)), steps=rng.randrange(2, 20))


# --------------------------------------------------------------------------
# geometry and 0D parameters: the instances of a case, kept between runs as a
# program keeps its patient's geometry

@functools.lru_cache(maxsize=16)
def _instances(key):
    case = dict(key)
    if case["kind"] == "aorta":
        return [aorta.build(0, nz=case["nz"])]
    if case["kind"] == "membrane":
        return [configs.ib_tube(case["n_xy"], case["n_xy"], case["nz"], radius=case["radius"],
                                filaments=case["filaments"])]
    if case["kind"] == "axi":
        return [axisym.convergence_tube(case["n_d"]) if case["workload"] == "conv"
                else axisym.straight_aorta(case["n_d"])]
    rng = np.random.default_rng(1000 + case["n"])
    params = batch.draw_params(rng, case["n"], e_min_range=(0.05, 0.07))
    R = rng.uniform(case["r_min"], case["r_max"], case["n"])
    L = rng.integers(case["l_min"], case["l_max"] + 1, case["n"])
    if case["inlet"] == "lv":
        return [batch.lv_tube_instance(params[q], R[q], int(L[q])) for q in range(case["n"])]
    # radius + 4 to each side gives the 24x24x64 box of the parity tube
    return [configs.rigid_tube(int(math.ceil(2 * R[q] + 8)), int(math.ceil(2 * R[q] + 8)), int(L[q]), radius=float(R[q]))
            for q in range(case["n"])]


def _geometry(case):
    return _instances(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "steps", "precision", "io"))))


def _waves(shape, gen, amp, axis_flow):
    """Smooth start: pressure falling along the vessel plus a few seeded long
    waves, axial plug flow plus seeded long waves (FP64, on the GPU)."""
    nz, ny, nx = shape
    z = torch.arange(nz, device="cuda", dtype=torch.float64).view(nz, 1, 1) / nz
    y = torch.arange(ny, device="cuda", dtype=torch.float64).view(1, ny, 1) / ny
    x = torch.arange(nx, device="cuda", dtype=torch.float64).view(1, 1, nx) / nx

    def wave(a):
        k = [float(gen.uniform(1.0, 5.0)) for _ in range(3)]
        return a * float(gen.uniform(0.5, 1.0)) * torch.sin(k[0] * x + k[1] * y + 2 * k[2] * z + float(gen.uniform(0, 6.3)))

    flow = amp * float(gen.uniform(0.6, 1.0))
    P = CS2 + 0.1 * amp * (1.0 - z) * float(gen.uniform(0.5, 1.0)) + wave(0.02 * amp)
    v = [wave(0.05 * amp) for _ in range(3)]
    v[axis_flow] = v[axis_flow] + flow
    return P, v


def _start_states(inst, gen):
    """Seeded 0D states: (state, valve) per boundary, None where there is none."""
    out = []
    for b in inst.boundaries:
        p = float(gen.uniform(0.5e-3, 2e-3))
        out.append((2 * p, 1.0) if b.kind == BC_LV else (p, 0.0) if b.kind == BC_RCR else None)
    return out


def _lattice_inputs(case, seed):
    """Per instance: P, (vx, vy, vz), 0D start states; then the outlet parameters of every step (io)."""
    gen = np.random.default_rng(seed)
    for inst in _geometry(case):
        P, v = _waves(inst.node.shape, gen, 0.02, 2)
        yield P, v, _start_states(inst, gen)


def _io_params(case, seed):
    base = np.array(_geometry(case)[0].boundaries[1].params, dtype=np.float64)
    gen = np.random.default_rng(seed + 7)
    k = np.arange(case["steps"])
    out = np.tile(base, (case["steps"], 1))
    out[:, 0] *= 1.0 + 0.3 * np.sin(2 * np.pi * k / 50.0 + gen.uniform(0, 6.3))
    return out


def _axi_inputs(case, seed):
    """f(t_0) of the axisymmetric lattice (9 x nr x nx, FP64, on the GPU): equilibrium of a smooth axial flow."""
    inst = _geometry(case)[0]
    nr, nx = inst.node.shape
    P, v = _waves((1, nr, nx), np.random.default_rng(seed), 0.01, 0)
    e, w = _d2q9()
    f = torch.empty(9, nr, nx, dtype=torch.float64, device="cuda")
    vx, vr = v[0][0], v[1][0] * 0.0
    for i in range(9):
        eu = e[i][0] * vx + e[i][1] * vr
        f[i] = w[i] * (3 * P[0] + 3 * eu + 4.5 * eu * eu - 1.5 * (vx * vx + vr * vr))
    return f


def _train_inputs(case, seed):
    gen = np.random.default_rng(seed)
    n, n_out = 4096, 64
    X = gen.standard_normal((n, case["n_in"])).astype(np.float32)
    Y = np.zeros((n, n_out), np.float32)           # 23 labels fill the first outputs
    Y[:, :23] = np.tanh(X @ gen.standard_normal((case["n_in"], 23)))
    dims = [case["n_in"]] + [case["hidden"]] * case["n_hidden"] + [n_out]
    theta = np.concatenate([np.concatenate([gen.standard_normal(dims[k + 1] * dims[k]) / math.sqrt(dims[k]),
                                            np.zeros(dims[k + 1])]) for k in range(len(dims) - 1)]).astype(np.float32)
    order = np.concatenate([gen.permutation(n) for _ in range(case["steps"] * case["batch"] // n + 1)])
    return X, Y, theta, order[:case["steps"] * case["batch"]].astype(np.int32), dims


LEARNING_RATE = 2e-3


def prepare(case, seed):
    if case["kind"] == "train":
        X, Y, theta, order, dims = _train_inputs(case, seed)
        net = MLP(case["n_in"], case["hidden"], case["n_hidden"], 64, max_batch=max(64, (case["batch"] + 63) // 64 * 64))
        net.set_params(theta)
        net.set_data(X, Y)
        return dict(kind="train", net=net, order=order, batch=case["batch"], x=X[:case["batch"]])
    insts = _geometry(case)
    if case["kind"] == "axi":
        lat = AxiLattice(insts[0], precision=case["precision"])
        lat.init_populations(_axi_inputs(case, seed).cpu().numpy())
        return dict(kind="axi", lat=lat, steps=case["steps"], f32=case["precision"] == "f32")
    # a program that reads every so many steps has the step graphs take as many, where that is an even count
    lat = Lattice(insts, precision=case["precision"], graph_steps=case["steps"] if case["steps"] % 2 == 0 else 0)
    for q, (P, v, states) in enumerate(_lattice_inputs(case, seed)):
        P = P.expand(insts[q].node.shape)
        lat.init_equilibrium(q, *[a.reshape(-1).cpu().numpy() for a in (P, *v)])
        for k, s in enumerate(states):
            if s is not None:
                lat.set_0d_state(q, k, s[0], valve_open=s[1])
    state = dict(kind=case["kind"], lat=lat, steps=case["steps"], io=None)
    # one array a field, the instances' boxes one after another
    state["sizes"] = [i.node.size for i in insts]
    state["out"] = [torch.empty(sum(state["sizes"]), dtype=torch.float32, device="cuda") for _ in range(4)]
    if case.get("io"):
        par = torch.from_numpy(_io_params(case, seed)).pin_memory()
        rows = torch.zeros(case["steps"], 8 * len(insts[0].boundaries), dtype=torch.float64, pin_memory=True)
        state["io"] = (par, rows)
    return state


def run(state):
    if state["kind"] == "train":
        losses = state["net"].train(state["order"], state["batch"], LEARNING_RATE)
        return dict(losses=losses, theta=state["net"].params(), y=state["net"].forward(state["x"]))
    lat = state["lat"]
    if state["kind"] == "axi":
        lat.step(state["steps"])
        # the snapshot of an FP32 run is kept in FP32, as the 3D read-out does
        return [a.astype(np.float32) for a in lat.fields()] if state["f32"] else list(lat.fields())
    out = []
    if state["io"] is not None:
        par, rows = state["io"]
        lat.step_io(0, 1, state["steps"], par.data_ptr(), par.shape[1], rows.data_ptr())
        lat.sync()                          # the outside model reads the rows
        out.append(rows.float())
    else:
        lat.step(state["steps"])
    at = 0
    for q, size in enumerate(state["sizes"]):
        lat.fields_device(q, *[a.data_ptr() + 4 * at for a in state["out"]])
        at += size
    return out + state["out"]


def work(case):
    if case["kind"] == "train":
        d = [case["n_in"]] + [case["hidden"]] * case["n_hidden"] + [64]
        mac = sum(d[k] * d[k + 1] for k in range(len(d) - 1))
        par = mac + sum(d[1:])
        rows = case["batch"] * case["steps"]
        return dict(bytes=4.0 * (rows * (case["n_in"] + 64) + 6 * par * case["steps"]),
                    flops=2.0 * mac * (3 * rows + case["batch"]))
    insts = _geometry(case)
    fluid = float(sum((i.node == 0).sum() for i in insts))
    box = float(sum(i.node.size for i in insts))
    if case["kind"] == "axi":
        b = {"f64": 8, "f32": 4}[case["precision"]]
        return dict(bytes=fluid * 18 * b * case["steps"] + 24.0 * box, flops=130.0 * fluid * case["steps"])
    per = 38 * POP_BYTES[case["precision"]]
    nodes = float(sum(i.ib.n for i in insts if i.ib is not None))
    r = 8 if case["precision"] == "f64" else 4
    # wall nodes: position, velocity, penalty integral read and written, force and fluid velocity written,
    # reference, stiffness and area read, and the 64 support cells of each gathered and spread
    # (a cell of the lattice once each way: about 6 cells a node)
    wall = nodes * r * (6 + 6 + 6 + 6 + 5 + 6 * 6)
    return dict(bytes=(fluid * per + wall) * case["steps"] + 16.0 * box,
                flops=(fluid * 250.0 + nodes * 64 * 14.0) * case["steps"])


# --------------------------------------------------------------------------
# the same discrete equations in FP64 torch

def _d3q19():
    e = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
         (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
         (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
    return e, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _d2q9():
    e = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]
    return e, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def _opp(i):
    return i if i == 0 else (i + 1 if i % 2 else i - 1)


class _Zero:
    """The 0D models of all boundaries, one forward-Euler step at a time."""

    def __init__(self, boundaries, states):
        self.b, self.n = boundaries, 0
        self.s = [dict(p=float(b.params[3]) if b.kind in (BC_LV, BC_RCR) else 0.0, valve=0.0, Td=-1e300 if b.kind == BC_LV else 0.0,
                       Q=0.0, Qu=0.0, pg=0.0) for b in boundaries]
        for s, given in zip(self.s, states):
            if given is not None:
                s["p"], s["valve"], s["Td"] = given[0], given[1], -1e300

    def step(self, Q, A, pbar):
        """From Q, layer area and mean gauge pressure of t_n: per boundary (pressure type?, gauge pressure,
        smoothing factor, closed in this step?, phase of the inlet)."""
        out, n = [], self.n
        for b, s, q, a, pg in zip(self.b, self.s, Q, A, pbar):
            u = q / a
            s.update(Q=q, Qu=u, pbar=pg)
            ptype, p, S, closed, phase = 1, 0.0, 0.0, 0, 0.0
            if b.kind == BC_RCR:
                Rp, C, Rd = b.params[:3]
                s["p"] += -u / C - s["p"] / (Rd * C)
                p = s["pg"] = s["p"] - Rp * u
            elif b.kind == BC_PRESSURE:
                p = s["pg"] = float(b.params[0])
            elif b.kind == BC_VELOCITY:
                ptype, phase = 0, float(b.params[0]) * (n + 1)
            else:
                E, Ed = (float(v) for v in b.elastance[n % len(b.elastance)])
                Pv = s["p"] + (Ed / E) * s["p"] - E * (u if s["valve"] else 0.0)
                if s["valve"]:
                    if u < 0:
                        s["valve"], s["Td"], closed = 0.0, float(n), 1
                else:
                    Pv = max(Pv, float(b.params[1]))
                    if Pv > pg:
                        s["valve"] = 1.0
                p = s["p"] = s["pg"] = Pv
                ptype = int(s["valve"] != 0)
                t = (n + 1 - s["Td"]) / float(b.params[2])
                S = 1.0 if t <= 0 else 0.0 if t >= 1 else math.exp(2.0 * math.exp(-1.0 / t) / (t - 1.0))
            out.append((ptype, p, S, closed, phase))
        self.n += 1
        return out

    def row(self):
        """The 8 values of every boundary after the steps so far."""
        r = []
        for b, s in zip(self.b, self.s):
            E = float(b.elastance[self.n % len(b.elastance)][0]) if b.kind == BC_LV else 0.0
            r += [float(self.n), s["Q"], s["Qu"], s["pbar"], s["p"] if b.kind in (BC_LV, BC_RCR) else s["pg"],
                  s["p"] / E if E else 0.0, s["valve"], s["Td"]]
        return r


def _exact_lattice(case, seed):
    e, w = _d3q19()
    insts = _geometry(case)
    tau = insts[0].tau
    dev, f64 = "cuda", torch.float64
    boxes, cells, pulls, fs, zero_states, boundaries = [], 0, [[] for _ in range(19)], [], [], []
    links = dict(x=[], i=[], b=[], prof=[])
    n_links, places, ibs = 0, [], []
    for inst, (P, v, states) in zip(insts, _lattice_inputs(case, seed)):
        node = torch.from_numpy(inst.node).to(dev)
        nz, ny, nx = node.shape
        fluid = node == 0
        at = torch.full(node.shape, -1, dtype=torch.int64, device=dev)
        m = int(fluid.sum())
        at[fluid] = torch.arange(m, device=dev) + cells
        place = torch.nonzero(fluid.reshape(-1)).squeeze(1)
        code = torch.nn.functional.pad(node, (1, 1, 1, 1, 1, 1), value=1)
        where = torch.nn.functional.pad(at, (1, 1, 1, 1, 1, 1), value=-1)
        order = [torch.cumsum((node == 2 + k).reshape(-1), 0).reshape(node.shape) - 1 for k in range(len(inst.boundaries))]
        own = at[fluid]
        for i in range(19):
            sl = tuple(slice(1 - c, 1 - c + s) for c, s in zip(reversed(e[i]), (nz, ny, nx)))
            src = code[sl][fluid]
            # (direction, cell) as one number: -1 - link for the ghosts, which follow all cells
            pull = torch.where(src == 0, where[sl][fluid] + (i << 32), own + (_opp(i) << 32))
            for k, b in enumerate(inst.boundaries):
                hit = torch.nonzero(src == 2 + k).squeeze(1)
                if not hit.numel():
                    continue
                pull[hit] = -1 - n_links - torch.arange(hit.numel(), device=dev)
                links["x"].append(own[hit])
                links["i"].append(torch.full_like(hit, i))
                links["b"].append(torch.full_like(hit, len(boundaries) + k))
                prof = torch.zeros(hit.numel(), 3, dtype=f64, device=dev)
                if b.kind == BC_VELOCITY:
                    o = torch.nn.functional.pad(order[k], (1, 1, 1, 1, 1, 1))[sl][fluid][hit]
                    prof = torch.from_numpy(np.ascontiguousarray(b.profile)).to(dev)[o]
                links["prof"].append(prof)
                n_links += hit.numel()
            pulls[i].append(pull)
        vv = [a.expand(node.shape)[fluid] for a in v]
        PP = P.expand(node.shape)[fluid]
        f = torch.empty(19, m, dtype=f64, device=dev)
        for i in range(19):
            eu = sum(c * a for c, a in zip(e[i], vv))
            f[i] = w[i] * (3 * PP + 3 * eu + 4.5 * eu * eu - 1.5 * sum(a * a for a in vv))
        fs.append(f)
        places.append((place, node.numel()))
        boundaries += inst.boundaries
        zero_states += states
        ibs.append((inst.ib, at) if inst.ib is not None and inst.ib.n else None)
        cells += m
        del node, fluid, code, where, order
    f = torch.cat(fs, 1)
    pull = torch.stack([torch.cat(p) for p in pulls])
    pull = torch.where(pull < 0, cells * 19 - 1 - pull, (pull >> 32) * cells + (pull & 0xffffffff))
    del fs, pulls
    lx, li, lb = (torch.cat(links[k]) for k in "xib")
    prof = torch.cat(links["prof"])
    E = torch.tensor(e, dtype=f64, device=dev)
    W = torch.tensor(w, dtype=f64, device=dev)
    axis = torch.tensor([b.axis for b in boundaries], device=dev)
    sign = torch.tensor([float(b.sign) for b in boundaries], dtype=f64, device=dev)
    pair = torch.unique(lb * cells + lx)               # first layers: (boundary, cell)
    xb, xc = pair // cells, pair % cells
    A = torch.zeros(len(boundaries), dtype=f64, device=dev).index_add_(0, xb, torch.ones_like(xc, dtype=f64)).tolist()
    v_close = torch.zeros(lx.numel(), 3, dtype=f64, device=dev)
    zero = _Zero([_with_params(b) for b in boundaries], zero_states)
    io = _io_params(case, seed) if case.get("io") else None
    rows = []
    wall = _Wall(ibs[0], dev) if ibs[0] is not None else None
    om = 1.0 / tau
    b_force = torch.zeros(cells, 3, dtype=f64, device=dev) if wall else None

    def moments(f):
        return f.sum(0), [sum(c[a] * f[i] for i, c in enumerate(e) if c[a]) for a in range(3)]

    def along(i, v):
        return sum(c * v[a] for a, c in enumerate(e[i]) if c) if i else torch.zeros_like(v[0])

    for n in range(case["steps"]):
        if io is not None:
            zero.b[1].params = list(io[n])
        sd, j = moments(f)
        v = j
        if wall:
            b_force = wall.step(torch.stack(j, 1) + 0.5 * b_force, b_force)
            b = b_force.unbind(1)
            v = [p + 0.5 * q for p, q in zip(j, b)]
            vb = sum(p * q for p, q in zip(v, b))
        vv = sum(a * a for a in v)
        post = torch.empty(cells * 19 + lx.numel(), dtype=f64, device=dev)
        for i in range(19):
            ev = along(i, v)
            p = f[i] - om * (f[i] - w[i] * (sd + 3 * ev + 4.5 * ev * ev - 1.5 * vv))
            if wall:
                eb = along(i, b)
                p += (1 - 0.5 * om) * w[i] * (3 * eb + 9 * ev * eb - 3 * vb)
            post[i * cells:(i + 1) * cells] = p
        # 0D boundaries: flow and pressure of the first layers, the 0D step, the ghosts of t_{n+1}
        jl = torch.stack([a[xc] for a in j])
        q = sign[xb] * jl.gather(0, axis[xb].unsqueeze(0)).squeeze(0) / sd[xc]
        Q = torch.zeros(len(boundaries), dtype=f64, device=dev).index_add_(0, xb, q).tolist()
        ps = torch.zeros(len(boundaries), dtype=f64, device=dev).index_add_(0, xb, sd[xc] / 3 - CS2).tolist()
        res = zero.step(Q, A, [p / a for p, a in zip(ps, A)])
        r = torch.tensor(res, dtype=f64, device=dev)[lb]
        ptype, closed = r[:, 0] > 0, r[:, 3] > 0
        vf, Pf = torch.stack([a[lx] for a in v], 1), sd[lx] / 3
        v_close = torch.where(closed.unsqueeze(1), vf, v_close)
        given = torch.zeros_like(vf)
        un = sign[lb] * (prof[:, 0] + prof[:, 1] * torch.cos(r[:, 4]) - prof[:, 2] * torch.sin(r[:, 4]))
        given.scatter_(1, axis[lb].unsqueeze(1), un.unsqueeze(1))
        is_lv = torch.tensor([b.kind == BC_LV for b in boundaries], device=dev)[lb]
        given = torch.where(is_lv.unsqueeze(1), v_close * r[:, 2:3], given)
        vs = torch.where(ptype.unsqueeze(1), vf, given)
        Ps = torch.where(ptype, CS2 + r[:, 1], Pf)
        el = E[li]
        a, c = (el * vs).sum(1), (el * vf).sum(1)
        d = W[li] * (3 * (Ps - Pf) + 3 * (a - c) + 4.5 * (a * a - c * c) - 1.5 * ((vs * vs).sum(1) - (vf * vf).sum(1)))
        post[cells * 19:] = post[li * cells + lx] + d
        f = post[pull]
        if io is not None:
            rows.append(zero.row())
    sd, j = moments(f)
    out, o = [[], [], [], []], 0
    for place, size in places:
        for k, a in enumerate((sd / 3, *j)):
            full = torch.zeros(size, dtype=f64, device=dev)
            full[place] = a[o:o + place.numel()]
            out[k].append(full)
        o += place.numel()
    fields = [torch.cat(a) for a in out]
    return ([torch.tensor(rows, dtype=f64).float().double()] if io is not None else []) + fields


class _with_params:
    """A boundary whose parameters can be replaced without touching the instance."""

    def __init__(self, b):
        self.kind, self.params, self.elastance = b.kind, list(b.params), b.elastance


class _Wall:
    """Penalty immersed boundary: wall nodes with springs and filaments."""

    def __init__(self, given, dev):
        ib, self.at = given
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
        self.X0, self.dA, self.ks = t(ib.X0), t(ib.dA), t(ib.ks)
        self.pinned = t(ib.pinned).bool()
        self.alpha, self.beta, self.ms = ib.alpha, ib.beta, ib.ms
        self.X, self.V, self.I = self.X0.clone(), torch.zeros_like(self.X0), torch.zeros_like(self.X0)
        self.fil = None if not ib.filaments else (t(np.stack(ib.filaments)), t(np.asarray(ib.fil_par)))

    def step(self, v, b_old):
        """Interpolates v, takes the penalty force and spreads it: the new force density; then the wall moves."""
        h = self.X - 0.5
        i0 = torch.floor(h)
        nz, ny, nx = self.at.shape
        k = torch.arange(-1, 3, device=v.device)
        pos = i0.long().unsqueeze(2) + k                      # node, axis, 4
        phi = 0.25 * (1 + torch.cos(0.5 * math.pi * (pos - h.unsqueeze(2))))
        inside = [(pos[:, a] >= 0) & (pos[:, a] < s) for a, s in enumerate((nx, ny, nz))]
        x, y, z = (pos[:, a].clamp(0, s - 1) for a, s in enumerate((nx, ny, nz)))
        cell = self.at[z[:, :, None, None], y[:, None, :, None], x[:, None, None, :]]
        ok = (cell >= 0) & inside[2][:, :, None, None] & inside[1][:, None, :, None] & inside[0][:, None, None, :]
        wt = phi[:, 2][:, :, None, None] * phi[:, 1][:, None, :, None] * phi[:, 0][:, None, None, :]
        wt = torch.where(ok, wt, torch.zeros_like(wt)).reshape(len(h), 64, 1)
        cell = cell.clamp(min=0).reshape(len(h), 64)
        Vf = (v[cell] * wt).sum(1)
        dv = Vf - self.V
        self.I += dv
        F = self.alpha * self.I + self.beta * dv
        b = torch.zeros_like(b_old)
        b.index_add_(0, cell.reshape(-1), ((F * self.dA.unsqueeze(1)).unsqueeze(1) * wt).reshape(-1, 3))
        G = -self.ks.unsqueeze(1) * (self.X - self.X0) - F
        if self.fil is not None:
            nodes, par = self.fil
            ds, Eh, EI = (par[:, a].view(-1, 1, 1) for a in range(3))
            X = self.X[nodes]
            d = (X[:, 1:] - X[:, :-1]) / ds
            TD = Eh * (d.norm(dim=2, keepdim=True) - 1) * d
            K = torch.zeros_like(X)
            K[:, 1:-1] = (X[:, 2:] - 2 * X[:, 1:-1] + X[:, :-2]) / ds ** 2
            fil = (TD[:, 1:] - TD[:, :-1]) / ds - EI * (K[:, 2:] - 2 * K[:, 1:-1] + K[:, :-2]) / ds ** 2
            G.index_add_(0, nodes[:, 1:-1].reshape(-1), fil.reshape(-1, 3))
        self.V = torch.where(self.pinned.unsqueeze(1), self.V, self.V + G / self.ms)
        self.X = torch.where(self.pinned.unsqueeze(1), self.X, self.X + self.V)
        return b


def _exact_axi(case, seed):
    e, w = _d2q9()
    mirror = [0, 1, 2, 4, 3, 7, 8, 5, 6]
    inst = _geometry(case)[0]
    dev, f64 = "cuda", torch.float64
    node = torch.from_numpy(np.ascontiguousarray(inst.node)).to(dev)
    nr, nx = node.shape
    fluid = node == 0
    tau = inst.tau
    om, k, nu = 1.0 / tau, 1.0 - 0.5 / tau, (tau - 0.5) / 3.0
    r = torch.arange(nr, device=dev, dtype=f64).view(nr, 1) + 0.5
    f = torch.where(fluid, _axi_inputs(case, seed), torch.tensor(w, dtype=f64, device=dev).view(9, 1, 1))
    zero = _Zero(inst.boundaries, [None] * len(inst.boundaries))
    col = [1 if b.sign > 0 else nx - 2 for b in inst.boundaries]      # first fluid layers
    edge = [0 if b.sign > 0 else nx - 1 for b in inst.boundaries]
    lay = [fluid[:, c] & (node[:, g] == 2 + m) for m, (c, g) in enumerate(zip(col, edge))]
    # nodes of a layer: fluid with a boundary node at any of the three pull sources
    for m, g in enumerate(edge):
        b = node[:, g] == 2 + m
        near = b.clone()
        near[1:] |= b[:-1]
        near[:-1] |= b[1:]
        lay[m] = fluid[:, col[m]] & near
    A = [float((2 * math.pi * r[:, 0] * m).sum()) for m in lay]
    prof = []
    for m, b in enumerate(inst.boundaries):
        p = torch.zeros(nr, 3, dtype=f64, device=dev)
        if b.kind == BC_VELOCITY:
            p[node[:, edge[m]] == 2 + m] = torch.from_numpy(np.ascontiguousarray(b.profile)).to(dev)
        prof.append(p)
    v_close = [torch.zeros(2, nr, dtype=f64, device=dev) for _ in inst.boundaries]
    wall = torch.nn.functional.pad(node == 1, (1, 1, 0, 1), value=True)  # outside columns and the row above
    wall = torch.cat([wall[:1], wall])                                   # the mirror row below the axis

    def macro(f):
        sd = f.sum(0) - 1.0
        jx, jr = (sum(c[a] * f[i] for i, c in enumerate(e) if c[a]) for a in (0, 1))
        m = -jr / r
        pxr = f[5] + f[6] - f[7] - f[8]
        prr = f[3] + f[4] + f[5] + f[6] + f[7] + f[8] - CS2
        gx = -k * (pxr - jx * jr) / r - jx * jr / r
        gr = -k * (prr - sd / 3 - jr * jr) / r - 2 * nu * jr / r ** 2 - jr * jr / r
        return sd, jx, jr, m, gx, gr, jx + 0.5 * gx, jr + 0.5 * gr

    for n in range(case["steps"]):
        sd, jx, jr, m, gx, gr, vx, vr = macro(f)
        sp, vv = sd + 0.5 * m, vx * vx + vr * vr
        post = torch.empty_like(f)
        for i in range(9):
            ev, eg = e[i][0] * vx + e[i][1] * vr, e[i][0] * gx + e[i][1] * gr
            feq = w[i] * (1 + sp + 3 * ev + 4.5 * ev * ev - 1.5 * vv)
            post[i] = f[i] - om * (f[i] - feq) + k * w[i] * (3 * (eg - vx * gx - vr * gr) + 9 * ev * eg + m)
        Q = [float((2 * math.pi * r[:, 0] * b.sign * jx[:, c] / (1 + sd[:, c]))[l].sum())
             for b, c, l in zip(inst.boundaries, col, lay)]
        pb = [float((2 * math.pi * r[:, 0] * sp[:, c] / 3)[l].sum()) / a for c, l, a in zip(col, lay, A)]
        res = zero.step(Q, A, pb)
        pad = torch.nn.functional.pad(post, (1, 1, 1, 1))
        new = torch.empty_like(f)
        for i in range(9):
            ii = mirror[i]
            ex, er = e[i]
            pad[i, 0, 1:-1] = post[ii, 0]                              # below the axis: the mirrored population
            src = pad[i, 1 - er:1 - er + nr, 1 - ex:1 - ex + nx]
            bb = wall[1 - er:1 - er + nr, 1 - ex:1 - ex + nx]
            new[i] = torch.where(bb, post[_opp(i)], src)
        for q, (b, c, g, (ptype, p, S, closed, phase)) in enumerate(zip(inst.boundaries, col, edge, res)):
            fx, fr, fp = vx[:, c], vr[:, c], sp[:, c]
            if closed:
                v_close[q] = torch.stack([fx, fr])
            bnode = torch.nn.functional.pad(node[:, g] == 2 + q, (0, 1))
            bnode = torch.cat([bnode[:1], bnode])
            for i in range(9):
                if e[i][0] != b.sign:
                    continue
                er = e[i][1]
                hit = bnode[1 - er:1 - er + nr] & fluid[:, c]
                if ptype:
                    ps, sx, sr = 3 * p + 0 * fp, fx, fr
                elif b.kind == BC_VELOCITY:
                    row = torch.cat([prof[q][:1], prof[q], prof[q][:1] * 0])[1 - er:1 - er + nr]
                    ps, sr = fp, 0 * fr
                    sx = b.sign * (row[:, 0] + row[:, 1] * math.cos(phase) - row[:, 2] * math.sin(phase))
                else:
                    ps, sx, sr = fp, v_close[q][0] * S, v_close[q][1] * S
                es, ef = e[i][0] * sx + er * sr, e[i][0] * fx + er * fr
                d = w[i] * ((ps - fp) + 3 * (es - ef) + 4.5 * (es * es - ef * ef)
                            - 1.5 * ((sx * sx + sr * sr) - (fx * fx + fr * fr)))
                new[i, :, c] = torch.where(hit, post[i, :, c] + d, new[i, :, c])
        f = torch.where(fluid, new, f)
    sd, jx, jr, m, gx, gr, vx, vr = macro(f)
    z = torch.zeros_like(sd)
    return [torch.where(fluid, a, z) for a in ((1 + sd + 0.5 * m) / 3, vx, vr)]


def _exact_train(case, seed):
    X, Y, theta, order, dims = _train_inputs(case, seed)
    dev, f64 = "cuda", torch.float64
    X, Y = torch.from_numpy(X).to(dev, f64), torch.from_numpy(Y).to(dev, f64)
    th = torch.from_numpy(theta).to(dev, f64).requires_grad_()

    def net(x, th):
        o = 0
        for k in range(len(dims) - 1):
            n = dims[k] * dims[k + 1]
            x = x @ th[o:o + n].view(dims[k + 1], dims[k]).T + th[o + n:o + n + dims[k + 1]]
            o += n + dims[k + 1]
            x = torch.nn.functional.silu(x) if k < len(dims) - 2 else x
        return x

    m, v, losses = torch.zeros_like(th), torch.zeros_like(th), []
    for s in range(case["steps"]):
        rows = torch.from_numpy(order[s * case["batch"]:(s + 1) * case["batch"]]).to(dev).long()
        loss = ((net(X[rows], th) - Y[rows]) ** 2).mean()
        g, = torch.autograd.grad(loss, th)
        losses.append(loss.item())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        step = LEARNING_RATE * (m / (1 - 0.9 ** (s + 1))) / ((v / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
        th = (th - step).detach().requires_grad_()
    with torch.no_grad():
        return dict(losses=torch.tensor(losses, dtype=f64), theta=th.detach(), y=net(X[:case["batch"]], th))


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    with torch.no_grad():
        return _exact_axi(case, seed) if case["kind"] == "axi" else _exact_lattice(case, seed)
