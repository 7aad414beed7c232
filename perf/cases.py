"""What users of this framework have it do, as cases that can be timed.

Each case is one call (or the few calls) a user's program makes through the
public entry points, with the sizes, storage modes, lattices and boundary
conditions of the repository's own workloads, tests and benchmark:

  interval   the time march between two checks of the stopping rule
             (``Solver.solve_budget``), then the readout and the state
  batch      the same for many uneven structures in one launch (``Batch``)
  setup      loading a structure: connectivity, 13-direction pore lengths,
             diffusivities, relaxation rates, link masks
  krylov     the diffusion-preconditioned steady solve
  lines      the line-eliminated steady solve (dissolved O2 in the ionomer)
  conv       one convolution layer of the warm-start network, forward and
             backward
  structure  generating a catalyst layer and its connectivity statistics

``exact`` forms the same outputs in 64 bits with plain torch.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1410_1914_gb300 import Solver, structures
from paper_1410_1914_gb300 import _lib as L
from paper_1410_1914_gb300.batch import Batch

# volume shares of the Pt layer at porosity 0.45 and its share of ionomer in
# the non-pore volume (the workloads of the inputs module)
IONOMER_SHARE = 0.343169
R_GAS = 8.314462618

# convolution layers of the warm-start network: name -> (input channels,
# output channels, level), level l running at edge / 2^l
LAYERS = {
    "e1a": (16, 16, 0), "e2a": (16, 32, 1), "e2b": (32, 32, 1), "e3a": (32, 64, 2), "e3b": (64, 64, 2),
    "bta": (64, 128, 3), "btb": (128, 128, 3), "d3a": (192, 64, 2), "d2a": (96, 32, 1), "d1a": (48, 16, 0),
}


def listed():
    return [
        # the smallest solves (test boxes, members of a screening study): launches and latency count
        dict(name="interval_24_fp32", kind="interval", recipe="pt", nx=24, ny=24, nz=24, porosity=0.5, storage="fp32",
             lattice="d3q7", knudsen=0, reactive=False, steps=200),
        # the quick start: D_eff of a 128^3 Pt layer, FP16 state, a check every 500 steps
        dict(name="interval_128_fp16", kind="interval", recipe="pt", nx=128, ny=128, nz=128, porosity=0.45,
             storage="fp16dev", lattice="d3q7", knudsen=1, reactive=False, steps=500),
        # the benchmark's layer: 256^3 Pt, 5 % catalytic faces
        dict(name="interval_256_fp16", kind="interval", recipe="pt", nx=256, ny=256, nz=256, porosity=0.45,
             storage="fp16dev", lattice="d3q7", knudsen=1, reactive=True, steps=300),
        # the largest layer: 400^3 NPMC at 1 nm, every solid-pore face catalytic
        dict(name="interval_400_npmc", kind="interval", recipe="npmc", nx=400, ny=400, nz=400, porosity=0.55,
             storage="fp16dev", lattice="d3q7", knudsen=1, reactive=True, steps=100),
        # a box of odd edges in the FP32 state (the default storage)
        dict(name="interval_odd_fp32", kind="interval", recipe="npmc", nx=161, ny=187, nz=203, porosity=0.55,
             storage="fp32", lattice="d3q7", knudsen=1, reactive=False, steps=200),
        # the paper's own lattice, on the state that reaches the 64-bit answer
        dict(name="interval_128_d3q19", kind="interval", recipe="pt", nx=128, ny=128, nz=128, porosity=0.45,
             storage="fp16dev", lattice="d3q19", knudsen=1, reactive=False, steps=200),
        # many structures of uneven size (a porosity study) in one launch
        dict(name="batch_24", kind="batch", members=24, edge_min=32, edge_max=160, storage="fp16dev", steps=200),
        # loading the benchmark's layer
        dict(name="setup_256", kind="setup", recipe="pt", nx=256, ny=256, nz=256, porosity=0.45, storage="fp16dev",
             lattice="d3q7", knudsen=1, reactive=True),
        # the steady state of a Knudsen layer without the time march
        dict(name="krylov_96", kind="krylov", nx=96, ny=96, nz=96, porosity=0.45, lattice="d3q7", reactive=False),
        # O2 dissolved in the ionomer, which only the line-eliminated solve reaches
        dict(name="lines_16", kind="lines", nx=16, ny=16, nz=16, porosity=0.45, dissolved=True),
        # the widest full-resolution layer of the warm-start network, at the batch it is trained with
        dict(name="conv_d1a_48", kind="conv", layer="d1a", batch=4, edge=48),
        # a 200^3 NPMC layer generated and labelled
        dict(name="structure_200", kind="structure", recipe="npmc", nx=200, ny=200, nz=200, porosity=0.55),
    ]


# ------------------------------------------------------------------ drawing
def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def _edges(rng, a, b, most):
    """Three edges around one size, log-uniform, at most `most` cells."""
    e = _log(rng, a, b)
    v = [max(a, min(b, int(round(e * math.exp(rng.uniform(-0.3, 0.3)))))) for _ in range(3)]
    if rng.random() < 0.3:
        v = [e, e, e]
    while v[0] * v[1] * v[2] > most:
        v = [max(a, int(x * 0.93)) for x in v]
    return dict(nx=v[0], ny=v[1], nz=v[2])


def draw(rng):
    kind = rng.choices(["interval", "batch", "setup", "krylov", "lines", "conv", "structure"],
                       [6, 1, 1.5, 1, 0.75, 1, 0.75])[0]
    recipe = rng.choice(["pt", "npmc"])
    porosity = round(rng.uniform(0.45, 0.65), 3)
    if kind == "interval":
        lattice = rng.choices(["d3q7", "d3q19"], [3, 1])[0]
        storage = rng.choices(["fp16dev", "fp32", "fp32pop"], [3, 2, 1])[0]
        most = 20e6 if lattice == "d3q7" else 6e6
        c = _edges(rng, 20, 288, most)
        cells = c["nx"] * c["ny"] * c["nz"] * (1 if lattice == "d3q7" else 4)
        steps = 2 * max(25, min(250, int(2e9 / cells)))
        return dict(kind=kind, recipe=recipe, **c, porosity=porosity, storage=storage, lattice=lattice,
                    knudsen=rng.choice([0, 1, 1]), reactive=rng.random() < 0.4, steps=steps)
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(4, 28), edge_min=rng.choice([24, 32, 40]),
                    edge_max=_log(rng, 64, 144), storage=rng.choice(["fp16dev", "fp32"]),
                    steps=2 * rng.randint(25, 100))
    if kind == "setup":
        return dict(kind=kind, recipe=recipe, **_edges(rng, 24, 300, 20e6), porosity=porosity,
                    storage=rng.choice(["fp16dev", "fp32", "fp32pop"]),
                    lattice=rng.choices(["d3q7", "d3q19"], [3, 1])[0], knudsen=1, reactive=rng.random() < 0.5)
    if kind == "krylov":
        return dict(kind=kind, **_edges(rng, 24, 96, 800_000), porosity=porosity,
                    lattice=rng.choices(["d3q7", "d3q19"], [3, 1])[0], reactive=rng.random() < 0.3)
    if kind == "lines":
        dissolved = rng.random() < 0.6
        return dict(kind=kind, **(_edges(rng, 10, 16, 4096) if dissolved else _edges(rng, 12, 30, 24_000)),
                    porosity=porosity, dissolved=dissolved)
    if kind == "conv":
        name = rng.choice(sorted(LAYERS))
        level = LAYERS[name][2]
        return dict(kind=kind, layer=name, batch=rng.choice([1, 2, 4]),
                    edge=rng.choice([6, 8, 12, 16] if level == 3 else [12, 16, 24, 32] if level else [32, 40, 48, 64]))
    return dict(kind=kind, recipe=recipe, **_edges(rng, 48, 224, 8e6), porosity=porosity)


# ---------------------------------------------------------------- preparing
def _structure(recipe, shape, porosity, seed):
    if recipe == "pt":
        return structures.pt_cl(shape, seed, porosity, (1.0 - porosity) * IONOMER_SHARE)
    base = porosity - 0.10
    return structures.npmc_cl(shape, seed, base, (1.0 - base) * IONOMER_SHARE, porosity)


def _layer(case, seed):
    """(phase, catalytic faces or None, solver parameters), as the workloads make them."""
    recipe = case.get("recipe", "pt")
    ph = _structure(recipe, (case["nz"], case["ny"], case["nx"]), case["porosity"], seed)
    params = dict(dx_m=2e-9 if recipe == "pt" else 1e-9, knudsen=case.get("knudsen", 1), T_K=353.0, p_atm=1.0,
                  M_kgmol=0.032, bc_in=0, bc_out=0, c_in=1.0, c_out=0.0, tau_ref=1.0, k_ms=0.0)
    react = None
    if case.get("reactive"):
        ph[:, :, 0] = 0  # the gas reservoir in front of the layer
        react = structures.reactive_faces(ph, 0.05 if recipe == "pt" else 1.0, seed)
        params.update(bc_out=1, k_ms=1e-3 if recipe == "pt" else 1e-5)
    return ph, react, params


def _batch_layers(case, seed):
    """The members of a batch: uneven cubes, Pt and NPMC in turn, porosity 0.35 to 0.65."""
    r = np.random.RandomState(seed % (1 << 32))
    sizes = np.random.RandomState(case["members"] * 1000 + case["edge_max"])  # the case's, not the seed's
    for i in range(case["members"]):
        # stratified edges: every batch has small and large members
        u = (i + sizes.rand()) / case["members"]
        e = case["edge_min"] + int(u * (case["edge_max"] - case["edge_min"] + 1))
        yield dict(recipe="pt" if i % 2 == 0 else "npmc", nx=e, ny=e, nz=e,
                   porosity=float(r.uniform(0.35, 0.65))), seed * 64 + i


def _out(case, s):
    return dict(C=torch.empty(s.n, dtype=torch.float32, device="cuda"),
                g=torch.empty(s.q * s.n, dtype=torch.float32, device="cuda"))


def _conv_inputs(case, seed):
    ci, co, _ = LAYERS[case["layer"]]
    n, d = case["batch"], case["edge"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    bf = torch.bfloat16
    x = torch.randn(n, d, d, d, ci, generator=g, device="cuda").clamp_(min=0).to(bf)  # activations after a ReLU
    w = (torch.randn(27, co, ci, generator=g, device="cuda") * math.sqrt(2.0 / (27 * ci))).to(bf)
    b = torch.randn(co, generator=g, device="cuda") * 0.05
    gy = (torch.randn(n, d, d, d, co, generator=g, device="cuda") * 1e-3).to(bf)
    return x, w, b, gy


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("interval", "setup", "krylov", "lines"):
        ph, react, params = _layer(case, seed)
        if kind == "lines":
            params.update(knudsen=1, ionomer_o2=1 if case["dissolved"] else 0)
        if kind == "interval":
            params.update(check_every=case["steps"])
        s = Solver(ph.shape, storage=case.get("storage", "fp32pop"), lattice=case.get("lattice", "d3q7"), **params)
        st = dict(case=case, s=s)
        if kind == "setup":
            st.update(ph=ph, react=react, active=torch.empty_like(ph),
                      omega=torch.empty(ph.shape, dtype=torch.float32, device="cuda"),
                      mask=torch.empty(ph.shape, dtype=torch.int16, device="cuda"))
        else:
            s.set_structure(ph, react)
            st.update(_out(case, s))
        return st
    if kind == "batch":
        solvers = []
        for c, sd in _batch_layers(case, seed):
            ph, _, params = _layer(c, sd)
            s = Solver(ph.shape, storage=case["storage"], check_every=case["steps"], **params)
            s.set_structure(ph)
            solvers.append(s)
        total = sum(s.n for s in solvers)
        return dict(batch=Batch(solvers), case=case, solvers=solvers,
                    C=torch.empty(total, dtype=torch.float32, device="cuda"),
                    g=torch.empty(7 * total, dtype=torch.float32, device="cuda"))
    if kind == "conv":
        x, w, b, gy = _conv_inputs(case, seed)
        ci, co, _ = LAYERS[case["layer"]]
        n, d = case["batch"], case["edge"]
        lib = L.load()
        lib.cl_nn_wgrad_workspace.restype = ctypes.c_longlong
        ws = lib.cl_nn_wgrad_workspace(*(ctypes.c_int(v) for v in (n, d, d, d, ci, co)))
        return dict(case=case, x=x, w=w, b=b, gy=gy, y=torch.empty_like(gy), gx=torch.empty_like(x),
                    dw=torch.empty(27, co, ci, device="cuda"), db=torch.empty(co, device="cuda"),
                    wd=torch.empty(27, ci, co, dtype=torch.bfloat16, device="cuda"),
                    ws=torch.empty(ws // 4 + 1, device="cuda"))
    return dict(case=case, seed=seed, labels=torch.empty((case["nz"], case["ny"], case["nx"]), dtype=torch.int32,
                                                         device="cuda"))


# ------------------------------------------------------------------ running
def _nn(name, *args):
    s = getattr(L.load(), name)(*args)
    if s != L.CL_OK:
        raise L.ClError(s, name, L.last_error_message())


def _readout(s, reactive):
    """The number a solve is made for, and its profiles along x.  It is as good as the
    f32 state that it is read from, and is handed on in that type."""
    if reactive:
        total, prof_r, prof_c = s.reaction_rate()
        return [np.float32(total), np.asarray(prof_r, np.float32), np.asarray(prof_c, np.float32)]
    return [np.float32(s.effective_diffusivity()[0])]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "interval":
        s = st["s"]
        info = s.solve_budget(case["steps"])
        flux = np.asarray([info["J_in"], info["J_out"], info["R"]], np.float32)
        read = _readout(s, case["reactive"])
        L.cl_lbm_get_field(s.h, st["C"])
        L.cl_lbm_get_populations(s.h, st["g"])
        return dict(flux=flux, read=read, C=st["C"], g=st["g"])
    if kind == "batch":
        _, infos, _ = st["batch"].solve(case["steps"])
        flux = np.asarray([[i["J_in"], i["J_out"]] for i in infos], np.float32)
        at = 0
        for s in st["solvers"]:
            L.cl_lbm_get_field(s.h, st["C"][at:at + s.n])
            L.cl_lbm_get_populations(s.h, st["g"][7 * at:7 * (at + s.n)])
            at += s.n
        return dict(flux=flux, C=st["C"], g=st["g"])
    if kind == "setup":
        s = st["s"]
        s.set_structure(st["ph"], st["react"])
        L.cl_lbm_get_setup(s.h, st["active"], st["omega"], None, st["mask"])
        return dict(info=s.info(), active=st["active"], omega=st["omega"], mask=st["mask"])
    if kind == "krylov":
        s = st["s"]
        s.init()
        s.solve_krylov_dsa(tol=1e-8, max_iter=2000, max_steps=0)
    elif kind == "lines":
        s = st["s"]
        s.init()
        s.solve_steady_lines(tol=1e-12, max_iter=4000)
    if kind in ("krylov", "lines"):
        read = _readout(s, case.get("reactive", False))
        L.cl_lbm_get_field(s.h, st["C"])
        L.cl_lbm_get_populations(s.h, st["g"])
        return dict(read=read, C=st["C"], g=st["g"])
    if kind == "conv":
        ci, co, _ = LAYERS[case["layer"]]
        n, d = case["batch"], case["edge"]
        P, I = (lambda t: ctypes.c_void_p(t.data_ptr())), ctypes.c_int
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        geo = [I(v) for v in (n, d, d, d)]
        m = ctypes.c_longlong(n * d ** 3)
        _nn("cl_nn_conv3d", P(st["x"]), P(st["w"]), P(st["b"]), P(st["y"]), *geo, I(ci), I(co), I(ci), I(0), I(co), I(0),
            I(1), I(1), stream)
        _nn("cl_nn_relu_bwd", P(st["y"]), P(st["gy"]), m, I(co), I(co), I(0), stream)
        _nn("cl_nn_conv3d_wgrad", P(st["x"]), P(st["gy"]), P(st["ws"]), P(st["dw"]), *geo, I(ci), I(co), I(ci), I(0),
            I(co), I(0), I(1), stream)
        _nn("cl_nn_bias_grad", P(st["gy"]), m, I(co), I(co), I(0), P(st["db"]), stream)
        _nn("cl_nn_wt_dgrad", P(st["w"]), P(st["wd"]), I(co), I(ci), stream)
        _nn("cl_nn_conv3d", P(st["gy"]), P(st["wd"]), None, P(st["gx"]), *geo, I(co), I(ci), I(co), I(0), I(ci), I(0),
            I(0), I(1), stream)
        return dict(y=st["y"], gx=st["gx"], dw=st["dw"], db=st["db"])
    ph = _structure(case["recipe"], (case["nz"], case["ny"], case["nx"]), case["porosity"], st["seed"])
    faces = structures.reactive_faces(ph, 0.05, st["seed"])
    stats = structures.connectivity(ph)
    L.cl_phase_connectivity(ph, (0, 3), 26, False, labels=st["labels"])
    return dict(phase=ph, faces=faces, stats=stats, labels=st["labels"])


# --------------------------------------------------------------------- work
# bytes a lattice step moves per cell of the box: the state read and written, the link mask and omega
STEP_BYTES = {("d3q7", "fp16dev"): 38, ("d3q7", "fp32"): 62, ("d3q7", "fp32pop"): 62,
              ("d3q19", "fp16dev"): 2 * (6 + 36) + 8, ("d3q19", "fp32"): 2 * (8 + 72) + 8, ("d3q19", "fp32pop"): 160}


def work(case):
    kind = case["kind"]
    if kind == "conv":
        ci, co, _ = LAYERS[case["layer"]]
        m = case["batch"] * case["edge"] ** 3
        return dict(bytes=2 * m * (2 * ci + 2 * co) + 27 * ci * co * 8, flops=3 * 2 * 27 * ci * co * m)
    if kind == "batch":
        e0, e1 = case["edge_min"], case["edge_max"]
        n = sum((e0 + (i + 0.5) / case["members"] * (e1 - e0)) ** 3 for i in range(case["members"]))
        return dict(bytes=n * (STEP_BYTES["d3q7", case["storage"]] * case["steps"] + 32), flops=60 * n * case["steps"])
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "interval":
        q = 7 if case["lattice"] == "d3q7" else 19
        return dict(bytes=n * (STEP_BYTES[case["lattice"], case["storage"]] * case["steps"] + 4 * (q + 1)),
                    flops=(60 if q == 7 else 180) * n * case["steps"])
    if kind == "setup":
        # phase and faces in; active, omega, mask and the initial state out, and the copies handed to the caller
        state = {"fp16dev": 18, "fp32": 32, "fp32pop": 28}[case["storage"]]
        return dict(bytes=n * (2 + 7 + 7 + state), flops=200 * n)
    if kind in ("krylov", "lines"):
        q = 7 if case.get("lattice", "d3q7") == "d3q7" else 19
        return dict(bytes=n * (2 + 4 + 4 * q + 4 * (q + 1)), flops=60 * n)
    return dict(bytes=n * 6, flops=100 * n)


# -------------------------------------------------------------------- exact
D13 = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1),
       (1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1)]
C7 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
C19 = C7 + [(1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1),
            (0, -1, -1), (0, 1, -1), (0, -1, 1)]


def _shift(a, c):
    """a(x - c): periodic in y and z, and in x too (the callers mend the ends)."""
    return torch.roll(a, (c[2], c[1], c[0]), (0, 1, 2))


def _connected(transport):
    """Transport cells 6-connected to the plane x = 0 (y, z periodic)."""
    act = torch.zeros_like(transport)
    act[:, :, 0] = transport[:, :, 0]
    count = -1
    while True:
        for _ in range(8):
            new = act.clone()
            for c in C7[1:]:
                s = _shift(act, c)
                if c[0]:
                    s[:, :, 0 if c[0] > 0 else -1] = False
                new |= s
            act = new & transport
        k = int(act.sum())
        if k == count:
            return act
        count = k


def _pore_diameter(ph, dx):
    """Mean over 13 directions of the pore run through each cell, times dx."""
    pore = (ph == 0) | (ph == 3)
    nz, ny, nx = ph.shape
    total = torch.zeros(ph.shape, dtype=torch.float64, device=ph.device)
    for e in D13:
        period = 10 ** 9
        if e[0] == 0:
            py, pz = ny if e[1] else 1, nz if e[2] else 1
            period = py * pz // math.gcd(py, pz)
        run = torch.full(ph.shape, -1, dtype=torch.int32, device=ph.device)
        for sgn in (1, -1):
            # pore cells ahead, this one included: length after k doublings is at most 2^k
            r, k = pore.to(torch.int32), 1
            while k < (nx if e[0] else min(period, 1 << 30)):
                c = tuple(-sgn * k * v for v in e)
                ahead = _shift(r, c)
                if e[0]:  # cells past an x end hold no pore
                    if sgn > 0:
                        ahead[:, :, max(0, nx - k):] = 0
                    else:
                        ahead[:, :, :min(nx, k)] = 0
                r = torch.where(r == k, k + ahead, r)
                k *= 2
            run += r
        total += torch.clamp(run, max=period).double() * math.sqrt(sum(v * v for v in e))
    return torch.where(pore, total * dx / 13.0, torch.zeros_like(total))


class _Exact:
    """The step of Eq. 21 and its set-up in 64 bits."""

    def __init__(self, ph, react, p, lattice="d3q7", ionomer_o2=False):
        self.c = C7 if lattice == "d3q7" else C19
        q = len(self.c)
        self.q, self.ph, self.p = q, ph, p
        cs2 = 0.25 if q == 7 else 1.0 / 3.0
        self.w = [0.25] + [0.125] * 6 if q == 7 else [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
        nz, ny, nx = ph.shape
        T, dx = p["T_K"], p["dx_m"]
        d_ion = 0.0
        if ionomer_o2:
            henry = 1.01325e-1 * math.exp(-666.0 / T + 14.1)
            d_ion = 1e-10 * (0.1543 * (T - 273.0) - 1.65) * R_GAS * T / henry
        transport = (ph == 0) | (ph == 3) | ((ph == 2) if d_ion > 0 else torch.zeros_like(ph, dtype=torch.bool))
        self.act = _connected(transport)
        self.n_transport = int(transport.sum())
        d_b = 0.22e-4 * (T / 293.2) ** 1.5 / p["p_atm"]
        self.dp = _pore_diameter(ph, dx)
        if p["knudsen"]:
            d_kn = self.dp / 3.0 * math.sqrt(8.0 * R_GAS * T / (math.pi * p["M_kgmol"]))
            D = 1.0 / (1.0 / d_kn + 1.0 / d_b)
        else:
            D = torch.full(ph.shape, d_b, dtype=torch.float64, device=ph.device)
        D = torch.where(ph == 2, torch.full_like(D, d_ion), D)
        self.d_b, self.d_max = d_b, float(D[self.act].max())
        self.omega = torch.where(self.act, 1.0 / (0.5 + (p["tau_ref"] - 0.5) * D / self.d_max), torch.zeros_like(D))
        self.dt = (p["tau_ref"] - 0.5) * cs2 * dx * dx / self.d_max
        self.k = p["k_ms"] * self.dt / dx
        self.sink = 2.0 * self.k / (cs2 + self.k)
        # per link: wall (its end cell does not transport), catalytic, or a boundary link of the x faces
        solid = ph == 1
        cat = []
        for f, c in enumerate(C7[1:]):
            e = _shift(solid, tuple(-v for v in c))
            if c[0]:
                e[:, :, -1 if c[0] > 0 else 0] = False
            cat.append(e & (((react >> f) & 1) > 0) if react is not None else torch.zeros_like(e))
        self.wall, self.react, self.bound = [None], [None], [None]
        for c in self.c[1:]:
            back, mirror = tuple(-v for v in c), (0, -c[1], -c[2])
            ends = []
            for a in (self.act, solid):
                e = _shift(a, back)
                if c[0]:
                    end = -1 if c[0] > 0 else 0
                    e[:, :, end] = _shift(a, mirror)[:, :, end]
                ends.append(e)
            wall = self.act & ~ends[0]
            crossed = torch.zeros_like(wall)
            for axis in range(3):
                if c[axis]:
                    crossed |= cat[2 * axis + (0 if c[axis] > 0 else 1)]
            self.wall.append(wall)
            self.react.append(wall & ends[1] & crossed)
            b = torch.zeros_like(wall)
            if c[0]:
                end = -1 if c[0] > 0 else 0
                b[:, :, end] = (self.act & ~wall)[:, :, end]
            self.bound.append(b)
        x = torch.arange(nx, dtype=torch.float64, device=ph.device)
        ramp = p["c_in"] + (p["c_out"] - p["c_in"]) * (x + 0.5) / nx
        C = torch.where(self.act, ramp.expand(ph.shape), torch.zeros_like(D))
        self.g = [w * C for w in self.w]

    def opp(self, i):
        return i + 1 if i & 1 else i - 1

    def arriving(self, i, g):
        """Population i as it arrives at each cell, and (bc) twice its boundary value."""
        j = self.opp(i)
        c, p = self.c[i], self.p
        v = torch.where(self.wall[j], g[j], _shift(g[i], c))
        if self.sink:
            v = torch.where(self.react[j], v - self.sink * v, v)
        if c[0]:
            bc, val = (p["bc_in"], p["c_in"]) if c[0] > 0 else (p["bc_out"], p["c_out"])
            v = torch.where(self.bound[j], 2.0 * self.w[i] * val - g[j] if bc == 0 else g[j], v)
        return v

    def step(self):
        h = [self.g[0]] + [self.arriving(i, self.g) for i in range(1, self.q)]
        C = sum(h[1:], h[0])
        for i in range(self.q):
            h[i] = torch.where(self.act, h[i] - self.omega * (h[i] - self.w[i] * C), torch.zeros_like(C))
        self.g = h

    def matrix(self):
        """(I - A, b) of the fixed point g = A g + b, dense, over the populations of the active cells."""
        idx = torch.full(self.ph.shape, -1, dtype=torch.int64, device=self.ph.device)
        n = int(self.act.sum())
        idx[self.act] = torch.arange(n, device=idx.device)
        q, p, om = self.q, self.p, self.omega[self.act]
        M = torch.zeros(q * n, q * n, dtype=torch.float64, device=idx.device)
        b = torch.zeros(q, n, dtype=torch.float64, device=idx.device)
        rows = torch.arange(n, device=idx.device)
        for i in range(q):  # every arriving population is a factor times one stored population, plus a constant
            coef = torch.ones(n, dtype=torch.float64, device=idx.device)
            const = torch.zeros_like(coef)
            col = i * n + rows
            if i:
                j, c = self.opp(i), self.c[i]
                own = (self.wall[j] | self.bound[j])[self.act]
                col = torch.where(own, j * n + rows, i * n + _shift(idx, c)[self.act])
                coef = torch.where(self.react[j][self.act], coef - self.sink, coef)
                if c[0]:
                    bc, val = (p["bc_in"], p["c_in"]) if c[0] > 0 else (p["bc_out"], p["c_out"])
                    if bc == 0:
                        at = self.bound[j][self.act]
                        coef, const = torch.where(at, -coef, coef), torch.where(at, 2.0 * self.w[i] * val, const)
            for k in range(q):  # collision: g*_k = (1 - omega) g_k + omega w_k sum_i g_i
                f = om * self.w[k] + ((1.0 - om) if k == i else 0.0)
                M.index_put_((k * n + rows, col), -f * coef, accumulate=True)
                b[k] += f * const
        M.diagonal().add_(1.0)
        return M, b.reshape(-1)

    def solve(self):
        M, b = self.matrix()
        v = torch.linalg.solve(M, b).reshape(self.q, -1)
        self.g = [torch.zeros(self.ph.shape, dtype=torch.float64, device=self.ph.device) for _ in range(self.q)]
        for i in range(self.q):
            self.g[i][self.act] = v[i]

    def field(self):
        return sum(self.g[1:], self.g[0]).reshape(-1)

    def flux(self, x=None):
        """J_in, J_out and the reaction per plane of the stored populations."""
        p, zero = self.p, torch.zeros((), dtype=torch.float64, device=self.ph.device)
        jin, jout = zero, zero
        R = torch.zeros(self.ph.shape[2], dtype=torch.float64, device=self.ph.device)
        for i in range(1, self.q):
            if self.c[i][0] < 0 and p["bc_in"] == 0:
                jin = jin + (2.0 * (self.w[i] * p["c_in"] - self.g[i]))[self.bound[i]].sum()
            if self.c[i][0] > 0 and p["bc_out"] == 0:
                jout = jout + (2.0 * (self.g[i] - self.w[i] * p["c_out"]))[self.bound[i]].sum()
            R += torch.where(self.react[i], self.g[i], torch.zeros_like(self.g[i])).sum((0, 1)) * self.sink
        return jin, jout, R

    def read(self, reactive):
        jin, jout, R = self.flux()
        nz, ny, nx = self.ph.shape
        dx = self.p["dx_m"]
        if reactive:
            scale = dx ** 3 / self.dt
            n = self.act.sum((0, 1)).double()
            C = self.field().reshape(self.ph.shape).sum((0, 1))
            return [R.sum() * scale, R * scale, torch.where(n > 0, C / n.clamp(min=1), torch.zeros_like(C))]
        return [jout / (ny * nz) * nx / (self.p["c_in"] - self.p["c_out"]) * dx * dx / self.dt]

    def all(self):
        return torch.cat([v.reshape(-1) for v in self.g])


def exact(case, seed):
    kind = case["kind"]
    if kind == "structure":
        return None  # whole numbers
    if kind == "conv":
        x, w, b, gy = _conv_inputs(case, seed)
        ci, co, _ = LAYERS[case["layer"]]
        if case["batch"] * case["edge"] ** 3 * ci * co > 1e9:
            return None

        def conv(v, k):  # x is zero padded, y and z wrap
            v = torch.nn.functional.pad(v.double().permute(0, 4, 1, 2, 3), (0, 0, 1, 1, 1, 1), mode="circular")
            v = torch.nn.functional.pad(v, (1, 1, 0, 0, 0, 0))
            d = v.shape[2] - 2
            out = 0.0
            for t in range(27):
                kz, ky, kx = t // 9, t // 3 % 3, t % 3
                out = out + torch.einsum("nczyx,oc->nzyxo", v[:, :, kz:kz + d, ky:ky + d, kx:kx + d], k[t].double())
            return out, v

        y, xp = conv(x, w)
        y = (y + b.double()).clamp(min=0)
        # the masked gradient; where the output rounds to 0 or not is the layer's own reading, so its sign is y's
        gm = torch.where(y.to(torch.bfloat16) > 0, gy.double(), torch.zeros_like(y))
        d = case["edge"]
        dw = torch.stack([torch.einsum("nczyx,nzyxo->oc", xp[:, :, t // 9:t // 9 + d, t // 3 % 3:t // 3 % 3 + d,
                                                              t % 3:t % 3 + d], gm) for t in range(27)])
        gx, _ = conv(gm, torch.flip(w, (0,)).permute(0, 2, 1))
        return dict(y=y, gx=gx, dw=dw, db=gm.sum((0, 1, 2, 3)))
    if kind == "batch":
        fl, C, g = [], [], []
        for c, sd in _batch_layers(case, seed):
            ph, _, params = _layer(c, sd)
            e = _Exact(ph, None, params)
            for _ in range(case["steps"]):
                e.step()
            jin, jout, _ = e.flux()
            fl.append(torch.stack([jin, jout]))
            C.append(e.field())
            g.append(e.all())
        return dict(flux=None if case["storage"] == "fp16dev" else torch.stack(fl), C=torch.cat(C), g=torch.cat(g))
    ph, react, params = _layer(case, seed)
    if kind == "setup":
        e = _Exact(ph, react, params, case["lattice"])
        pore = (ph == 0) | (ph == 3)
        # the whole-number outputs have no other value than the start's; the rest of info is derived from D
        info = {k: None for k in ("n_cells", "n_transport", "n_active", "n_wall_links", "n_react_links")}
        info.update(D_b=e.d_b, D_max=e.d_max, dt_s=e.dt, k_lu=e.k, mean_pore_diameter_m=float(e.dp[pore].mean()))
        return dict(info=info, active=None, omega=e.omega, mask=None)
    if kind == "interval":
        e = _Exact(ph, react, params, case["lattice"])
        for _ in range(case["steps"]):
            e.step()
        jin, jout, R = e.flux()
        # a single flux of an FP16 state carries one draw of its rounding noise, which says nothing about the step
        half = case["storage"] == "fp16dev"
        return dict(flux=None if half else torch.stack([jin, jout, R.sum()]),
                    read=None if half else e.read(case["reactive"]), C=e.field(), g=e.all())
    # the steady solves: the fixed point by a dense solve, where that is small enough
    e = _Exact(ph, react, params, case.get("lattice", "d3q7"), bool(case.get("dissolved")))
    if int(e.act.sum()) * e.q > 20_000:
        return None
    e.solve()
    return dict(read=e.read(case.get("reactive", False)), C=e.field(), g=e.all())
