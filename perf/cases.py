"""The work that programs built on this library have it do, as cases that can be timed and checked.

A case is one call sequence through the public entry points of paper_2607_17929_gb300.pm.  The
largest part are particle-mesh boxes: load the particles (which runs the bootstrap solve), make a
few steps, read the state back.  Beside them stand the batched ensemble, the power spectrum, the
3^3 convolution and its weight gradient, a training step of the correction network, and the step
with that network attached.

Mixed-precision results leave the library as f64 copies of FP32 values (pm_get_particles,
pm_get_field); the cases keep them in FP32, the precision they were computed in.

exact() restates every case in 64-bit torch, from the equations (include/pm.h), without this
repository's code.
"""
import math

import numpy as np
import torch

from paper_2607_17929_gb300 import pm

OMEGA_M, H, NS, SIGMA8 = 0.31, 0.67, 0.96, 0.8
HUBBLE_LENGTH = 2997.92458
NEWTONIAN, FULL_HC, B_SPACESPACE = pm.PM_NEWTONIAN, pm.PM_FULL_HC, pm.PM_B_SPACESPACE
FIELDS = ("phi", "chi", "Bx", "By", "Bz")


# ---------------------------------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------------------------------

def _box(name, n, side, box, z, steps, fp64=False, flags=0, graph=False):
    """n: mesh side; side: particles per axis; box: Mpc/h; z: first redshift; steps after the load."""
    return {"name": name, "kind": "box", "n": n, "side": side, "box": box, "z": z, "steps": steps,
            "fp64": fp64, "flags": flags, "graph": graph}


def listed():
    return [
        # the FP64 parity configuration: 32^3 in 320 Mpc/h, ten steps; launches and host work count
        _box("fp64_32", 32, 32, 320.0, 100.0, 10, fp64=True),
        # the plain FP64 run at 256^3, the accuracy reference of the mixed runs
        _box("fp64_256", 256, 256, 1000.0, 100.0, 1, fp64=True),
        # a small mixed box stepped as captured graphs, as many seeds of it are run
        _box("mixed_64_graph", 64, 64, 200.0, 20.0, 8, graph=True),
        # the mixed run at 256^3, early (nearly uniform load)
        _box("mixed_256", 256, 256, 1000.0, 100.0, 4),
        # the headline: 512^3 in 2 Gpc/h, all ten stress-energy components
        _box("mixed_512", 512, 512, 2000.0, 100.0, 4),
        # late, clustered particles with both equation variants, on a mesh with a factor of three
        _box("mixed_192_late_variants", 192, 192, 500.0, 1.0, 4, flags=FULL_HC | B_SPACESPACE),
        # a Newtonian box with another particle number than cells (an odd one), late
        _box("newton_288_sparse", 288, 201, 700.0, 2.0, 4, flags=NEWTONIAN),
        # the batched ensemble of uneven boxes (64^3, 128^3, 192^3), four of each
        {"name": "ensemble_12", "kind": "ensemble", "sizes": "64,128,192", "copies": 4, "z": 30.0, "steps": 3,
         "batched": True},
        # the matter power spectrum of a running mixed box, taken as a diagnostic between steps
        {"name": "power_256", "kind": "power", "n": 256, "side": 256, "box": 1000.0, "z": 3.0, "fp64": False},
        # one hidden layer of the correction network at the mesh size it is run at
        {"name": "conv_256", "kind": "conv", "n": 256, "c_out": 16, "relu": True},
        # one training step of the correction network
        {"name": "train_128", "kind": "train", "n": 128},
        # the Newtonian step with the network's force correction attached
        {"name": "corrected_256", "kind": "corrected", "n": 256, "side": 256, "box": 500.0, "z": 20.0, "steps": 2},
    ]


# mesh sizes 2^a 3^b (a >= 3) over the range that is run: powers of two, and the others between them
MESHES = [16, 24, 32, 48, 64, 72, 96, 128, 144, 192, 216, 256, 288, 384]


def _mesh(rng, lo, hi):
    """A mesh side in [lo, hi], its logarithm spread evenly."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((m for m in MESHES if lo <= m <= hi), key=lambda m: abs(math.log(m / want)))


def draw(rng):
    kind = rng.choices(["box", "ensemble", "power", "conv", "convgrad", "train", "corrected"], [9, 2, 2, 2, 1, 1, 2])[0]
    z = round(math.exp(rng.uniform(math.log(1.0), math.log(100.0))), 3)
    cell = math.exp(rng.uniform(math.log(1.5), math.log(8.0)))   # Mpc/h per mesh cell
    if kind == "box":
        fp64 = rng.random() < 0.3
        n = _mesh(rng, 16, 192 if fp64 else 384)
        side = max(8, round(n * rng.choice([1.0, 1.0, rng.uniform(0.5, 1.2)])))
        # the spatial-spatial B and the full constraint are mostly left off, as in the paper's runs
        flags = rng.choices([0, NEWTONIAN, FULL_HC, B_SPACESPACE], [6, 2, 1, 1])[0]
        return dict(_box("", n, side, round(cell * n, 2), z, rng.randint(1, 6 if n < 200 else 3), fp64, flags,
                         rng.random() < 0.3))
    if kind == "ensemble":
        sizes = [_mesh(rng, 16, 160) for _ in range(rng.randint(1, 3))]
        return {"kind": "ensemble", "sizes": ",".join(map(str, sizes)), "copies": rng.randint(2, 6), "z": z,
                "steps": rng.randint(2, 4), "batched": rng.random() < 0.5}
    if kind == "power":
        n = _mesh(rng, 32, 256)
        return {"kind": "power", "n": n, "side": max(8, round(n * rng.uniform(0.5, 1.1))), "box": round(cell * n, 2),
                "z": z, "fp64": rng.random() < 0.5}
    if kind in ("conv", "convgrad"):
        n = 8 * round(math.exp(rng.uniform(math.log(2), math.log(31))))
        if kind == "convgrad":
            return {"kind": kind, "n": n}
        c_out = rng.choice([16, 16, 8])
        return {"kind": kind, "n": n, "c_out": c_out, "relu": c_out == 16 and rng.random() < 0.7}
    if kind == "train":
        return {"kind": kind, "n": 8 * rng.randint(3, 20)}
    n = rng.choice([32, 48, 64, 96, 128, 192])
    return {"kind": kind, "n": n, "side": max(8, round(n * rng.uniform(0.6, 1.1))), "box": round(cell * n, 2), "z": z,
            "steps": rng.randint(1, 3)}


# ---------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------

def _generator(seed, part=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + part)
    return g


def _transfer(k):
    """BBKS transfer function, k in h/Mpc."""
    q = k / (OMEGA_M * H)
    return torch.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3
                                                 + (6.71 * q) ** 4) ** -0.25


def _amplitude():
    lk = torch.linspace(math.log(1e-4), math.log(1e2), 20001, dtype=torch.float64)
    k = lk.exp()
    x = 8.0 * k
    w = 3 * (x.sin() - x * x.cos()) / x ** 3
    return SIGMA8 ** 2 / (torch.trapezoid(k ** (3 + NS) * _transfer(k) ** 2 * w ** 2, lk).item() / (2 * math.pi ** 2))


def _growth(a):
    """Linear growth factor of flat LCDM (the fit of Carroll, Press & Turner), D(1) = 1."""
    def g(x):
        om = OMEGA_M / (OMEGA_M + (1 - OMEGA_M) * x ** 3)
        ol = 1 - om
        return x * 2.5 * om / (om ** (4 / 7) - ol + (1 + om / 2) * (1 + ol / 70))
    return g(a) / g(1.0)


def _particles(side, box, z, seed, part=0):
    """Zel'dovich-displaced lattice of side^3 particles: f64 positions (box units) and momenta on the GPU."""
    noise = torch.randn((side, side, side), generator=_generator(seed, part), device="cuda", dtype=torch.float32)
    spec = torch.fft.rfftn(noise)
    del noise
    kf = 2 * math.pi / box                                  # h/Mpc
    ax = torch.fft.fftfreq(side, 1.0 / side, device="cuda")
    kx = torch.fft.rfftfreq(side, 1.0 / side, device="cuda")
    k2 = (ax[:, None, None] ** 2 + ax[None, :, None] ** 2 + kx[None, None, :] ** 2) * kf ** 2
    k2[0, 0, 0] = 1.0
    k = k2.sqrt()
    spec *= (_amplitude() * k ** NS * _transfer(k) ** 2 * (side / box) ** 3).sqrt() / k2
    spec[0, 0, 0] = 0
    a = 1 / (1 + z)
    om_a = OMEGA_M / (OMEGA_M + (1 - OMEGA_M) * a ** 3)
    d, f = _growth(a), om_a ** 0.55
    hc = a * (box / HUBBLE_LENGTH) * math.sqrt(OMEGA_M / a ** 3 + 1 - OMEGA_M)
    pos = torch.empty((side, side, side, 3), dtype=torch.float64, device="cuda")
    mom = torch.empty_like(pos)
    q = (torch.arange(side, device="cuda", dtype=torch.float64) + 0.5) / side
    for c, (kk, qq) in enumerate(((kx[None, None, :], q[None, None, :]), (ax[None, :, None], q[None, :, None]),
                                  (ax[:, None, None], q[:, None, None]))):
        psi = torch.fft.irfftn(1j * kf * kk * spec, s=(side,) * 3).double() / box
        pos[..., c] = torch.remainder(qq + d * psi, 1.0)
        mom[..., c] = a * hc * f * d * psi
    return pos.view(-1, 3), mom.view(-1, 3)


def _wrap(ptr, nbytes):
    class Buffer:
        __cuda_array_interface__ = {"shape": (nbytes,), "typestr": "|u1", "data": (ptr, False), "version": 3}
    return torch.as_tensor(Buffer(), device="cuda")


class _Ensemble:
    def __init__(self, configs, batched):
        self.e = pm.pm_ensemble_init(configs)
        pm.pm_ensemble_set_batched(self.e, batched)

    def __del__(self):
        pm.pm_ensemble_destroy(self.e)


class _Net:
    def __init__(self, n, seed):
        self.net = pm.pm_net_create(n, seed)

    def __del__(self):
        pm.pm_net_destroy(self.net)


def _net_params(seed, tag=7):
    """FP32 parameters of the 2-16-16-16-3 network in the library's padded layout, He-normal."""
    g = _generator(seed, tag)
    th = torch.zeros((4, 27 * 256 + 16), device="cuda")
    for layer, (ci, co) in enumerate(((2, 16), (16, 16), (16, 16), (16, 3))):
        w = torch.randn((27, co, ci), generator=g, device="cuda") * math.sqrt(2 / (27 * ci))
        th[layer, :27 * 256].view(27, 16, 16)[:, :co, :ci] = w * (0.1 if layer == 3 else 1.0)
        th[layer, 27 * 256:27 * 256 + co] = 0.05 * torch.randn(co, generator=g, device="cuda")
    return th.view(-1)


def _smooth(n, channels, seed, part):
    """BF16 [n^3][channels] activations of unit size with some correlation between neighbours."""
    x = torch.randn((n, n, n, channels), generator=_generator(seed, part), device="cuda")
    for d in range(3):
        x = (x + x.roll(1, d)) * math.sqrt(0.5)
    return x.view(-1, channels)


def _train_inputs(n, seed):
    x = torch.zeros((n ** 3, 16), device="cuda")
    x[:, :2] = _smooth(n, 2, seed, 1)
    t = torch.zeros((n ** 3, 8), device="cuda")
    t[:, :3] = 0.3 * _smooth(n, 3, seed, 2)
    return x.bfloat16(), t


def _conv_inputs(case, seed):
    n = case["n"]
    x = _smooth(n, 16, seed, 1).bfloat16()
    if case["kind"] == "convgrad":
        return x, _smooth(n, 16, seed, 2).bfloat16()
    w = torch.randn((27, 16, 16), generator=_generator(seed, 3), device="cuda") * math.sqrt(2 / (27 * 16))
    if case["c_out"] == 8:
        w[:, 8:] = 0
    return x, w.bfloat16(), 0.1 * torch.randn(16, generator=_generator(seed, 4), device="cuda")


def _sizes(case):
    return [int(n) for n in case["sizes"].split(",") for _ in range(case["copies"])]


def _ensemble_boxes(case, seed):
    """(mesh side, box side in Mpc/h) of every box: sides uniform in 200 to 1000 Mpc/h."""
    r = np.random.default_rng(seed)
    return [(n, float(r.uniform(200, 1000))) for n in _sizes(case)]


STEPS = 100   # length of every schedule


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("box", "power", "corrected"):
        n, side = case["n"], case["side"]
        fp64 = case.get("fp64", False)
        flags = case.get("flags", NEWTONIAN if kind == "corrected" else 0)
        s["pos"], s["mom"] = _particles(side, case["box"], case["z"], seed)
        s["sim"] = pm.PM(n, side ** 3, case["box"], OMEGA_M, case["z"], 0.0, STEPS,
                         pm.PM_FP64 if fp64 else pm.PM_MIXED, flags)
        if kind == "power":
            s["sim"].set_particles(s["pos"], s["mom"])
            return s
        s["sim"].step_graph(case.get("graph", False))
        s["out"] = torch.empty_like(s["pos"]), torch.empty_like(s["mom"])
        s["field"] = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
        if kind == "corrected":
            s["net"] = _Net(n, seed)
            pm.pm_net_set_params(s["net"].net, _net_params(seed))
        return s
    if kind == "ensemble":
        boxes = _ensemble_boxes(case, seed)
        s["ens"] = _Ensemble([dict(n_mesh=n, n_part=n ** 3, box_mpch=b, omega_m=OMEGA_M, z_init=case["z"],
                                   n_steps=STEPS, precision=pm.PM_MIXED) for n, b in boxes], case["batched"])
        s["in"] = [_particles(n, b, case["z"], seed, i) for i, (n, b) in enumerate(boxes)]
        s["out"] = [(torch.empty_like(p), torch.empty_like(u)) for p, u in s["in"]]
        return s
    if kind == "train":
        s["x"], s["target"] = _train_inputs(case["n"], seed)
        s["net"] = _Net(case["n"], seed)
        pm.pm_net_set_params(s["net"].net, _net_params(seed))
        _wrap(pm.pm_net_buffer(s["net"].net, pm.PM_NET_INPUT), s["x"].numel() * 2).copy_(s["x"].view(torch.uint8).view(-1))
        s["params"] = torch.empty(pm.pm_net_param_count(), device="cuda")
        return s
    if kind == "conv":
        s["x"], s["w"], s["b"] = _conv_inputs(case, seed)
        s["y"] = torch.empty((case["n"] ** 3, case["c_out"]), device="cuda",
                             dtype=torch.bfloat16 if case["c_out"] == 16 else torch.float32)
        return s
    s["x"], s["g"] = _conv_inputs(case, seed)
    s["dw"] = torch.empty((27, 16, 16), device="cuda")
    return s


# ---------------------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------------------

def _read(s, sim, keep):
    """Particles and the fields that this mode computes."""
    pos, mom = s["out"]
    pm.pm_get_particles(sim.ctx, pos, mom)
    got = {"pos": keep(pos), "mom": keep(mom)}
    case = s["case"]
    # B in the mixed form is the small transverse rest of FP32 momentum sums (1e-4 accurate early), so
    # the mixed cases return the potentials and the particles, the FP64 cases every field
    fp64 = case.get("fp64", False)
    newtonian = case["kind"] == "corrected" or case["flags"] & NEWTONIAN
    names = ("phi",) if newtonian else FIELDS if fp64 else ("phi", "chi")
    for name in names:
        pm.pm_get_field(sim.ctx, name, s["field"])
        got[name] = s["field"].clone() if fp64 else keep(s["field"])
    if fp64 and not newtonian:
        n = case["n"]
        for name in ("h+", "hx"):
            t = torch.empty((n, n, n // 2 + 1, 2), dtype=torch.float64, device="cuda")
            pm.pm_get_tensor(sim.ctx, name, t)
            got[name] = t
    return got


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "box":
        sim = state["sim"]
        sim.set_particles(state["pos"], state["mom"])
        for _ in range(case["steps"]):
            sim.step()
        return _read(state, sim, (lambda t: t) if case["fp64"] else torch.Tensor.float)
    if kind == "corrected":
        sim = state["sim"]
        sim.set_particles(state["pos"], state["mom"])
        for _ in range(case["steps"]):
            sim.project()
            sim.solve()
            pm.pm_net_apply(state["net"].net, sim.ctx)
            sim.update()
        return _read(state, sim, torch.Tensor.float)
    if kind == "ensemble":
        e = state["ens"].e
        for i, (pos, mom) in enumerate(state["in"]):
            pm.pm_ensemble_set_particles(e, i, pos, mom)
        for k in range(case["steps"]):
            pm.pm_ensemble_step(e, use_graph=k > 0)
        pm.pm_ensemble_sync(e)
        for i, (pos, mom) in enumerate(state["out"]):
            pm.pm_get_particles(pm.pm_ensemble_box(e, i), pos, mom)
        torch.cuda.synchronize()   # the boxes read on streams of the ensemble
        return [(p.float(), u.float()) for p, u in state["out"]]
    if kind == "power":
        k, pk, nmodes = state["sim"].power_spectrum(case["n"] // 2 + 1)
        if not case["fp64"]:   # the spectrum of an FP32 mesh
            k, pk = k.astype(np.float32), pk.astype(np.float32)
        return {"k": k, "pk": pk, "nmodes": nmodes}
    if kind == "train":
        loss = pm.pm_net_train_step(state["net"].net, state["target"], 1e-3)
        pm.pm_net_get_params(state["net"].net, state["params"])
        return {"loss": np.float32(loss), "params": state["params"]}
    if kind == "conv":
        pm.pm_conv3d_forward(case["n"], state["x"], state["w"], state["b"], case["c_out"], int(case["relu"]), state["y"])
        return state["y"]
    state["dw"].zero_()
    pm.pm_conv3d_backward_weight(case["n"], state["x"], state["g"], state["dw"])
    return state["dw"]


# ---------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------------

def _box_work(n, npart, steps, real, newtonian):
    """Bytes and operations of a load, `steps` steps and a read.

    Per step and particle: cell and offset and momentum read by the deposit, read and written by the
    kick, read and written by the sort.  Per step and cell: the sources and potentials written and
    read once, and the spectra between the transforms (9 forward, 5 inverse; Newtonian 1 and 1) in
    two passes each.
    """
    cells = n ** 3
    record = 4 + 6 * real
    fields = 2 if newtonian else 14
    per_cell = real * ((1 + 1 + 1) if newtonian else (9 + 5 + 3 + 8)) + 2 * real * fields
    flop_cell = fields * 2.5 * math.log2(cells) + (50 if newtonian else 400)
    flop_part = 100 if newtonian else 600
    load = npart * (48 + record) + cells * real * 6
    return {"bytes": load + steps * (5 * record * npart + per_cell * cells) + 48 * npart,
            "flops": (steps + 0.2) * (flop_cell * cells + flop_part * npart)}


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        each = [_box_work(n, n ** 3, case["steps"], 4, False) for n in _sizes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n = case["n"]
    cells = n ** 3
    if kind == "box":
        return _box_work(n, case["side"] ** 3, case["steps"], 8 if case["fp64"] else 4, case["flags"] & NEWTONIAN)
    if kind == "corrected":
        w = _box_work(n, case["side"] ** 3, case["steps"], 4, True)
        return {"bytes": w["bytes"] + case["steps"] * cells * (8 + 4 + 6 * 32 + 32),
                "flops": w["flops"] + case["steps"] * cells * 2 * 27 * (2 * 16 + 2 * 256 + 48)}
    if kind == "power":
        real = 8 if case["fp64"] else 4
        return {"bytes": case["side"] ** 3 * (4 + 3 * real) + 4 * real * cells,
                "flops": 30 * case["side"] ** 3 + 2.5 * math.log2(cells) * cells}
    if kind == "train":
        macs = 27 * (2 * 16 + 2 * 256 + 48)
        return {"bytes": cells * (4 + 3 * 64 + 12 + 12 + 3 * 128), "flops": 2 * cells * (3 * macs - 27 * 32)}
    if kind == "conv":
        return {"bytes": cells * (32 + case["c_out"] * (2 if case["c_out"] == 16 else 4)),
                "flops": 2 * 27 * 16 * case["c_out"] * cells}
    return {"bytes": cells * 64, "flops": 2 * 27 * 256 * cells}


# ---------------------------------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------------------------------

class _Background:
    def __init__(self, box, z):
        self.h0 = box / HUBBLE_LENGTH
        self.x, self.w = np.polynomial.legendre.leggauss(64)
        a0 = 1 / (1 + z)
        self.a = [a0 * (1 / a0) ** (i / STEPS) for i in range(STEPS + 1)]
        self.dtau = [self.tau(self.a[i], self.a[i + 1]) for i in range(STEPS)]
        self.a_half = [self.after(self.a[i], 0.5 * self.dtau[i]) for i in range(STEPS)]

    def hc(self, a):
        return a * self.h0 * np.sqrt(OMEGA_M / a ** 3 + 1 - OMEGA_M)

    def tau(self, a0, a1):
        a = 0.5 * (a0 + a1) + 0.5 * (a1 - a0) * self.x
        return float(0.5 * (a1 - a0) * (self.w / (a * self.hc(a))).sum())

    def after(self, a0, dt):
        a = a0 * math.exp(dt * self.hc(a0))
        for _ in range(30):
            a -= (self.tau(a0, a) - dt) * a * self.hc(a)
        return float(a)


def _grad(f, d):
    """Centred difference along axis d (0: x) of a [z][y][x] mesh."""
    return (f.roll(-1, 2 - d) - f.roll(1, 2 - d)) * (0.5 * f.shape[0])


class _Exact:
    """One box in FP64 torch: the same equations with plain FFTs and index sums."""

    def __init__(self, n, box, z, pos, mom, flags):
        self.n, self.flags, self.bg = n, flags, _Background(box, z)
        self.newton = bool(flags & NEWTONIAN)
        self.pos, self.mom = pos.clone(), mom.clone()
        self.m = OMEGA_M / pos.shape[0]
        self.g4 = 1.5 * self.bg.h0 ** 2
        zero = torch.zeros((n, n, n), dtype=torch.float64, device="cuda")
        self.phi1 = self.phi2 = self.chi = zero
        nf = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64).round().long()
        nf[n // 2] = n // 2
        nx = torch.arange(n // 2 + 1, device="cuda")
        self.nv = torch.stack(torch.broadcast_tensors(nx[None, None, :], nf[None, :, None], nf[:, None, None]))
        self.kt = [2 * n * torch.sin(math.pi * self.nv[d].double() / n) for d in range(3)]
        self.k2 = sum(k * k for k in self.kt)
        self.k2s = self.k2.clone()
        self.k2s[0, 0, 0] = 1
        dead = (self.nv.abs() * 2 == n).any(0)
        dead[0, 0, 0] = True
        self.live = (~dead).double()
        self.h = [torch.zeros((n, n, n // 2 + 1), dtype=torch.complex128, device="cuda") for _ in range(4)]
        self.b = None
        self.step_no = 0
        self.phi1 = self.phi2 = self._solve(True)
        self.chi = zero

    def _corners(self):
        n = self.n
        s = torch.remainder(self.pos, 1.0) * n
        c = s.floor()
        f = s - c
        c = c.long() % n
        for i in range(8):
            d = (i & 1, (i >> 1) & 1, (i >> 2) & 1)
            w = torch.ones_like(f[:, 0])
            idx = []
            for a in range(3):
                w = w * (f[:, a] if d[a] else 1 - f[:, a])
                idx.append((c[:, a] + d[a]) % n)
            yield (idx[2] * n + idx[1]) * n + idx[0], w

    def _deposit(self, charges):
        out = [torch.zeros(self.n ** 3, dtype=torch.float64, device="cuda") for _ in charges]
        for idx, w in self._corners():
            for o, q in zip(out, charges):
                o.index_add_(0, idx, w * q)
        return [o.view(self.n, self.n, self.n) for o in out]

    def _gather(self, fields):
        out = [torch.zeros_like(self.pos[:, 0]) for _ in fields]
        for idx, w in self._corners():
            for o, f in zip(out, fields):
                o += w * f.reshape(-1)[idx]
        return out

    def _solve(self, boot):
        n, k, bg = self.n, self.step_no, self.bg
        full = not (boot or self.newton)
        a, hc = bg.a[k], bg.hc(bg.a[k])
        dprev = bg.dtau[k - 1] if k >= 1 else bg.dtau[0]
        dprev2 = bg.dtau[k - 2] if k >= 2 else bg.dtau[0]
        c1 = 0.0 if boot or self.newton else 3 * hc / dprev
        c2 = 0.0 if self.newton else 3 * hc * hc
        u = [self.mom[:, d] for d in range(3)]
        if self.newton:
            r = self._deposit([torch.full_like(u[0], self.m)])[0]
            r = self.g4 / a * (r * n ** 3 - OMEGA_M)
        else:
            u2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
            en = (a * a + u2).sqrt()
            ph, ch = self._gather([self.phi1, self.chi]) if full else (0.0, 0.0)
            v2 = u2 / en ** 2
            charges = [self.m * en * (1 + 3 * ph + ph * v2)]
            if full:
                wv, ws = self.m * (1 + 4 * ph - ch), self.m * (1 + 3 * ph - ph * v2) / en
                charges += [wv * x for x in u]
                charges += [ws * u[i] * u[j] for i in range(3) for j in range(i, 3)]
            dep = self._deposit(charges)
            g = self.g4 / (a * a)
            r = g * (dep[0] * n ** 3 - a * OMEGA_M) - c1 * self.phi1 - c2 * self.chi
        dphi = (self.phi1 - self.phi2) / dprev2
        if full:
            gphi = [_grad(self.phi1, d) for d in range(3)]
            gpsi = [gphi[d] - _grad(self.chi, d) for d in range(3)]
            if self.flags & FULL_HC:
                psi = self.phi1 - self.chi
                lap = sum(self.phi1.roll(1, d) + self.phi1.roll(-1, d) for d in range(3)) - 6 * self.phi1
                x = -2 * psi
                small = x * x * (0.5 + x * (1 / 6 + x * (1 / 24 + x * (1 / 120 + x * (1 / 720 + x / 5040)))))
                ex2 = torch.where(x.abs() < 1e-2, small, torch.expm1(x) - x)
                r = r - (torch.expm1(2 * self.phi1) * lap * n * n
                         - 0.5 * torch.exp(2 * self.phi1) * sum(q * q for q in gphi)
                         + 1.5 * (hc * hc * ex2 - 2 * hc * dphi * torch.expm1(x) + dphi * dphi * torch.exp(x)))
        rk = torch.fft.rfftn(r)
        den = self.k2 + c1 + c2
        if self.newton:
            rk[0, 0, 0] = 0
            den = self.k2s
        phi = torch.fft.irfftn(-rk / den, s=(n, n, n))
        if not full:
            return phi
        quad = [[2 * gphi[i] * gphi[j] - (gphi[i] + gpsi[i]) * (gphi[j] + gpsi[j]) for j in range(3)] for i in range(3)]
        raw = {}
        it = iter(dep[4:])
        for i in range(3):
            for j in range(i, 3):
                raw[i, j] = 4 * g * n ** 3 * next(it) - 2 * quad[i][j]
        tr = (raw[0, 0] + raw[1, 1] + raw[2, 2]) / 3
        sk = {}
        for i in range(3):
            for j in range(i, 3):
                sk[i, j] = sk[j, i] = torch.fft.rfftn(raw[i, j] - tr if i == j else raw[i, j]) * self.live
        kt, k2 = self.kt, self.k2s
        kks = sum(kt[i] * kt[j] * sk[i, j] for i in range(3) for j in range(3))
        self.chi_new = torch.fft.irfftn(-0.75 / (k2 * k2) * kks, s=(n, n, n))
        # B
        if self.flags & B_SPACESPACE and k > 0:
            v = [sum(kt[i] * sk[i, j] for i in range(3)) for j in range(3)]
            kv = sum(kt[j] * v[j] for j in range(3))
            decay = (bg.a[k - 1] / a) ** 2
            self.b = [decay * self.b[j] - 1j * dprev / k2 * (v[j] - kt[j] * kv / k2) for j in range(3)]
        else:
            fk = [torch.fft.rfftn(g * n ** 3 * dep[1 + d] - dphi * gpsi[d]) * self.live for d in range(3)]
            kf = sum(kt[j] * fk[j] for j in range(3))
            self.b = [4 / k2 * (fk[j] - kt[j] * kf / k2) for j in range(3)]
        self.bx = [torch.fft.irfftn(b, s=(n, n, n)) for b in self.b]
        # tensor modes: helicity basis from the axis with the smallest |n_i|, implicit midpoint
        ab = self.nv.abs()
        ax = torch.zeros_like(ab[0])
        ax = torch.where(ab[1] < ab[0], 1, ax)
        ax = torch.where(ab[2] < torch.minimum(ab[0], ab[1]), 2, ax)
        kn = k2.sqrt()
        kh = [q / kn for q in kt]
        km = torch.where(ax == 0, kh[0], torch.where(ax == 1, kh[1], kh[2]))
        e1 = [(ax == d).double() - km * kh[d] for d in range(3)]
        ln = sum(e * e for e in e1).sqrt()
        ln[0, 0, 0] = 1
        e1 = [e / ln for e in e1]
        e2 = [kh[1] * e1[2] - kh[2] * e1[1], kh[2] * e1[0] - kh[0] * e1[2], kh[0] * e1[1] - kh[1] * e1[0]]
        is2 = math.sqrt(0.5)
        dt, hh = bg.dtau[k], bg.hc(bg.a_half[k])
        for p in range(2):
            s = sum(((e1[i] * e1[j] - e2[i] * e2[j]) if p == 0 else (e1[i] * e2[j] + e2[i] * e1[j])) * is2 * sk[i, j]
                    for i in range(3) for j in range(3))
            y, v = self.h[p], self.h[2 + p]
            r1 = y + 0.5 * dt * v
            r2 = -0.5 * dt * self.k2 * y + (1 - dt * hh) * v + dt * s
            m22 = 1 + dt * hh
            det = m22 + 0.25 * dt * dt * self.k2
            self.h[p] = (m22 * r1 + 0.5 * dt * r2) / det * self.live
            self.h[2 + p] = (r2 - 0.5 * dt * self.k2 * r1) / det * self.live
        return phi

    def step(self):
        n, k, bg = self.n, self.step_no, self.bg
        phi = self._solve(False)
        a, ah = bg.a[k], bg.a_half[k]
        dk = 0.5 * ((bg.dtau[k - 1] if k >= 1 else bg.dtau[0]) + bg.dtau[k])
        u = [self.mom[:, d] for d in range(3)]
        if self.newton:
            gp = self._gather([_grad(phi, d) for d in range(3)])
            u = [u[d] - dk * a * gp[d] for d in range(3)]
            dx = [bg.dtau[k] * u[d] / ah for d in range(3)]
        else:
            chi, b = self.chi_new, self.bx
            u2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
            en = (a * a + u2).sqrt()
            new = []
            for d in range(3):
                gp, gc, b0, b1, b2 = self._gather([_grad(f, d) for f in (phi, chi, *b)])
                new.append(u[d] + dk * (-en * (gp - gc) - u2 / en * gp - (u[0] * b0 + u[1] * b1 + u[2] * b2)))
            u = new
            v2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
            en = (ah * ah + v2).sqrt()
            p, c, *bv = self._gather([phi, chi, *b])
            fac = (1 + 3 * p - c - p * v2 / en ** 2) / en
            dx = [bg.dtau[k] * (u[d] * fac + bv[d]) for d in range(3)]
            self.chi = chi
        self.mom = torch.stack(u, 1)
        self.pos = torch.remainder(self.pos + torch.stack(dx, 1), 1.0)
        self.phi2, self.phi1 = self.phi1, phi
        self.step_no += 1


def _conv64(x, w, n):
    """Periodic 3^3 convolution in FP64: x [n^3][ci], w [27][co][ci]."""
    y = None
    x = x.view(n, n, n, -1)
    for d in range(27):
        off = (d // 9 - 1, (d // 3) % 3 - 1, d % 3 - 1)
        t = x.roll((-off[0], -off[1], -off[2]), (0, 1, 2)).reshape(n ** 3, -1) @ w[d].T
        y = t if y is None else y.add_(t)
    return y


def _dw64(x, g, n):
    x = x.view(n, n, n, -1)
    return torch.stack([g.T @ x.roll(tuple(-o for o in (d // 9 - 1, (d // 3) % 3 - 1, d % 3 - 1)), (0, 1, 2)).reshape(n ** 3, -1)
                        for d in range(27)])


def _train64(case, seed):
    n = case["n"]
    x, t = _train_inputs(n, seed)
    th = _net_params(seed).double().view(4, -1)
    w = [th[i, :27 * 256].view(27, 16, 16) for i in range(4)]
    act = [x.double()]
    for i in range(4):
        y = _conv64(act[i], w[i], n) + th[i, 27 * 256:]
        act.append(y.clamp_min(0) if i < 3 else y)
    diff = act[4][:, :3] - t[:, :3].double()
    loss = (diff ** 2).mean()
    g = torch.zeros_like(act[4])
    g[:, :3] = 2 * diff / diff.numel()
    grad = torch.zeros_like(th)
    for i in range(3, -1, -1):
        grad[i, :27 * 256] = _dw64(act[i], g, n).reshape(-1)
        grad[i, 27 * 256:] = g.sum(0)
        if i:
            g = _conv64(g, w[i].flip(0).transpose(1, 2), n) * (act[i] > 0)
    # layer 0 has 2 inputs and layer 3 has 3 outputs; the padded entries keep zero gradient
    grad[0, :27 * 256].view(27, 16, 16)[:, :, 2:] = 0
    grad[3, :27 * 256].view(27, 16, 16)[:, 3:] = 0
    # the first Adam step: m / (1 - b1) = g, sqrt(v / (1 - b2)) = |g|
    return {"loss": loss.view(()), "params": (th - 1e-3 * grad / (grad.abs() + 1e-8)).view(-1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "corrected":
        return None   # its forces pass through BF16 activations
    if kind == "conv":
        x, w, b = _conv_inputs(case, seed)
        y = (_conv64(x.double(), w.double(), case["n"]) + b.double())[:, :case["c_out"]]
        return y.clamp_min(0) if case["relu"] else y.contiguous()
    if kind == "convgrad":
        x, g = _conv_inputs(case, seed)
        return _dw64(x.double(), g.double(), case["n"])
    if kind == "train":
        return _train64(case, seed)
    if kind == "ensemble":
        got = []
        for i, (n, b) in enumerate(_ensemble_boxes(case, seed)):
            e = _Exact(n, b, case["z"], *_particles(n, b, case["z"], seed, i), 0)
            for _ in range(case["steps"]):
                e.step()
            got.append((e.pos, e.mom))
        return got
    n = case["n"]
    pos, mom = _particles(case["side"], case["box"], case["z"], seed)
    if kind == "power":
        rho = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
        for idx, w in _Exact._corners(type("P", (), {"n": n, "pos": pos})()):
            rho.index_add_(0, idx, w)
        dk = torch.fft.rfftn(rho.view(n, n, n) * (n ** 3 / pos.shape[0]) - 1)
        f = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
        x = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
        kn = (f[:, None, None] ** 2 + f[None, :, None] ** 2 + x[None, None, :] ** 2).sqrt()
        wt = torch.where((x > 0) & (2 * x < n), 2.0, 1.0).double()[None, None, :].expand_as(kn)
        nb = n // 2 + 1
        b = kn.round().long().reshape(-1)
        use = (b >= 1) & (b < nb)
        tot = [torch.bincount(b[use], (wt * q).reshape(-1)[use], nb)
               for q in (torch.ones_like(kn), 2 * math.pi * kn, dk.abs() ** 2 / float(n) ** 6)]
        cnt = tot[0].clamp_min(1)
        return {"k": tot[1] / cnt, "pk": tot[2] / cnt, "nmodes": None}
    if n > 400:
        return None   # the index sums of this size take more than 20 s
    e = _Exact(n, case["box"], case["z"], pos, mom, case["flags"])
    for _ in range(case["steps"]):
        e.step()
    got = {"pos": e.pos, "mom": e.mom, "phi": e.phi1}
    if not e.newton:
        got["chi"] = e.chi
        if case["fp64"]:
            got.update({"Bx": e.bx[0], "By": e.bx[1], "Bz": e.bx[2], "h+": torch.view_as_real(e.h[0].resolve_conj()),
                        "hx": torch.view_as_real(e.h[1].resolve_conj())})
    return got
