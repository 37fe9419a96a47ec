"""The work that programs have this library do, as measurable cases.

A case is one call sequence of the public interface on one input:

  step      coupled steps of one grid: the state goes in (pf_set_fields, device
            arrays), `steps` steps are taken, the whole state comes out
  update    the same with the mechanics off: the fused field update alone
  batch     coupled steps of several uneven grids advanced together
  implicit  one backward-Euler step at the paper's diffusivities
  finite    one step coupled to finite-strain mechanics (host arrays, as that
            interface has them)
  unet      one inference and one training step of the warm-start network
            (loss, gradient, Adam)

The state that goes in is a fresh one on every pass, so every pass does the
same work.  The mixed method's outputs are read as the single precision that
the method computes them in, and the displacement without its rigid
translation, which the periodic problem leaves free.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2111_11538_gb300 import Batch, FiniteStrainSimulation, Simulation, native, warmstart, workloads

DEV = "cuda" if torch.cuda.is_available() else "cpu"

STATE = ("phi_f", "phi_w", "xO", "xH", "xW", "theta", "phig", "u", "Ebar", "eps_p", "alpha", "sigma")
FIELDS = STATE[:7]
SUMS = ("sum_O", "sum_H", "sum_H2O", "removed_H2O", "supplied_H")


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def _grid(kind, shape, precision, steps, geometry, **more):
    nx, ny = shape[0], shape[1]
    return dict({"kind": kind, "ndim": len(shape), "nx": nx, "ny": ny, "nz": shape[2] if len(shape) == 3 else 1,
                 "precision": precision, "steps": steps, "geometry": geometry}, **more)


def listed():
    J2 = {"plasticity": 1}
    EL = {"plasticity": 0}

    def named(name, case):
        return dict(case, name=name)
    return [
        # the smallest grids anyone steps: parity checks, parameter scans, odd
        # sizes that no multigrid level divides (Jacobi-preconditioned CG);
        # FP64 solves run as tight as the parity checks'
        named("step2d_37x29_fp64", _grid("step", (37, 29), "fp64", 10, "core", rtol=1e-13, warm="prev", **J2)),
        # the 64^2 core-shell workload: a small particle in FP64
        named("step2d_64_fp64", _grid("step", (64, 64), "fp64", 10, "core", rtol=1e-13, warm="prev", **EL)),
        # the 512^2 core-shell workload with J2 flow, and its plain FP64 method
        # at half the size
        named("step2d_512_mixed", _grid("step", (512, 512), "mixed", 10, "core", rtol=1e-10, warm="extrap", **J2)),
        named("step2d_256_fp64", _grid("step", (256, 256), "fp64", 5, "core", rtol=1e-13, warm="extrap", **J2)),
        # the 2048^2 porous workload
        named("step2d_2048_mixed", _grid("step", (2048, 2048), "mixed", 2, "porous", rtol=1e-8, warm="extrap2", **EL)),
        # a small ragged 3D sample (Jacobi-preconditioned CG)
        named("step3d_53x47x61_mixed", _grid("step", (53, 47, 61), "mixed", 2, "core", rtol=1e-10, warm="prev", **J2)),
        # the 256^3 porous J2 workload, the benchmark's headline: the first step
        # of a run, whose solve starts from rest
        named("step3d_256_mixed", _grid("step", (256, 256, 256), "mixed", 1, "porous", rtol=1e-8, warm="extrap", **J2)),
        # field evolution without mechanics at the largest size
        named("update3d_256_mixed", _grid("update", (256, 256, 256), "mixed", 20, "porous")),
        # the batched workload: uneven 2D grids advanced together
        named("batch2d_16_mixed", {"kind": "batch", "count": 16, "nmin": 128, "nmax": 1024, "precision": "mixed",
                                   "steps": 2, "rtol": 1e-9, "warm": "extrap2"}),
        # a backward-Euler step at the diffusivities of the paper's Table 1
        named("implicit2d_256", {"kind": "implicit", "nx": 256, "ny": 256, "dt": 0.05, "rtol": 1e-13}),
        # a step coupled to finite-strain mechanics, 3D
        named("finite3d_48", {"kind": "finite", "ndim": 3, "nx": 48, "ny": 48, "nz": 48, "omega": 0.2, "nload": 2,
                              "newton_tol": 1e-11}),
        # a training step of the warm-start network on the batch it is trained with
        named("unet2d_train_8x128", {"kind": "unet", "nb": 8, "nx": 128, "ny": 128}),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case.  Coupled steps take any grid up to 160 nodes an axis in
    2D and 40 in 3D (Jacobi where the sizes do not coarsen), and above that
    the sizes a user gives a multigrid solve: multiples of 32 (2D, to 1536)
    and of 16 (3D, to 160); the other kinds take any size their interface
    does."""
    kind = rng.choice(["step2"] * 6 + ["step3"] * 4 + ["update"] * 4 + ["batch"] + ["implicit"] * 2 + ["finite"] * 2
                      + ["unet"] * 2)
    if kind == "step2":
        precision = rng.choice(["fp64", "mixed"])
        top = 256 if precision == "fp64" else 1536

        def size(n):
            return n if n <= 160 else 32 * max(5, round(n / 32))
        nx = _logint(rng, 24, top)
        ny = max(24, min(top, int(nx * rng.uniform(0.6, 1.6))))
        return _grid("step", (size(nx), size(ny)), precision, rng.randint(2, 6), rng.choice(["core", "porous"]),
                     rtol=1e-13 if precision == "fp64" else 1e-10, warm=rng.choice(["prev", "extrap"]),
                     plasticity=rng.randint(0, 1))
    if kind == "step3":
        n = _logint(rng, 16, 160)
        ax = [max(16, min(160, int(n * rng.uniform(0.7, 1.3)))) for _ in range(3)]
        if max(ax) > 40:
            ax = [16 * max(2, round(a / 16)) for a in ax]
        precision = "fp64" if max(ax) <= 40 and rng.random() < 0.3 else "mixed"
        return _grid("step", tuple(ax), precision, rng.randint(1, 3), rng.choice(["core", "porous"]),
                     rtol=1e-13 if precision == "fp64" else 1e-10, warm=rng.choice(["prev", "extrap"]), plasticity=rng.randint(0, 1))
    if kind == "update":
        nd = rng.choice([2, 3])
        lo, hi = (32, 2048) if nd == 2 else (16, 224)
        n = _logint(rng, lo, hi)
        ax = [max(lo, min(hi, int(n * rng.uniform(0.7, 1.3)))) for _ in range(nd)]
        return _grid("update", tuple(ax), rng.choice(["fp64", "mixed"]), rng.randint(4, 12), rng.choice(["core", "porous"]))
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 12), "nmin": 128, "nmax": rng.choice([256, 512]),
                "precision": "mixed", "steps": 2, "rtol": 1e-9, "warm": "extrap2"}
    if kind == "implicit":
        nx = _logint(rng, 40, 224)
        return {"kind": "implicit", "nx": nx, "ny": max(40, min(224, int(nx * rng.uniform(0.7, 1.3)))),
                "dt": rng.uniform(0.02, 0.06), "rtol": 1e-13}
    if kind == "finite":
        nd = rng.choice([2, 3])
        lo, hi = (24, 96) if nd == 2 else (12, 40)
        n = _logint(rng, lo, hi)
        ax = [max(lo, min(hi, int(n * rng.uniform(0.8, 1.25)))) for _ in range(nd)] + [1]
        return {"kind": "finite", "ndim": nd, "nx": ax[0], "ny": ax[1], "nz": ax[2], "omega": rng.uniform(0.1, 0.25),
                "nload": 2, "newton_tol": 1e-11}
    return {"kind": "unet", "nb": rng.randint(1, 12), "nx": 128 * rng.randint(1, 3), "ny": 64 * rng.randint(1, 4)}


def _shape(case):
    """Array shape (slowest axis first) of a grid case."""
    return (case["nz"], case["ny"], case["nx"]) if case.get("ndim", 2) == 3 else (case["ny"], case["nx"])


# ---------------------------------------------------------------------------
# Inputs: the two geometries of the workloads, drawn from a seed
# ---------------------------------------------------------------------------
def _step01(d, delta):
    return 0.5 * (1.0 + torch.tanh(d / delta))


def _axes(shape):
    return [torch.arange(n, dtype=torch.float64, device=DEV) + 0.5 for n in shape]


def _core_shell(shape, rng, delta=None):
    """A wuestite core with an iron shell in a gas box, a little off the
    centre; the gas away from the shell supplies hydrogen."""
    n = min(shape)
    delta = (3.0 if n >= 48 else n / 16.0) if delta is None else delta
    radius = rng.uniform(0.28, 0.32) * n
    shell = rng.uniform(0.055, 0.07) * n
    r = torch.zeros(shape, dtype=torch.float64, device=DEV)
    for ax, a in enumerate(_axes(shape)):
        o = a - (shape[ax] / 2.0 + rng.uniform(-0.02, 0.02) * n)
        view = [1] * len(shape)
        view[ax] = -1
        r = r + o.reshape(view) ** 2
    r = r.sqrt()
    phi_w = 1.0 - _step01(r - radius, delta)
    phi_f = _step01(r - radius, delta) - _step01(r - radius - shell, delta)
    mask = r > radius + shell + 2.0 * delta
    mob = torch.ones(shape, dtype=torch.float64, device=DEV)
    return _mixture(phi_f, phi_w, mob, mask)


def _mixture(phi_f, phi_w, mob, mask):
    phi_g = 1.0 - phi_f - phi_w
    return {"phi_f": phi_f, "phi_w": phi_w, "xO": 0.571 * phi_w + 0.01 * phi_f, "xH": 0.01 * phi_g,
            "xW": torch.zeros_like(phi_f), "mob": mob, "mask": mask.to(torch.uint8)}


def _porous(shape, rng, fraction=None):
    """Voronoi grains with lognormal pores, an iron rim around every pore and
    a supply layer on every outer face."""
    nd, cells = len(shape), float(np.prod(shape))
    grains = max(4, round(cells * (200 / 2048.0 ** 2 if nd == 2 else 500 / 256.0 ** 3)))
    median, sigma, frac = (12.0, 0.5, 0.2) if nd == 2 else (6.0, 0.4, 0.15)
    frac = frac if fraction is None else fraction
    box = torch.tensor(shape, dtype=torch.float32, device=DEV)
    seeds = torch.tensor(rng.uniform(0.0, 1.0, (grains, nd)), dtype=torch.float32, device=DEV) * box
    gmob = torch.tensor(rng.uniform(0.8, 1.2, grains), dtype=torch.float64, device=DEV)
    best = torch.full(shape, math.inf, dtype=torch.float32, device=DEV)
    which = torch.zeros(shape, dtype=torch.int32, device=DEV)
    axes = [a.float() for a in _axes(shape)]
    sq = []                                             # squared periodic distance along each axis, per grain
    for ax in range(nd):
        d = (axes[ax][None] - seeds[:, ax:ax + 1]).abs()
        sq.append(torch.minimum(d, box[ax] - d) ** 2)
    for g in range(grains):
        d = sq[0][g].reshape([-1] + [1] * (nd - 1))
        for ax in range(1, nd):
            view = [1] * nd
            view[ax] = -1
            d = d + sq[ax][g].reshape(view)
        near = d < best
        best = torch.where(near, d, best)
        which.masked_fill_(near, g)
    mob = gmob[which.long()]
    # balls until their volume covers the wanted fraction of the box
    # (overlapping at random: 1 - exp(-V / cells))
    want, volume = -math.log(1.0 - frac) * cells, 0.0
    dist = torch.full(shape, 1.0e3, dtype=torch.float64, device=DEV)
    top = 0.3 * min(shape)
    while volume < want:
        rad = min(top, math.exp(math.log(median) + sigma * rng.standard_normal()))
        volume += math.pi * rad * rad if nd == 2 else 4.0 / 3.0 * math.pi * rad ** 3
        c = rng.uniform(0.0, 1.0, nd) * np.array(shape)
        reach = min(int(math.ceil(rad + 12.0)), (min(shape) - 1) // 2)
        ids, rr = [], 0.0
        for ax in range(nd):
            i = np.arange(int(c[ax]) - reach, int(c[ax]) + reach + 1)
            o = torch.tensor((i + 0.5 - c[ax]) ** 2, device=DEV)
            view = [1] * nd
            view[ax] = -1
            rr = rr + o.reshape(view)
            ids.append(torch.tensor(i % shape[ax], device=DEV).reshape(view))
        dist[tuple(ids)] = torch.minimum(dist[tuple(ids)], rr.sqrt() - rad)
    phi_g = 1.0 - _step01(dist, 3.0)
    mask = torch.zeros(shape, dtype=torch.bool, device=DEV)
    for ax in range(nd):
        mask.narrow(ax, 0, 2).fill_(True)
        mask.narrow(ax, shape[ax] - 2, 2).fill_(True)
    phi_g = torch.where(mask, torch.ones_like(phi_g), phi_g)
    theta = 1.0 - _step01(dist - 3.0, 3.0)
    return _mixture((1.0 - phi_g) * theta, (1.0 - phi_g) * (1.0 - theta), mob, mask)


def _fields(case, seed):
    rng = np.random.default_rng(seed)
    return (_core_shell if case["geometry"] == "core" else _porous)(_shape(case), rng)


def _batch(case, seed):
    """Instances of a batch: sizes by the case (the seed changes geometry,
    pore fraction and prestress, not the amount of work)."""
    sizes = [s for s in (128, 256, 512, 1024) if case["nmin"] <= s <= case["nmax"]]
    pick = np.random.default_rng(case["count"])
    ns = [int(sizes[pick.integers(0, len(sizes))]) for _ in range(case["count"])]
    rng = np.random.default_rng(seed)
    return [{"n": n, "fraction": float(rng.uniform(0.05, 0.3)), "prestress": float(rng.uniform(0.0, 0.002)),
             "fields": None, "seed": int(rng.integers(1 << 30))} for n in ns]


def _params(case):
    if case["kind"] == "implicit":
        return workloads.paper_params(cg_rtol=case["rtol"])
    if case["kind"] == "finite":
        return workloads.params(plasticity=1, sigma_Y=0.002, H_hard=0.01)
    if case["kind"] == "update":
        return workloads.params(mechanics=0)
    return workloads.params(plasticity=case.get("plasticity", 0), cg_rtol=case["rtol"], warm_start=case["warm"])


# ---------------------------------------------------------------------------
# What a program holds before the call, and the call
# ---------------------------------------------------------------------------
def _centred(u):
    """A displacement (components last) without its mean."""
    return u - u.mean(tuple(range(u.ndim - 1)), keepdims=True)


class _Out:
    """Device arrays for the whole state of one grid and the pf_fields that
    points at them."""

    def __init__(self, shape, keys):
        nd = len(shape)
        last = {"u": (nd,), "eps_p": (4 if nd == 2 else 6,), "sigma": (4 if nd == 2 else 6,)}
        self.arrays, self.f = {}, native.pf_fields()
        for k in keys:
            s = ((3 if nd == 2 else 6),) if k == "Ebar" else tuple(shape) + last.get(k, ())
            t = torch.empty(s, dtype=torch.float64, device=DEV)
            self.arrays[k] = t
            name = {"xO": "x_O", "xH": "x_H", "xW": "x_H2O", "phig": "phi_g"}.get(k, k)
            setattr(self.f, name, ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double)))

    def read(self, single):
        res = dict(self.arrays)
        if "u" in res:
            res["u"] = _centred(res["u"])
        return {k: (t.float() if single else t) for k, t in res.items()}


def _ok(rc):
    if rc != native.PF_OK:
        raise RuntimeError("status %s" % native.STATUS_NAMES.get(rc, rc))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("step", "update", "implicit"):
        shape = _shape(case)
        if kind == "implicit":
            s["fields"] = _core_shell(shape, np.random.default_rng(seed))
            s["sim"] = Simulation(shape, _params(case), precision="fp64")
        else:
            s["fields"] = _fields(case, seed)
            s["sim"] = Simulation(shape, _params(case), precision=case["precision"])
        s["out"] = _Out(shape, FIELDS if kind == "update" else STATE)
    elif kind == "batch":
        inst = _batch(case, seed)
        base = _params(case)
        s["sim"] = Batch([(d["n"], d["n"]) for d in inst], [dict(base, prestress=d["prestress"]) for d in inst],
                         precision=case["precision"])
        s["fields"] = [_porous((d["n"], d["n"]), np.random.default_rng(d["seed"]), d["fraction"]) for d in inst]
        s["out"] = [_Out((d["n"], d["n"]), STATE) for d in inst]
    elif kind == "finite":
        shape = _shape(case)
        f = _core_shell(shape, np.random.default_rng(seed), delta=1.0)
        s["fields"] = {k: v.cpu().numpy() for k, v in f.items()}
        s["sim"] = FiniteStrainSimulation(shape, _params(case), case["omega"], nload=case["nload"],
                                          newton_tol=case["newton_tol"])
    else:
        x, t, theta = _unet_data(case, seed)
        s["net"] = warmstart.WarmStartNet(ndim=2)
        s["net"].set_loss("grad")
        s.update(x=x, t=t, theta=theta)
    if DEV == "cuda":
        torch.cuda.synchronize()
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("step", "update", "implicit"):
        sim, out = state["sim"], state["out"]
        sim.set_fields(state["fields"], where="device")
        if kind == "implicit":
            sim.step_implicit(1, case["dt"])
        else:
            sim.step(case["steps"])
        d = sim.diagnostics()
        _ok(native.pf_get_fields(sim.h, out.f, native.PF_DEVICE))
        res = out.read(case.get("precision") == "mixed")
        res.update({k: d[k] for k in SUMS})
        return res
    if kind == "batch":
        sim = state["sim"]
        for i, f in enumerate(state["fields"]):
            sim.set_fields(i, f, where="device")
        sim.step(case["steps"])
        d = [sim.diagnostics(i) for i in range(len(state["out"]))]
        for i, o in enumerate(state["out"]):
            _ok(native.pf_batch_get_fields(sim.h, i, o.f, native.PF_DEVICE))
        parts = [o.read(True) for o in state["out"]]
        res = {k: torch.cat([p[k].reshape(-1) for p in parts]) for k in STATE}
        res.update({k: np.array([x[k] for x in d], dtype=np.float32) for k in SUMS})
        return res
    if kind == "finite":
        sim = state["sim"]
        sim.set_fields(state["fields"])
        sim.step(1)
        res = dict(sim.get_fields(keys=FIELDS))
        res.update(u=_centred(sim.u), Fbar=sim.Fbar, FP=sim.FP, epsP=sim.epsP)
        return res
    net = state["net"]
    net.set_params(state["theta"])
    y = net.forward(state["x"])
    loss, grad = net.loss_grad(state["x"], state["t"], want_grad=True)
    net.adam_step(1e-3)
    return {"loss": loss, "grad": grad, "forward": y}


def _unet_data(case, seed):
    """Smoothed phase fields as inputs, a smooth random displacement rate as
    target, He-uniform weights."""
    nb, ny, nx = case["nb"], case["ny"], case["nx"]
    g = torch.Generator(device="cpu").manual_seed(int(seed))

    def smooth(c):
        z = torch.fft.rfft2(torch.randn(nb, c, ny, nx, generator=g, dtype=torch.float64).to(DEV))
        ky = torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[:, None]
        kx = torch.fft.rfftfreq(nx, device=DEV, dtype=torch.float64)[None]
        v = torch.fft.irfft2(z * torch.exp(-200.0 * (kx * kx + ky * ky)), s=(ny, nx))
        return v / v.std()
    s = smooth(4)
    wg = torch.sigmoid(4.0 * (s[:, 0] - 1.0))
    wf = (1.0 - wg) * torch.sigmoid(4.0 * s[:, 1])
    p = torch.rand(nb, 1, 1, generator=g, dtype=torch.float64).to(DEV).expand(nb, ny, nx) * 0.4
    x = torch.stack([wf, wg, p, 0.1 * s[:, 2]], dim=-1).float().contiguous()
    t = smooth(2).permute(0, 2, 3, 1).float().contiguous()
    parts = []
    for ci, co, taps in _unet_shapes():
        b = math.sqrt(6.0 / (ci * taps))
        parts += [(2.0 * torch.rand(ci * co * taps, generator=g) - 1.0) * b, 0.05 * torch.randn(co, generator=g)]
    return x, t, torch.cat(parts).numpy().astype(np.float32)


def _unet_shapes():
    ch, prev, out = warmstart.DEFAULT_CHANNELS, warmstart.INPUT_CHANNELS, []
    for c in ch:
        out += [(prev, c, 9), (c, c, 9)]
        prev = c
    for l in range(len(ch) - 2, -1, -1):
        out += [(ch[l] + ch[l + 1], ch[l], 9), (ch[l], ch[l], 9)]
    return out + [(ch[0], 2, 1)]


# ---------------------------------------------------------------------------
# What a pass cannot do without.  The state in and out once per pass; per
# step one read of the fields and one write of those that change, the moduli
# and eigenstress, the return map; per solve ten applications of the operator
# with the vectors of a CG iteration, which is what a preconditioner of
# size-independent quality needs for these tolerances.
# ---------------------------------------------------------------------------
def _work_cells(cells, nd, word, steps, mechanics):
    io = (8 + (nd + 5 if mechanics else 0)) * 16
    per, fl = 12 * word + 1, 300
    if mechanics:
        per += (11 if nd == 2 else 15) * word + (20 if nd == 2 else 28) * word + 10 * (16 if nd == 2 else 24) * word
        fl += 10 * (110 if nd == 2 else 430)
    return {"bytes": cells * (io + steps * per), "flops": cells * steps * fl}


def work(case):
    kind = case["kind"]
    word = 4 if case.get("precision") == "mixed" else 8
    if kind in ("step", "update"):
        return _work_cells(float(np.prod(_shape(case))), case["ndim"], word, case["steps"], kind == "step")
    if kind == "batch":
        cells = float(sum(d["n"] ** 2 for d in _batch(case, 0)))
        return _work_cells(cells, 2, word, case["steps"], True)
    if kind == "implicit":
        # four Newton steps, fifteen Krylov vectors each (exact block solves)
        cells = float(case["nx"] * case["ny"])
        return {"bytes": cells * 4 * 8 * 4 * 15 * 4, "flops": cells * 4 * 15 * (400 + 15 * 16)}
    if kind == "finite":
        # eight Newton steps of fifty products each: 2^d Gauss points, the
        # tangent of a cell applied to its corner displacements
        cells, nd = float(np.prod(_shape(case))), case["ndim"]
        return {"bytes": cells * 8 * 50 * (24 * nd + 80), "flops": cells * 8 * 50 * (2 ** nd) * 300}
    px = float(case["nb"] * case["nx"] * case["ny"])
    mac = 0.0
    convs = _unet_shapes()
    levels = [0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0]
    act = 0.0
    for (ci, co, taps), lv in zip(convs, levels):
        mac += px / 4 ** lv * ci * co * taps
        act += px / 4 ** lv * (ci + co)
    return {"bytes": 3 * 2 * act, "flops": 4 * 2 * mac}


# ---------------------------------------------------------------------------
# The same results in 64 bits, from the definitions
# ---------------------------------------------------------------------------
def _h(x):
    return x * x * x * (x * (6.0 * x - 15.0) + 10.0)


def _hp(x):
    return 30.0 * x * x * (1.0 - x) * (1.0 - x)


def _m(x):
    return x * x * (1.0 - x) * (1.0 - x)


def _nb(v, ax, s):
    """v at the neighbour c + s along axis ax (arrays slowest axis first)."""
    return torch.roll(v, -s, dims=ax)


def _rates(p, th, pg, xO, xH, xW, mob, trE, devE2):
    """Right-hand sides of the field relations."""
    nd, c = th.dim(), p["c_chem"]
    Ks, Gs = p["E_s"] / (3 * (1 - 2 * p["nu"])), p["E_s"] / (2 * (1 + p["nu"]))
    Kg = Ks * p["E_g_ratio"]
    hg = _h(pg)
    sol = 1.0 - hg
    Wf, Ww = sol * _h(th), sol * (1.0 - _h(th))

    def lap(v):
        return sum(_nb(v, a, 1) + _nb(v, a, -1) - 2.0 * v for a in range(nd))

    def div(k, v):
        return sum(0.5 * (k + _nb(k, a, s)) * (_nb(v, a, s) - v) for a in range(nd) for s in (1, -1))
    f1 = Wf * (((4 * 163.708 * xO - 3 * 182.510) * xO + 2 * 90.573) * xO - 36.031) + Ww * (2 * 173.263 * xO - 213.460) \
        + hg * 2.0e3 * xO
    f2 = Wf * ((12 * 163.708 * xO - 6 * 182.510) * xO + 2 * 90.573) + Ww * (2 * 173.263) + hg * 2.0e3
    mu = c * f1 - p["kappa_O"] * lap(xO)
    M = (sol * p["D_O_s"] + hg * p["D_O_g"]) / (c * f2)
    ff = (((163.708 * xO - 182.510) * xO + 90.573) * xO - 36.031) * xO - 4.372
    fw = (173.263 * xO - 213.460) * xO + 41.953
    Kmix = sol * Ks + hg * Kg
    force = sol * _hp(th) * c * (ff - fw) + 2 * p["w"] * 2.0 * th * (1.0 - th) * (1.0 - 2.0 * th) \
        - 3.0 * p["eig0"] * sol * _hp(th) * Kmix * trE
    r = _m(pg) * p["k_for"] * xO * xH * (xW < 1.0)
    return (-0.5 * p["L"] * mob * (force - 2 * p["eps_phi"] * lap(th)), div(M, mu) - r,
            div(sol * p["D_H_s"] + hg * p["D_H_g"], xH) - 2.0 * r, div(sol * p["D_W_s"] + hg * p["D_W_g"], xW) + r)


def _dt(p, nd):
    D = max(p["D_%s_%s" % (s, q)] for s in "OHW" for q in "sg")
    xm = 6.0 * 182.510 / (24.0 * 163.708)
    fmin = min(12.0 * 163.708 * xm * xm - 6.0 * 182.510 * xm + 2.0 * 90.573, 2.0 * 173.263)
    return 0.2 * min(1.0 / (2 * nd * D), 2.0 / (D / (p["c_chem"] * fmin) * p["kappa_O"] * (4.0 * nd) ** 2),
                     1.0 / (1.2 * p["L"] * (2 * nd * p["eps_phi"] + 2 * p["w"])),
                     16.0 / (p["k_for"] * (0.571 + 2 * p["xH_bc"])))


class _Mechanics:
    """Q1 voxel elements on the periodic grid, the displacement and the mean
    strain by conjugate gradients with the homogeneous operator's inverse
    (Fourier) as preconditioner."""

    def __init__(self, p, shape):
        self.p, self.shape, self.nd = p, tuple(shape), len(shape)
        nd, na = self.nd, 1 << self.nd
        nv = 3 if nd == 2 else 6
        g = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
        pairs = [(0, 1)] if nd == 2 else [(1, 2), (0, 2), (0, 1)]
        ML, MM = np.zeros((nv, nv)), np.eye(nv)
        ML[:nd, :nd] = 1.0
        MM[:nd, :nd] *= 2.0
        Kl, Km, Bb = np.zeros((na * nd, na * nd)), np.zeros((na * nd, na * nd)), np.zeros((nv, na * nd))
        for q in range(na):
            xi = [g[(q >> l) & 1] for l in range(nd)]
            B = np.zeros((nv, na * nd))
            for a in range(na):
                dn = [np.prod([(1.0 if (a >> l) & 1 else -1.0) if l == k else (xi[l] if (a >> l) & 1 else 1.0 - xi[l])
                               for l in range(nd)]) for k in range(nd)]
                for k in range(nd):
                    B[k, a * nd + k] = dn[k]
                for r, (i, j) in enumerate(pairs):
                    B[nd + r, a * nd + i] = dn[j]
                    B[nd + r, a * nd + j] = dn[i]
            Kl += B.T @ ML @ B / na
            Km += B.T @ MM @ B / na
            Bb += B / na
        t = lambda m: torch.tensor(m, dtype=torch.float64, device=DEV)    # noqa: E731
        self.Kl, self.Km, self.Bb, self.ML, self.MM, self.nv = t(Kl), t(Km), t(Bb), t(ML), t(MM), nv
        nu, E = p["nu"], p["E_s"]
        self.Ks, self.Gs = E / (3 * (1 - 2 * nu)), E / (2 * (1 + nu))
        # Fourier symbol of the homogeneous operator
        one = torch.ones(self.shape, dtype=torch.float64, device=DEV)
        cols = []
        for k in range(nd):
            e = torch.zeros((nd,) + self.shape, dtype=torch.float64, device=DEV)
            e[(k,) + (0,) * nd] = 1.0
            q = self._scatter(self._element(e, one * (self.Ks - 2 * self.Gs / 3), one * self.Gs))
            cols.append(torch.fft.rfftn(q, dim=tuple(range(1, nd + 1))))
        S = torch.stack(cols, dim=1)
        S = S.permute(tuple(range(2, nd + 2)) + (0, 1)).contiguous()
        S[(0,) * nd] = torch.eye(nd, dtype=S.dtype, device=DEV)
        S = torch.linalg.inv(S)
        S[(0,) * nd] = 0.0
        self.Sinv = S

    def _corners(self, u):
        nd = self.nd
        return torch.cat([torch.roll(u, tuple(-((a >> l) & 1) for l in range(nd)), dims=tuple(nd - l for l in range(nd)))
                          for a in range(1 << nd)])

    def _scatter(self, f):
        nd = self.nd
        out = 0.0
        for a in range(1 << nd):
            out = out + torch.roll(f[a * nd:(a + 1) * nd], tuple((a >> l) & 1 for l in range(nd)),
                                   dims=tuple(nd - l for l in range(nd)))
        return out

    def _mul(self, m, v):
        return (m @ v.reshape(v.shape[0], -1)).reshape((m.shape[0],) + self.shape)

    def _element(self, u, lam, mu):
        ue = self._corners(u)
        return lam * self._mul(self.Kl, ue) + mu * self._mul(self.Km, ue)

    def _stress(self, e, lam, mu):
        return lam * self._mul(self.ML, e) + mu * self._mul(self.MM, e)

    def apply(self, u, E, lam, mu):
        ue = self._corners(u)
        ef = E.reshape((-1,) + (1,) * self.nd).expand((self.nv,) + self.shape)
        f = lam * self._mul(self.Kl, ue) + mu * self._mul(self.Km, ue) + self._mul(self.Bb.T, self._stress(ef, lam, mu))
        sE = self._stress(self._mul(self.Bb, ue) + ef, lam, mu)
        return self._scatter(f), sE.reshape(self.nv, -1).sum(1)

    def solve(self, lam, mu, sig, prestress, u, E, rtol=1e-13):
        nd, N = self.nd, float(np.prod(self.shape))
        dims = tuple(range(1, nd + 1))
        bu = self._scatter(self._mul(self.Bb.T, sig))
        bE = sig.reshape(self.nv, -1).sum(1)
        bE[:nd] -= N * prestress
        dE = float(lam.sum()) * torch.diagonal(self.ML) + float(mu.sum()) * torch.diagonal(self.MM)

        def prec(ru, rE):
            z = torch.fft.rfftn(ru, dim=dims)
            z = torch.einsum("...ij,j...->i...", self.Sinv, z)
            return torch.fft.irfftn(z, s=self.shape, dim=dims), rE / dE

        def dot(a, b):
            return (a[0] * b[0]).sum() + (a[1] * b[1]).sum()
        Au, AE = self.apply(u, E, lam, mu)
        r = (bu - Au, bE - AE)
        stop = rtol * rtol * float(dot((bu, bE), (bu, bE)))
        z = prec(*r)
        p = z
        rz = dot(r, z)
        for it in range(4000):
            if it % 8 == 0 and float(dot(r, r)) <= stop:
                break
            q = self.apply(p[0], p[1], lam, mu)
            al = rz / dot(p, q)
            u, E = u + al * p[0], E + al * p[1]
            r = (r[0] - al * q[0], r[1] - al * q[1])
            z = prec(*r)
            rn = dot(r, z)
            p = (z[0] + rn / rz * p[0], z[1] + rn / rz * p[1])
            rz = rn
        return u, E

    def step(self, th, pg, u, E, ep, alpha, plastic):
        """Equilibrium and one radial return: the new u, E, ep, alpha, then
        sigma, tr eps_e and |dev eps_e|^2.  ep, sigma: components last to
        first axis, in the library's order (2D xx yy zz xy)."""
        p, nd = self.p, self.nd
        hg = _h(pg)
        Wf = (1.0 - hg) * _h(th)
        K = (1.0 - hg) * self.Ks + hg * self.Ks * p["E_g_ratio"]
        G = (1.0 - hg) * self.Gs + hg * self.Gs * p["E_g_ratio"]
        lam = K - 2.0 * G / 3.0
        full = torch.zeros((6,) + self.shape, dtype=torch.float64, device=DEV)
        full[list(range(6)) if nd == 3 else [0, 1, 2, 5]] = ep
        es = full.clone()
        es[:3] += p["eig0"] * Wf
        tr = es[0] + es[1] + es[2]
        sg = 2.0 * G * es
        sg[:3] += lam * tr
        sig = sg if nd == 3 else sg[[0, 1, 5]]
        u, E = self.solve(lam, G, sig.contiguous(), p["prestress"], u, E)
        e = self._mul(self.Bb, self._corners(u)) + E.reshape((-1,) + (1,) * nd)
        et = torch.zeros_like(full)
        if nd == 3:
            et[:3], et[3:] = e[:3], 0.5 * e[3:]
        else:
            et[0], et[1], et[5] = e[0], e[1], 0.5 * e[2]
        ee = et - es
        w = torch.tensor([1.0, 1, 1, 2, 2, 2], dtype=torch.float64, device=DEV).reshape((6,) + (1,) * nd)
        tr = ee[0] + ee[1] + ee[2]
        dev = ee.clone()
        dev[:3] -= tr / 3.0
        if plastic:
            nrm = (w * dev * dev).sum(0).sqrt()
            s23 = math.sqrt(2.0 / 3.0)
            f = 2.0 * G * nrm - s23 * (p["sigma_Y"] + p["H_hard"] * alpha)
            dl = torch.clamp(f, min=0.0) / (2.0 * G + s23 * p["H_hard"])
            d = dl / torch.clamp(nrm, min=1e-300) * dev
            full, dev, alpha = full + d, dev - d, alpha + dl
        n2 = (w * dev * dev).sum(0)
        so = 2.0 * G * dev
        so[:3] += K * tr
        keep = list(range(6)) if nd == 3 else [0, 1, 2, 5]
        return u, E, full[keep], alpha, so[keep], tr, n2


def _split(f):
    s = f["phi_f"] + f["phi_w"]
    th = torch.where(s > 0.0, f["phi_f"] / torch.where(s > 0.0, s, torch.ones_like(s)), torch.zeros_like(s))
    return th, 1.0 - s


def _coupled(p, f, steps, mechanics, plastic):
    """`steps` explicit steps in 64 bits from the fields f."""
    th, pg = _split(f)
    xO, xH, xW, mob = f["xO"], f["xH"], f["xW"], f["mob"]
    mask = f["mask"].bool()
    shape, nd = tuple(th.shape), th.dim()
    dt = _dt(p, nd)
    zero = torch.zeros_like(th)
    trE, dev2 = zero, zero
    removed, supplied = 0.0, 0.0
    npl, nv = (4, 3) if nd == 2 else (6, 6)
    u = torch.zeros((nd,) + shape, dtype=torch.float64, device=DEV)
    E = torch.zeros(nv, dtype=torch.float64, device=DEV)
    ep, alpha, sig = torch.zeros((npl,) + shape, dtype=torch.float64, device=DEV), zero, None
    mech = _Mechanics(p, shape) if mechanics else None
    for _ in range(steps):
        if mech:
            u, E, ep, alpha, sig, trE, dev2 = mech.step(th, pg, u, E, ep, alpha, plastic)
        R = _rates(p, th, pg, xO, xH, xW, mob, trE, dev2)
        th, xO, xH, xW = th + dt * R[0], xO + dt * R[1], xH + dt * R[2], xW + dt * R[3]
        removed += float(xW[mask].sum())
        supplied += float((p["xH_bc"] - xH[mask]).sum())
        xH = torch.where(mask, torch.full_like(xH, p["xH_bc"]), xH)
        xW = torch.where(mask, zero, xW)
    res = {"phi_f": (1.0 - pg) * th, "phi_w": (1.0 - pg) * (1.0 - th), "xO": xO, "xH": xH, "xW": xW, "theta": th,
           "phig": pg, "sum_O": float(xO.sum()), "sum_H": float(xH.sum()), "sum_H2O": float(xW.sum()),
           "removed_H2O": removed, "supplied_H": supplied}
    if mech:
        last = tuple(range(1, nd + 1)) + (0,)
        res.update(u=_centred(u.permute(last)).contiguous(), Ebar=E, eps_p=ep.permute(last).contiguous(), alpha=alpha,
                   sigma=sig.permute(last).contiguous())
    return res


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "update"):
        cells = float(np.prod(_shape(case)))
        if kind == "step" and case["ndim"] == 3 and cells * case["steps"] > 8e6:
            return None                              # a 64-bit solve of that size takes over 20 seconds
        p = _params(case)
        return _coupled(p, _fields(case, seed), case["steps"], kind == "step", bool(p["plasticity"]))
    if kind == "batch":
        base, parts = _params(case), []
        for d in _batch(case, seed):
            f = _porous((d["n"], d["n"]), np.random.default_rng(d["seed"]), d["fraction"])
            parts.append(_coupled(dict(base, prestress=d["prestress"]), f, case["steps"], True, False))
        res = {k: torch.cat([q[k].reshape(-1) for q in parts]) for k in STATE}
        res.update({k: np.array([q[k] for q in parts]) for k in SUMS})
        return res
    if kind == "implicit":
        return _implicit(case, seed)
    if kind == "finite":
        return _finite(case, seed)
    return _unet(case, seed)


def _implicit(case, seed):
    """One backward-Euler step: Newton's method, each system by GMRES with
    Chebyshev-preconditioned diffusion blocks, tangents in forward mode."""
    p, f = _params(case), _core_shell(_shape(case), np.random.default_rng(seed))
    th, pg = _split(f)
    shape, dt = tuple(th.shape), case["dt"]
    mask, mob = f["mask"].bool(), f["mob"]
    zero = torch.zeros_like(th)
    mech = _Mechanics(p, shape)
    z3 = torch.zeros(3, dtype=torch.float64, device=DEV)
    u, E, ep, alpha, sig, trE, dev2 = mech.step(th, pg, torch.zeros((2,) + shape, dtype=torch.float64, device=DEV), z3,
                                                torch.zeros((4,) + shape, dtype=torch.float64, device=DEV), zero, False)
    y0 = torch.stack([th, f["xO"], f["xH"], f["xW"]])
    held = torch.stack([torch.zeros_like(mask), torch.zeros_like(mask), mask, mask])
    hv = torch.zeros_like(y0)
    hv[2] = torch.where(mask, torch.full_like(zero, p["xH_bc"]), zero)

    def F(y):
        R = torch.stack(_rates(p, y[0], pg, y[1], y[2], y[3], mob, trE, dev2))
        return torch.where(held, y - hv, y - y0 - dt * R)
    hg = _h(pg)
    D = torch.stack([zero] + [(1.0 - hg) * p["D_%s_s" % s] + hg * p["D_%s_g" % s] for s in "OHW"])
    cth = dt * p["L"] * p["eps_phi"] * mob
    faces = [torch.stack([cth, *(0.5 * dt * (D[b] + _nb(D[b], a, s)) for b in (1, 2, 3))]) for a in (0, 1) for s in (1, -1)]
    faces = [torch.where(held, torch.zeros_like(k), k) for k in faces]
    dirs = [(a, s) for a in (1, 2) for s in (1, -1)]
    off = sum(faces)
    dg = 1.0 + off
    rad = (off / dg).reshape(4, -1).max(1).values.clamp(min=1e-12).reshape(4, 1, 1)

    def prec(v, degree=32):
        z, r, d, rho = torch.zeros_like(v), v, v / dg, rad
        for _ in range(degree - 1):
            z = z + d
            q = d
            for k, (a, s) in zip(faces, dirs):
                q = q + k * (d - _nb(d, a, s))
            r = r - q
            rho1 = 1.0 / (2.0 / rad - rho)
            d = rho1 * rho * d + 2.0 * rho1 / rad * r / dg
            rho = rho1
        return z + d
    y = torch.where(held, hv, y0)
    for newton in range(12):
        Fy = F(y)
        if float(Fy.abs().max()) <= 1e-14:
            break
        x, r = torch.zeros_like(y), Fy
        goal = 1e-6 * float(Fy.norm())
        for _ in range(40):
            beta = float(r.norm())
            if beta <= goal:
                break
            m = 60
            V, H = torch.zeros((m + 1, y.numel()), dtype=torch.float64, device=DEV), np.zeros((m + 1, m))
            V[0] = r.reshape(-1) / beta
            for j in range(m):
                z = prec(V[j].reshape(y.shape))
                w = torch.func.jvp(F, (y,), (z,))[1].reshape(-1)
                h = V[:j + 1] @ w
                w = w - h @ V[:j + 1]
                h2 = V[:j + 1] @ w
                w = w - h2 @ V[:j + 1]
                H[:j + 1, j] = (h + h2).cpu().numpy()
                H[j + 1, j] = float(w.norm())
                V[j + 1] = w / H[j + 1, j]
                c, res = np.linalg.lstsq(H[:j + 2, :j + 1], beta * np.eye(j + 2)[0], rcond=None)[:2]
                if len(res) == 0 or res[0] <= goal * goal:
                    break
            x = x + prec((torch.tensor(c, device=DEV) @ V[:j + 1]).reshape(y.shape))
            r = Fy - torch.func.jvp(F, (y,), (x,))[1]
        y = y - x
        if float(x.abs().max()) <= 1e-12 * max(1.0, float(y.abs().max())):
            break
    last = (1, 2, 0)
    R = _rates(p, y[0], pg, y[1], y[2], y[3], mob, trE, dev2)
    return {"phi_f": (1.0 - pg) * y[0], "phi_w": (1.0 - pg) * (1.0 - y[0]), "xO": y[1], "xH": y[2], "xW": y[3],
            "theta": y[0], "phig": pg, "u": _centred(u.permute(last)).contiguous(), "Ebar": E, "eps_p": ep.permute(last).contiguous(), "alpha": alpha,
            "sigma": sig.permute(last).contiguous(), "sum_O": float(y[1].sum()), "sum_H": float(y[2].sum()),
            "sum_H2O": float(y[3].sum()), "removed_H2O": float((y0[3] + dt * R[3])[mask].sum()),
            "supplied_H": float((p["xH_bc"] - y0[2] - dt * R[2])[mask].sum())}


def _finite(case, seed):
    """The finite-strain equilibrium of the step: Newton's method on the
    energy, each system by conjugate gradients with the small-strain
    homogeneous operator's inverse; the other outputs follow from the return
    map, which is not restated here."""
    p, shape = _params(case), _shape(case)
    f = _core_shell(shape, np.random.default_rng(seed), delta=1.0)
    th, pg = _split(f)
    nd, na, N = len(shape), 1 << len(shape), float(np.prod(shape))
    mech = _Mechanics(p, shape)
    hg = _h(pg)
    Wf = (1.0 - hg) * _h(th)
    K = ((1.0 - hg) + hg * p["E_g_ratio"]) * mech.Ks
    G = ((1.0 - hg) + hg * p["E_g_ratio"]) * mech.Gs
    g = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
    dN = np.zeros((na, nd, na))                                       # [Gauss point, axis, corner]
    for q in range(na):
        xi = [g[(q >> l) & 1] for l in range(nd)]
        for a in range(na):
            for k in range(nd):
                dN[q, k, a] = np.prod([(1.0 if (a >> l) & 1 else -1.0) if l == k
                                       else (xi[l] if (a >> l) & 1 else 1.0 - xi[l]) for l in range(nd)])
    dN = torch.tensor(dN, device=DEV)
    idx = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)] if nd == 3 else [(0, 0), (1, 1), (0, 1)]
    sym = torch.zeros((len(idx), 3, 3), dtype=torch.float64, device=DEV)
    for r, (i, j) in enumerate(idx):
        sym[r, i, j] = sym[r, j, i] = 1.0
    dims = tuple(range(1, nd + 1))
    hold = torch.ones((nd,) + shape, dtype=torch.float64, device=DEV)
    hold[(slice(None),) + (0,) * nd] = 0.0

    def forces(u, e, dT):
        """d(energy)/d(u, e) from the first Piola stress at the Gauss points
        (leading axis: the points of a cell)."""
        s = dT ** (-1.0 / 3.0)
        fb = torch.einsum("r,rij->ij", e, sym)
        ue = mech._corners(u).reshape(na, nd, -1)
        Gr = torch.einsum("qka,ain->qikn", dN, ue)
        F = torch.nn.functional.pad(Gr, (0, 0, 0, 3 - nd, 0, 3 - nd)) + fb[None, :, :, None]
        if nd == 2:
            F = F + torch.diag(torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device=DEV))[None, :, :, None]
        s, dTn, Kn, Gn = s.reshape(-1), dT.reshape(-1), K.reshape(-1), G.reshape(-1)
        X = s * F
        r1, r2 = torch.roll(X, -1, 1), torch.roll(X, -2, 1)
        cof = torch.roll(r1, -1, 2) * torch.roll(r2, -2, 2) - torch.roll(r1, -2, 2) * torch.roll(r2, -1, 2)
        J = (X[:, 0] * cof[:, 0]).sum(1)
        I1 = (X * X).sum((1, 2))
        a2 = Gn * J ** (-2.0 / 3.0)
        a1 = 0.5 * Kn * (J * J - 1.0) / J - a2 * I1 / (3.0 * J)
        P = (dTn * s) * (a1[:, None, None] * cof + a2[:, None, None] * X)
        fc = torch.einsum("qka,qikn->ain", dN / na, P[:, :nd, :nd])
        fe = torch.einsum("rij,ij->r", sym, P.sum((0, 3))) / na
        return hold * mech._scatter(fc.reshape((na * nd,) + shape)), fe

    def prec(ru, re):
        z = torch.einsum("...ij,j...->i...", mech.Sinv, torch.fft.rfftn(ru, dim=dims))
        z = torch.fft.irfftn(z, s=shape, dim=dims)
        return hold * (z - z[(slice(None),) + (0,) * nd].reshape((nd,) + (1,) * nd)), re / (float(K.sum() + 4 * G.sum() / 3))

    def dot(a, b):
        return (a[0] * b[0]).sum() + (a[1] * b[1]).sum()
    u = torch.zeros((nd,) + shape, dtype=torch.float64, device=DEV)
    e = torch.tensor([1.0] * nd + [0.0] * (len(idx) - nd), dtype=torch.float64, device=DEV)
    for load in range(1, case["nload"] + 1):
        dT = 1.0 - Wf * (case["omega"] * load / case["nload"])
        for it in range(8):
            ru, re = forces(u, e, dT)
            worst = max(float(ru.abs().max()), float(re.abs().max()) / N)
            if worst <= (5e-16 if load == case["nload"] else 1e-8):
                break
            r = (-ru, -re)
            z = prec(*r)
            d, rz, x = z, dot(r, z), (torch.zeros_like(u), torch.zeros_like(e))
            stop = 1e-5 * math.sqrt(float(dot(r, r)))
            for k in range(400):
                q = torch.func.jvp(lambda a, b: forces(a, b, dT), (u, e), d)[1]
                al = rz / dot(d, q)
                x = (x[0] + al * d[0], x[1] + al * d[1])
                r = (r[0] - al * q[0], r[1] - al * q[1])
                if k % 4 == 3 and math.sqrt(float(dot(r, r))) <= stop:
                    break
                z = prec(*r)
                rn = dot(r, z)
                d, rz = (z[0] + rn / rz * d[0], z[1] + rn / rz * d[1]), rn
            u, e = u + x[0], e + x[1]
            if float(x[0].abs().max()) <= 1e-13:
                break
    fb = torch.einsum("r,rij->ij", e, sym)[:nd, :nd]
    res = {k: None for k in FIELDS + ("FP", "epsP")}
    res.update(phig=pg, u=_centred(u.reshape(nd, -1).T).contiguous(), Fbar=fb.contiguous())
    return res


def _unet(case, seed):
    """The network, its loss and its gradient in 64 bits."""
    x, t, theta = _unet_data(case, seed)
    w = torch.tensor(theta, dtype=torch.float64, device=DEV, requires_grad=True)
    ch, shapes, P, o = warmstart.DEFAULT_CHANNELS, _unet_shapes(), [], 0
    for ci, co, taps in shapes:
        k = 3 if taps > 1 else 1
        P.append((w[o:o + ci * co * taps].reshape(co, ci, k, k), w[o + ci * co * taps:o + ci * co * taps + co]))
        o += ci * co * taps + co

    def conv(v, k):
        W, b = P[k]
        out = b.reshape(1, -1, 1, 1)
        for iy in range(W.shape[2]):
            for ix in range(W.shape[3]):
                h = W.shape[2] // 2
                out = out + torch.einsum("oc,ncyx->noyx", W[:, :, iy, ix], torch.roll(v, (h - iy, h - ix), dims=(2, 3)))
        return out

    def block(v, k):
        return torch.relu(conv(torch.relu(conv(v, k)), k + 1))
    with torch.enable_grad():
        v, skips, k = x.double().permute(0, 3, 1, 2), [], 0
        for l in range(len(ch)):
            if l:
                v = v.reshape(v.shape[0], v.shape[1], v.shape[2] // 2, 2, v.shape[3] // 2, 2).mean((3, 5))
            v = block(v, k)
            skips.append(v)
            k += 2
        for l in range(len(ch) - 2, -1, -1):
            v = block(torch.cat([skips[l], v.repeat_interleave(2, 2).repeat_interleave(2, 3)], 1), k)
            k += 2
        y = conv(v, k)
        err = y - t.double().permute(0, 3, 1, 2)
        wt = 0.01 + 0.99 * (1.0 - x[..., 1:2].double().permute(0, 3, 1, 2))
        loss = sum((wt * (torch.roll(err, -1, dims=a) - err) ** 2).sum() for a in (2, 3)) / err.numel()
        grad, = torch.autograd.grad(loss, w)
    return {"loss": float(loss.detach()), "grad": grad, "forward": y.detach().permute(0, 2, 3, 1).contiguous()}
