"""The work that programs built on this library have it do, as cases that can be timed
and compared: single lattices and batches stepped through the public binding, the
whole-batch upload-step-diagnose loop, and the discrete adjoint.

Every pass runs what a user's time loop runs between two looks at the result: some
timesteps, the diagnostics, and (where the program keeps snapshots) the fields.
The 64-bit values of the same pass come from ``exact``, a plain torch FP64
restatement of the scheme over a flat list of sites (no kernel of this package),
with torch's own autograd for the gradients.

Parameters lie in the range where the scheme itself is stable (tau 0.8 .. 1.2,
G -5.2 .. -4.8; the threads at paper scale use tau = 1, G = -6).
"""
from __future__ import annotations

import ctypes
import math
from functools import lru_cache

import numpy as np
import torch

from paper_1310_1871_gb300 import amlbm, inputs

F64 = torch.float64
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
# floating-point operations of one site update (moments, force stencils, collision,
# sources, psi), and of its transposed step
FLOPS, FLOPS_ADJ = 300, 500


# ------------------------------------------------------------------ the cases --
def listed():
    return [
        # the paper's verification drop in the parity form, monitored every 20 steps:
        # the smallest lattice a program steps, bound by latency
        dict(name="static_drop_f64", kind="lattice", flow="drop", Nz=64, Nr=32, storage="f64", steps=20),
        # the oscillating drop's a2(t) series (256 x 128, R = 40), the everyday single run
        dict(name="osc_drop_f32", kind="lattice", flow="drop", Nz=256, Nr=128, storage="f32", steps=50),
        # Hagen-Poiseuille pipe: no-slip wall and body force, odd sizes
        dict(name="pipe_odd_f32", kind="lattice", flow="pipe", Nz=255, Nr=65, storage="f32", steps=50),
        # flow between two discs (Sec. III.2): z walls, inlet and outlet rows, FP64
        dict(name="discs_f64", kind="lattice", flow="discs", Nz=32, Nr=111, storage="f64", steps=50),
        # the 64-drop sweep (R 10 .. 60, grids 4R x 2R): long stepping, then a snapshot of all
        dict(name="sweep_f32", kind="sweep", n=64, rmin=10, rmax=60, odd=False, storage="f32", steps=500,
             snapshot=64),
        # the sweep in the most accurate 16-bit form
        dict(name="sweep_f16eq", kind="sweep", n=64, rmin=10, rmax=60, odd=False, storage="f16", steps=100,
             snapshot=4),
        # the sweep end to end: fields up from pinned host memory, one step, all diagnostics back
        dict(name="sweep_e2e_f32", kind="e2e", n=64, rmin=10, rmax=60, odd=False, storage="f32", steps=1),
        # Rayleigh-Plateau threads at the paper's scale, lambda x 450, eight in one batch
        dict(name="threads_f32", kind="threads", n=8, Nr=450, storage="f32", steps=100, snapshot=1),
        # one lattice far larger than L2 (the oscillating drop scaled 32 times)
        dict(name="large_drop_f32", kind="lattice", flow="drop", Nz=8192, Nr=4096, storage="f32", steps=3),
        # the Laplace test: radii 16 .. 64 with both forcings, FP64, one batch
        dict(name="laplace_f64", kind="laplace", storage="f64", steps=20, snapshot=10),
        # gradients of the differentiable drop (512 x 128, R = 48, 16 amplitudes)
        dict(name="adjoint_f32", kind="adjoint", Nz=512, Nr=128, storage="f32", T=100, ckpt=10, amps=16),
        dict(name="adjoint_f64", kind="adjoint", Nz=256, Nr=128, storage="f64", T=50, ckpt=7, amps=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: lattices from 48 x 24 to 4096 x 2048 of any
    parity, batches of 16 to 160 lattices, gradients of 20 to 120 steps."""
    kind = rng.choice(["lattice", "lattice", "lattice", "sweep", "sweep", "e2e", "threads", "adjoint"])
    if kind == "lattice":
        flow = rng.choice(["drop", "drop", "drop", "pipe", "thread", "discs"])
        storage = rng.choice(["f32", "f32", "f64"])
        if flow == "discs":
            return dict(kind=kind, flow=flow, Nz=rng.randint(16, 72), Nr=_log(rng, 40, 400), storage=storage,
                        steps=rng.randint(10, 60))
        Nz = _log(rng, 48, 4096 if storage == "f32" else 1024)
        Nr = max(24, min(_log(rng, max(24, Nz // 4), max(32, Nz)), 2048))
        sites = Nz * Nr
        steps = max(1, min(60, int((6e7 if storage == "f32" else 3e6) / sites)))
        case = dict(kind=kind, flow=flow, Nz=Nz, Nr=Nr, storage=storage, steps=steps)
        if flow == "drop":
            case["forcing"] = rng.choice(["shift", "shift", "shift", "guo"])
        return case
    if kind == "adjoint":
        storage = rng.choice(["f32", "f64"])
        Nz = _log(rng, 96, 512 if storage == "f32" else 256)
        T = rng.randint(20, 120 if storage == "f32" else 60)
        return dict(kind=kind, Nz=Nz, Nr=max(32, Nz // rng.choice([2, 3, 4])), storage=storage, T=T,
                    ckpt=max(1, int(round(math.sqrt(T)))), amps=rng.randint(1, 16))
    if kind == "threads":
        return dict(kind=kind, n=rng.randint(2, 8), Nr=rng.randint(200, 450), storage=rng.choice(["f32", "f32", "f16"]),
                    steps=rng.randint(10, 60), snapshot=1)
    n = _log(rng, 16, 160)
    rmin = rng.randint(10, 24)
    case = dict(kind=kind, n=n, rmin=rmin, rmax=rng.randint(rmin + 8, 60), odd=rng.random() < 0.2,
                storage=rng.choice(["f32", "f32", "f16", "bf16"]))
    if kind == "e2e":
        return dict(case, storage=rng.choice(["f32", "f32", "f64"]), steps=rng.randint(1, 4))
    return dict(case, steps=rng.randint(20, 120), snapshot=rng.choice([1, 4, n]))


# ------------------------------------------------------------------ the inputs --
@lru_cache(maxsize=None)
def _pair(G):
    return inputs.coexistence(G)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _tanh(d, R, rl, rv):
    return rv + 0.5 * (rl - rv) * (1.0 - torch.tanh((d - R) / 2.0))


def _grid(L, dev):
    z = torch.arange(L["Nz"], dtype=F64, device=dev)[None, :]
    r = torch.arange(L["Nr"], dtype=F64, device=dev)[:, None] + 0.5 + L["r_off"]
    return z, r


def _drop(L, dev):
    z, r = _grid(L, dev)
    dz = z - L["zc"]
    d = torch.sqrt(dz * dz + r * r)
    ct = dz / d
    rho = _tanh(d, L["R"] * (1.0 + L["a2"] * 0.5 * (3.0 * ct * ct - 1.0)), L["rho_l"], L["rho_v"])
    return rho, None, None


def _thread(L, dev):
    z, r = _grid(L, dev)
    wave = 2.0 * math.pi * (z - L["shift"]) / L["Nz"]
    rho = _tanh(r + 0.0 * z, L["R"] * (1.0 + L["a2"] * torch.cos(wave)), L["rho_l"], L["rho_v"])
    uz = L["eps_u"] * torch.sin(wave) * (rho - L["rho_v"]) / (L["rho_l"] - L["rho_v"])
    return rho, uz, torch.zeros_like(rho)


def _pipe(L, dev):
    z, r = _grid(L, dev)
    w = 2.0 * math.pi * z / L["Nz"]
    rho = 1.0 + 0.01 * torch.cos(w + L["shift"]) * torch.cos(0.2 * r)
    uz = 3e-3 * (1.0 - (r / L["Nr"]) ** 2) * (1.0 + 0.1 * torch.sin(w + L["shift"]))
    return rho, uz, 1e-4 * torch.sin(w) * torch.sin(math.pi * r / L["Nr"])


def _discs(L, dev):
    rho = torch.ones((L["Nr"], L["Nz"]), dtype=F64, device=dev)
    ur = torch.zeros_like(rho)
    ur[0] = torch.as_tensor(L["inlet"], dtype=F64, device=dev)
    return rho, torch.zeros_like(rho), ur


FIELDS = {"drop": _drop, "thread": _thread, "pipe": _pipe, "discs": _discs}


def _lattice(flow, Nz, Nr, rng, **kw):
    """Parameters of one lattice: plain numbers, made from the seed."""
    L = dict(flow=flow, Nz=Nz, Nr=Nr, tau=1.0, G=-5.0, gz=0.0, wall="freeslip", z_bc="periodic", r_lo="axis",
             r_off=0.0, rho_out=1.0, forcing="shift", rho_l=1.93, rho_v=0.16, R=1.0, zc=Nz / 2.0, a2=0.0,
             shift=0.0, eps_u=0.0, inlet=None)
    L.update(kw)
    if flow == "drop":
        L["a2"] = float(rng.uniform(0.02, 0.08))
        L["zc"] = Nz / 2.0 + float(rng.uniform(-0.5, 0.5))
        if "R" not in kw:
            L["R"] = 0.31 * min(Nz, 2 * Nr)
    elif flow == "thread":
        L["shift"] = float(rng.uniform(0.0, 4.0))
        if "R" not in kw:
            L["R"], L["a2"] = 0.2 * Nr, float(rng.uniform(0.05, 0.1))
    elif flow == "pipe":
        L.update(wall="noslip", gz=1e-5, G=0.0, R=float(Nr), shift=float(rng.uniform(0.0, 1.0)))
    elif flow == "discs":
        U2, Ri = 3.93e-4 * float(rng.uniform(0.8, 1.2)), 9.5
        z = np.arange(Nz) + 0.5
        L.update(wall="outlet", z_bc="noslip", r_lo="inlet", r_off=Ri - 0.5, G=0.0, R=float(Nr),
                 inlet=-U2 * (4.0 / Nz ** 2) * z * (z - Nz))
    return L


def _lattices(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "lattice":
        return [_lattice(case["flow"], case["Nz"], case["Nr"], rng, forcing=case.get("forcing", "shift"))]
    if kind == "threads":
        lam = [448, 576, 640, 768, 1024, 1280, 1536, 1792][:case["n"]]
        R = 80.0 * case["Nr"] / 450.0
        return [_lattice("thread", z, case["Nr"], rng, G=-6.0, rho_l=2.68, rho_v=0.078, R=R,
                         eps_u=4e-3 * float(rng.uniform(0.8, 1.2))) for z in lam]
    if kind == "laplace":
        rl, rv = _pair(-5.0)
        return [_lattice("drop", 4 * R + 16, 2 * R + 8, rng, forcing=f, R=float(R), rho_l=rl, rho_v=rv)
                for f in ("shift", "guo") for R in (16, 24, 32, 48, 64)]
    shapes = np.random.default_rng(1234)  # the sweep's grids are the case's, its physics the seed's
    out = []
    for q in range(case["n"]):
        R = int(round(shapes.uniform(case["rmin"], case["rmax"])))
        G = round(float(rng.uniform(-5.25, -4.75)), 1)
        rl, rv = _pair(G)
        odd = 1 if case["odd"] and q % 3 == 0 else 0
        out.append(_lattice("drop", 4 * R + odd, 2 * R, rng, G=G, tau=float(rng.uniform(0.8, 1.2)), R=0.95 * R,
                            rho_l=rl, rho_v=rv))
    return out


def _spec(L, shift):
    return amlbm.InstanceSpec(L["Nz"], L["Nr"], L["tau"], L["G"], wall=L["wall"], gz=L["gz"], shift=shift,
                              z_bc=L["z_bc"], r_lo=L["r_lo"], r_off=L["r_off"], rho_out=L["rho_out"],
                              forcing=L["forcing"])


def _shift(storage):
    return "equilibrium" if storage == "f16" else "default"


def _amps(case, seed):
    return np.random.default_rng(seed).normal(0.0, 0.02, size=case["amps"])


def _run_of(case):
    Nz, Nr = case["Nz"], case["Nr"]
    return dict(zc=Nz / 2.0, R=0.375 * min(Nz / 2.0, Nr), w=2.0, rho_l=1.93, rho_v=0.16)


# ------------------------------------------------------------- prepare and run --
def prepare(case, seed):
    kind, storage = case["kind"], case["storage"]
    if kind == "adjoint":
        rng = np.random.default_rng(seed + 1)
        lat = amlbm.Lattice(case["Nz"], case["Nr"], tau=1.0, G=float(rng.uniform(-5.1, -4.9)), storage=storage)
        return dict(case=case, lat=lat, amps=_amps(case, seed))
    lats = _lattices(case, seed)
    params = np.array([[L["zc"], L["R"], L["rho_l"], L["rho_v"]] for L in lats])
    if kind == "lattice":
        L = lats[0]
        lat = amlbm.Lattice(L["Nz"], L["Nr"], tau=L["tau"], G=L["G"], wall=L["wall"], gz=L["gz"], storage=storage,
                            z_bc=L["z_bc"], r_lo=L["r_lo"], r_off=L["r_off"], rho_out=L["rho_out"],
                            forcing=L["forcing"])
        if L["inlet"] is not None:
            lat.set_inlet(0.0 * L["inlet"], L["inlet"])
        rho, uz, ur = FIELDS[L["flow"]](L, "cuda")
        lat.init_fields_device(rho, uz, ur)
        torch.cuda.synchronize()  # the fields go when this function returns
        return dict(case=case, lat=lat, diag=dict(zc=L["zc"], R=L["R"], rho_l=L["rho_l"], rho_v=L["rho_v"]))
    b = amlbm.Batch([_spec(L, _shift(storage)) for L in lats], storage=storage)
    parts = [FIELDS[L["flow"]](L, "cuda") for L in lats]
    dt = torch.float64 if storage == "f64" else torch.float32
    host = []
    for q in range(3):
        if parts[0][q] is None:
            host.append(None)
        else:
            host.append(torch.cat([p[q].reshape(-1) for p in parts]).to(dt).cpu().pin_memory().numpy())
    if kind == "e2e" and host[1] is None:
        zero = torch.zeros(b.sites, dtype=dt).pin_memory().numpy()
        host[1] = host[2] = zero
    b.init_all(*host)
    state = dict(case=case, b=b, params=params, host=host)
    if case.get("snapshot"):
        n = sum(L["Nz"] * L["Nr"] for L in lats[:case["snapshot"]])
        state["fields"] = np.empty((3, n), dtype=np.float64 if storage == "f64" else np.float32)
    return state


def _device_state(lat):
    """The lattice's populations and psi as views of its own device memory."""
    f, psi, pitch = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_int()
    lat.lib.amlbm_device_state(lat.h, ctypes.byref(f), ctypes.byref(psi), ctypes.byref(pitch))
    dt = torch.float64 if lat.storage == "f64" else torch.float32
    es, P = dt.itemsize, pitch.value

    def view(p, planes):
        at = p.value - lat.workspace.data_ptr()
        t = lat.workspace[at:at + planes * lat.Nr * P * es].view(dt)
        return t.view(planes, lat.Nr, P)[:, :, :lat.Nz]

    return view(f, 9), view(psi, 1)


def run(state):
    case = state["case"]
    kind, wide = case["kind"], case["storage"] == "f64"
    ft = np.float64 if wide else np.float32  # the precision the values were computed in
    if kind == "adjoint":
        lat, p = state["lat"], _run_of(case)
        J, dG, dT, dA = lat.adjoint(case["T"], state["amps"], p["zc"], p["R"], p["w"], p["rho_l"], p["rho_v"],
                                    ckpt_every=case["ckpt"])
        return {"J": np.array([J], dtype=ft), "grad": np.concatenate([[dG, dT], dA]).astype(ft)}
    if kind == "lattice":
        lat = state["lat"]
        lat.step(case["steps"])
        d = lat.diagnostics(check=False, **state["diag"])
        f, psi = _device_state(lat)
        return {"f": f, "psi": psi, "diag": np.array([d[q] for q in amlbm.DIAG_FIELDS[:13]], dtype=ft)}
    b = state["b"]
    if kind == "e2e":
        b.init_all(*state["host"])
    b.step(case["steps"])
    d = b.diagnostics_all(state["params"], check=False, as_array=True)
    out = {"diag": d[:, :13].astype(ft)}
    if case.get("snapshot"):
        at, buf = 0, state["fields"]
        for k in range(min(case["snapshot"], case["n"] if "n" in case else 10)):
            for q, a in enumerate(b.read(k)):
                buf[q, at:at + a.size] = a.reshape(-1)
            at += a.size
        out["fields"] = buf
    return out


def work(case):
    """Every timestep reads and writes the populations and psi of every site once; a
    gradient steps forward, steps again from its checkpoints, and goes back over
    every step reading the state and the adjoint state and writing the latter."""
    es, ps = BYTES[case["storage"]], 8 if case["storage"] == "f64" else 4
    if case["kind"] == "adjoint":
        n = case["Nz"] * case["Nr"] * case["T"]
        return {"bytes": n * (2 * (18 * es + 2 * ps) + 27 * es + ps), "flops": n * (2 * FLOPS + FLOPS_ADJ)}
    lats = _lattices(case, 0)
    sites = sum(L["Nz"] * L["Nr"] for L in lats)
    per = 18 * es + 2 * ps + (16 if case["storage"] == "f16" else 0)
    nbytes = sites * case["steps"] * per + sites * (9 * es + ps)  # the steps, then the diagnostics' read
    if case["kind"] == "e2e":
        nbytes += sites * (3 * ps + 9 * es + ps)
    n = sum(L["Nz"] * L["Nr"] for L in lats[:case.get("snapshot", 0)])
    return {"bytes": nbytes + 2 * n * 3 * ps, "flops": sites * case["steps"] * FLOPS}


# ------------------------------------------------------- the same in 64 bits --
CZ = [0, 1, 0, -1, 0, 1, -1, -1, 1]
CR = [0, 0, 1, 0, -1, 1, 1, -1, -1]
W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
MIRROR = [0, 1, 4, 3, 2, 8, 7, 6, 5]
OPPOSITE = [0, 3, 4, 1, 2, 7, 8, 5, 6]


class _Exact:
    """The scheme of Sec. II on a flat list of the sites of several lattices: every
    stencil tap is a gather through a table of neighbours that holds the wraps and
    the mirrors."""

    def __init__(self, lats, dev):
        self.lats, self.dev = lats, dev
        cat = lambda f: torch.cat([f(L) for L in lats])  # noqa: E731
        full = lambda v: cat(lambda L: torch.full((L["Nz"] * L["Nr"],), v(L), dtype=F64, device=dev))  # noqa: E731
        ints = lambda v: cat(lambda L: torch.full((L["Nz"] * L["Nr"],), v(L), dtype=torch.int64, device=dev))  # noqa: E731
        self.Nz, self.Nr = ints(lambda L: L["Nz"]), ints(lambda L: L["Nr"])
        site = cat(lambda L: torch.arange(L["Nz"] * L["Nr"], device=dev))
        off = np.concatenate([[0], np.cumsum([L["Nz"] * L["Nr"] for L in lats])])
        self.off = off
        self.base = torch.cat([torch.full((int(off[q + 1] - off[q]),), int(off[q]), device=dev) for q in range(len(lats))])
        self.j, self.k = site // self.Nz, site % self.Nz
        self.N = int(off[-1])
        self.tau, self.G, self.gz = full(lambda L: L["tau"]), full(lambda L: L["G"]), full(lambda L: L["gz"])
        self.r = self.j + 0.5 + full(lambda L: L["r_off"])
        flag = lambda key, v: ints(lambda L: int(L[key] == v)).bool()  # noqa: E731
        self.zw, self.inl = flag("z_bc", "noslip"), flag("r_lo", "inlet")
        self.outl, self.nos, self.guo = flag("wall", "outlet"), flag("wall", "noslip"), flag("forcing", "guo")
        self.rho_out = full(lambda L: L["rho_out"])
        self.bin, self.bout = self.inl & (self.j == 0), self.outl & (self.j == self.Nr - 1)
        self.open = bool((self.bin | self.bout).any())
        self.inlet = cat(lambda L: torch.as_tensor(L["inlet"] if L["inlet"] is not None else np.zeros(L["Nz"]),
                                                   dtype=F64, device=dev).repeat(L["Nr"]))
        self.tap = {}
        for dz, dr in [(0, 0)] + [(m * a, m * b) for a in (-1, 0, 1) for b in (-1, 0, 1) if a or b for m in (1, 2)]:
            self.tap[dz, dr] = self._tap(dz, dr)
        src = []
        for i in range(9):
            k, j = self.k - CZ[i], self.j - CR[i]
            d = torch.full_like(j, i)
            kk = torch.where(self.zw, k, k % self.Nz)
            axis, wall = (j < 0) & ~self.inl, (j >= self.Nr) & ~self.outl
            d = torch.where(axis | wall, torch.full_like(d, MIRROR[i]), d)
            bb = wall & self.nos
            d = torch.where(bb, torch.full_like(d, OPPOSITE[i]), d)
            kk = torch.where(bb, self.k, kk)
            jj = torch.where(axis | wall, self.j, j)
            out = self.zw & ((k < 0) | (k >= self.Nz))
            d = torch.where(out, torch.full_like(d, OPPOSITE[i]), d)
            kk, jj = torch.where(out, self.k, kk), torch.where(out, self.j, jj)
            own = self.bin | self.bout
            d = torch.where(own, torch.full_like(d, i), d)
            kk, jj = torch.where(own, self.k, kk), torch.where(own, self.j, jj)
            src.append(d * self.N + self.base + jj * self.Nz + kk)
        self.src = torch.stack(src).reshape(-1)

    def _tap(self, dz, dr):
        k, j = self.k + dz, self.j + dr
        zg = self.zw & ((k < 0) | (k >= self.Nz))
        km = torch.where(k < 0, -1 - k, torch.where(k >= self.Nz, 2 * self.Nz - 1 - k, k))
        kk = torch.where(self.zw, km, k % self.Nz)
        lo, hi = j < 0, j >= self.Nr
        jj = torch.where(lo, torch.where(self.inl, -j, -1 - j), j)
        jj = torch.where(hi, torch.where(self.outl, 2 * (self.Nr - 1) - j, 2 * self.Nr - 1 - j), jj)
        one = torch.ones(self.N, dtype=F64, device=self.dev)
        odd_r = torch.where(lo | hi, -one, one)
        zs = torch.where(zg, -one, one)
        # u beyond a boundary: mirrored with the boundary's signs, or continued
        # linearly (2 u(b) - u) about an inlet or outlet row b
        cont = (lo & self.inl) | (hi & self.outl)
        jb = torch.where(lo, torch.zeros_like(jj), self.Nr - 1)
        uz_s = zs * torch.where(cont | (hi & self.nos), -one, one)
        ur_s = zs * odd_r
        edge = (cont, self.base + jb * self.Nz + self.k) if bool(cont.any()) else None
        return self.base + jj * self.Nz + kk, odd_r, uz_s, ur_s, edge

    # stencils: even fields (psi), fields odd about the axis and the walls (d_r psi), velocities
    def _at(self, a, dz, dr, kind):
        idx, odd, uz_s, ur_s, edge = self.tap[dz, dr]
        v = a.index_select(0, idx)
        if kind == "even":
            return v
        if kind == "odd":
            return v * odd
        v = v * (uz_s if kind == "uz" else ur_s)
        return v if edge is None else v + torch.where(edge[0], 2.0 * a.index_select(0, edge[1]), torch.zeros_like(v))

    def iso_r(self, a, kind):
        s = 0.0
        for c in ((0, 1), (1, 1), (-1, 1)):
            for sg in (1, -1):
                z, r = c[0], sg * c[1]
                s = s + sg * (8.0 * self._at(a, z, r, kind) - self._at(a, 2 * z, 2 * r, kind))
        return s / 36.0

    def d1(self, a, dz, dr, kind):
        p = lambda m: self._at(a, m * dz, m * dr, kind)  # noqa: E731
        return (8.0 * (p(1) - p(-1)) - (p(2) - p(-2))) / 12.0

    def feq(self, rho, vz, vr):
        v2 = vz * vz + vr * vr
        out = []
        for i in range(9):
            cv = CZ[i] * vz + CR[i] * vr
            out.append(W[i] * rho * (1.0 + 3.0 * cv + 4.5 * cv * cv - 1.5 * v2))
        return torch.stack(out)

    def init(self, fields):
        z = lambda a, b: torch.zeros_like(b) if a is None else a  # noqa: E731
        rho = torch.cat([p[0].reshape(-1) for p in fields])
        uz = torch.cat([z(p[1], p[0]).reshape(-1) for p in fields])
        ur = torch.cat([z(p[2], p[0]).reshape(-1) for p in fields])
        return self.feq(rho, uz, ur)

    def macro(self, f):
        rho = f.sum(0)
        psi = 1.0 - torch.exp(-rho)
        sz = sr = 0.0
        for i in range(1, 9):
            p = self._at(psi, CZ[i], CR[i], "even")
            if CZ[i]:
                sz = sz + W[i] * CZ[i] * p
            if CR[i]:
                sr = sr + W[i] * CR[i] * p
        dr = self.iso_r(psi, "even")
        drr = self.iso_r(dr, "odd")
        dzr = self.d1(self.d1(psi, 0, 1, "even"), 1, 0, "even")
        g = -self.G / 18.0 * psi / self.r
        Fz = -self.G * psi * sz + g * dzr + rho * self.gz
        Fr = -self.G * psi * sr + g * (drr - dr / self.r)
        jz, jr = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]), (f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7])
        return rho, psi, Fz, Fr, jz, jr, (jz + 0.5 * Fz) / rho, (jr + 0.5 * Fr) / rho

    def step(self, f):
        rho, psi, Fz, Fr, jz, jr, uz, ur = self.macro(f)
        mu = rho * (self.tau - 0.5) / 3.0
        S = -rho * ur / self.r
        Hz = (mu * (self.d1(uz, 0, 1, "uz") + self.d1(ur, 1, 0, "ur")) - rho * ur * uz) / self.r
        Hr = (2.0 * mu * (self.d1(ur, 0, 1, "ur") - ur / self.r) - rho * ur * ur) / self.r
        vz, vr = (jz + self.tau * Fz) / rho, (jr + self.tau * Fr) / rho
        if bool(self.guo.any()):
            vz, vr = torch.where(self.guo, uz, vz), torch.where(self.guo, ur, vr)
        fe = self.feq(rho, vz, vr)
        post = []
        gk = torch.where(self.guo, 1.0 - 0.5 / self.tau, torch.zeros_like(self.tau))
        for i in range(9):
            p = f[i] + (fe[i] - f[i]) / self.tau + W[i] * (S + 3.0 * (CZ[i] * Hz + CR[i] * Hr))
            cF, cu = CZ[i] * Fz + CR[i] * Fr, CZ[i] * uz + CR[i] * ur
            post.append(p + gk * W[i] * (3.0 * (cF - uz * Fz - ur * Fr) + 9.0 * cu * cF))
        post = torch.stack(post)
        if self.open:
            up, down = self.tap[0, 1][0], self.tap[0, -1][0]
            b = torch.where(self.bin, rho[up], self.rho_out)
            bz = torch.where(self.bin, torch.zeros_like(uz), uz[down])
            br = torch.where(self.bin, self.inlet, ur[down])
            post = torch.where(self.bin | self.bout, self.feq(b, bz, br), post)
        return post.reshape(-1).index_select(0, self.src).reshape(9, self.N)

    def diag(self, f, params):
        rho, psi, _, _, _, _, uz, ur = self.macro(f)
        rows = []
        for q, L in enumerate(self.lats):
            a, b = int(self.off[q]), int(self.off[q + 1])
            zc, R, rl, rv = (float(v) for v in params[q])
            shp = (L["Nr"], L["Nz"])
            p, s, wz, wr, r = (t[a:b].reshape(shp) for t in (rho, psi, uz, ur, self.r))
            k = self.k[a:b].reshape(shp)
            w, u2 = 2 * math.pi * r * p, wz * wz + wr * wr
            q2 = (2 * math.pi * r * (p - rv) / (rl - rv) * ((k - zc) ** 2 - 0.5 * r * r)).sum()
            below = p < 0.5 * (rl + rv)
            first = torch.where(below.any(0), below.int().argmax(0), torch.full_like(k[0], L["Nr"]))
            hi, lo = first.clamp(max=L["Nr"] - 1)[None], (first - 1).clamp(min=0)[None]
            v0, v1 = p.gather(0, lo)[0], p.gather(0, hi)[0]
            r0 = 0.5 + L["r_off"]
            rad = (first - 1 + r0) + (v0 - 0.5 * (rl + rv)) / torch.where(v0 == v1, torch.ones_like(v0), v0 - v1)
            rad = torch.where(first == 0, torch.full_like(rad, r0 - 0.5), rad)
            rad = torch.where(first == L["Nr"], torch.full_like(rad, L["Nr"] + r0 - 0.5), rad)
            kc = int(math.floor(zc + 0.5)) % L["Nz"]
            ko = (kc + L["Nz"] // 2) % L["Nz"]
            pres = lambda c, j: p[j, c] / 3.0 + L["G"] * s[j, c] ** 2 / 6.0  # noqa: E731
            pi_, po = pres(kc, 0), pres(ko, L["Nr"] - 1)
            rows.append(torch.stack([p.sum(), w.sum(), (w * wz).sum(), 0.5 * (w * u2).sum(), u2.max().sqrt(),
                                     5.0 / (4 * math.pi * R ** 5) * q2, rad[kc], rad.min(), pi_, po, pi_ - po,
                                     torch.zeros_like(pi_), (-p * wr / r).sum()]))
        return torch.stack(rows), (rho, uz, ur)


def _exact_adjoint(case, seed, dev):
    p = _run_of(case)
    L = _lattice("drop", case["Nz"], case["Nr"], np.random.default_rng(0))
    M = _Exact([L], dev)
    rng = np.random.default_rng(seed + 1)
    G = torch.tensor(float(rng.uniform(-5.1, -4.9)), dtype=F64, device=dev, requires_grad=True)
    tau = torch.tensor(1.0, dtype=F64, device=dev, requires_grad=True)
    amps = torch.tensor(_amps(case, seed), dtype=F64, device=dev, requires_grad=True)
    M.G, M.tau = G.expand(M.N), tau.expand(M.N)
    z, r = M.k - p["zc"], M.r
    d = torch.sqrt(z * z + r * r)
    x = z / d
    p0, p1, s = torch.ones_like(x), x, 0.0
    for m in range(1, case["amps"] + 1):
        p0, p1 = p1, ((2 * m + 1) * x * p1 - m * p0) / (m + 1)
        s = s + amps[m - 1] * p1
    f = M.feq(_tanh(d, p["R"] * (1.0 + s), p["rho_l"], p["rho_v"]), 0.0 * d, 0.0 * d)
    for _ in range(case["T"]):
        f = M.step(f)
    phi = (f.sum(0) - p["rho_v"]) / (p["rho_l"] - p["rho_v"])
    a2 = 5.0 / (4 * math.pi * p["R"] ** 5) * (2 * math.pi * r * phi * (z * z - 0.5 * r * r)).sum()
    J = a2 * a2
    g = torch.autograd.grad(J, [G, tau, amps])
    return {"J": J.detach().reshape(1).cpu().numpy(),
            "grad": torch.cat([g[0].reshape(1), g[1].reshape(1), g[2]]).cpu().numpy()}


def exact(case, seed):
    dev = _device()
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed, dev)
    lats = _lattices(case, seed)
    params = np.array([[L["zc"], L["R"], L["rho_l"], L["rho_v"]] for L in lats])
    with torch.no_grad():
        M = _Exact(lats, dev)
        f = M.init([FIELDS[L["flow"]](L, dev) for L in lats])
        for _ in range(case["steps"]):
            f = M.step(f)
        d, fields = M.diag(f, params)
        if case["kind"] == "lattice":
            shp = (lats[0]["Nr"], lats[0]["Nz"])
            return {"f": f.reshape(9, *shp), "psi": (1.0 - torch.exp(-f.sum(0))).reshape(1, *shp),
                    "diag": d[0].cpu().numpy()}
        out = {"diag": d.cpu().numpy()}
        if case.get("snapshot"):
            n = int(M.off[min(case["snapshot"], len(lats))])
            out["fields"] = torch.stack([a[:n] for a in fields]).cpu().numpy()
        return out
