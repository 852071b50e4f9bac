"""Performance cases: the runs that users of this library make, through its
public entry points, from the smallest to the largest.

A pass is one segment of a run as a program makes it: the state goes in
(``set_state`` or a host buffer), a few CFL time steps are taken, and the
state comes out again.  FP32 contexts return their state as float64 tensors
that hold FP32 values; the passes store those as float32 snapshots, as an
FP32 run would.

``exact`` restates the method in plain torch float64: HLLD (Miyoshi & Kusano
2005) with the GLM interface step (Dedner et al. 2002) or constrained
transport (Gardiner & Stone 2005, CT-contact), PLM (minmod / MC) or WENO-Z
(Borges et al. 2008) on primitives, RK2 / SSP-RK3.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2510_24175_gb300 as m
from paper_2510_24175_gb300.adjoint import MHDRollout

RHO, VX, BX, PRS, PSI = 0, 1, 4, 7, 8
TP = 2.0 * math.pi


def _case(name, path, ic, n, steps, prec="fp64", lim="mc", rk=2, divb="glm", bc="periodic",
          **more):
    return {"name": name, "path": path, "ic": ic, "nx": n[0], "ny": n[1], "nz": n[2],
            "steps": steps, "prec": prec, "lim": lim, "rk": rk, "divb": divb, "bc": bc, **more}


def listed():
    return [
        # the 1-D shock tube, the library's smallest grid: bound by launches and
        # latency, so its steps are replayed from one graph
        _case("shock_tube_1024_fp64", "graph", "shock", (1024, 1, 1), 20, lim="minmod",
              bc="outflow"),
        # one step of a small 3-D box (a coupled code that asks for a step at a time)
        _case("box_48_one_step_fp64", "steps", "vortex", (48, 48, 48), 1),
        # the benchmark run: 3-D Orszag-Tang at 256^3 in FP64
        _case("vortex_256_fp64", "steps", "vortex", (256, 256, 256), 2),
        # a ragged production grid with open boundaries and the minmod limiter
        _case("open_box_ragged_fp64", "steps", "turbulent", (150, 101, 67), 4, lim="minmod",
              bc="outflow"),
        # host-resident state, streamed through the device one step at a time
        _case("host_step_256_fp64", "host", "vortex", (256, 256, 256), 1),
        # gradient of a 2-D rollout with every step kept (forward + backward)
        _case("adjoint_2d_512_kept", "adjoint", "vortex", (512, 512, 1), 8, every=0),
        # gradient of a 3-D open-boundary rollout, recomputed from checkpoints
        _case("adjoint_3d_checkpointed", "adjoint", "turbulent", (64, 52, 41), 6,
              bc="outflow", every=3),
        # the FP32 benchmark run: turbulent box at 512^3, with its conservation sums
        _case("turbulence_512_fp32", "steps", "turbulent", (512, 512, 512), 2, prec="fp32",
              sums=True),
        # a ragged FP32 box replayed from one graph
        _case("turbulence_ragged_fp32", "graph", "turbulent", (203, 134, 77), 6, prec="fp32"),
        # the paper's strong-scaling scheme: WENO-Z + SSP-RK3 with GLM cleaning
        _case("wenoz_rk3_glm_256_fp64", "steps", "vortex", (256, 256, 256), 1, lim="wenoz", rk=3),
        # the paper's weak-scaling scheme: WENO-Z + SSP-RK3 with constrained transport
        _case("wenoz_rk3_ct_256_fp32", "steps", "vortex", (256, 256, 256), 3, prec="fp32",
              lim="wenoz", rk=3, divb="ct"),
        # a parameter study: 64 independent FP32 boxes in one persistent launch
        _case("ensemble_64_fp32", "ensemble", "vortex", (0, 0, 0), 5, prec="fp32", boxes=64,
              shapes=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """The same runs at other sizes: even, odd and ragged extents from a few
    cells to the benchmark grids, each scheme, precision and boundary that the
    path accepts."""
    path = rng.choice(["steps", "steps", "steps", "graph", "host", "adjoint", "ensemble"])
    if path == "ensemble":
        case = _case("", path, "vortex", (0, 0, 0), rng.randint(2, 5), prec="fp32",
                     boxes=rng.randint(4, 64), shapes=rng.randint(1, 10000))
        del case["name"]
        return case
    dim = rng.choice([2, 3]) if path in ("adjoint", "graph") else 3
    prec = rng.choice(["fp64", "fp32"]) if path in ("steps", "graph") else "fp64"
    lim = rng.choice(["mc", "minmod"] if path == "adjoint" else ["mc", "minmod", "wenoz"])
    rk = 3 if lim == "wenoz" else 2
    divb = "ct" if path == "steps" and rng.random() < 0.3 else "glm"
    bc = "periodic" if divb == "ct" else rng.choice(["periodic", "outflow"])
    top = {"adjoint": 96, "host": 224, "steps": 288, "graph": 160}[path]
    if path == "steps" and prec == "fp32" and lim != "wenoz":
        top = 448
    if dim == 2:
        n = [_log(rng, 64, 640), _log(rng, 64, 640), 1]
    else:
        edge = math.exp(rng.uniform(math.log(24), math.log(top)))
        n = [max(16, min(top, int(round(edge * rng.uniform(0.7, 1.3))))) for _ in range(3)]
    steps = {"adjoint": rng.randint(2, 6), "host": 1, "graph": rng.randint(2, 8)}.get(
        path, rng.randint(1, 2))
    # about nanoseconds per zone-update: a drawn pass stays below 0.3 s
    cost = (20.0 if lim == "wenoz" else 15.0 if path == "adjoint" else 5.0) * (
        0.05 if prec == "fp32" else 1.0) * n[0] * n[1] * n[2]
    steps = max(1, min(steps, int(3e8 / cost)))
    while cost > 3e8:
        n[2] -= 1
        cost *= n[2] / (n[2] + 1)
    ic = rng.choice(["vortex", "turbulent"]) if divb == "glm" else "vortex"
    more = {"every": rng.choice([0, 2])} if path == "adjoint" else {}
    case = _case("", path, ic, n, steps, prec, lim, rk, divb, bc, **more)
    del case["name"]
    return case


# ------------------------------------------------------------------- inputs --
def _random_field(n, gen, ncomp, dev, kmax=16, slope=-2.0):
    """Seeded Gaussian fields with an E(k) ~ k^slope shell spectrum."""
    nx, ny, nz = n
    k = [torch.fft.fftfreq(s, 1.0 / s, device=dev, dtype=torch.float64) if s > 1
         else torch.zeros(1, device=dev, dtype=torch.float64) for s in (nz, ny)]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, device=dev, dtype=torch.float64)
    K = (k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + kx[None, None, :] ** 2).sqrt()
    dim = sum(s > 1 for s in n)
    amp = torch.where((K >= 1) & (K <= min(kmax, min(s for s in n if s > 1) / 3)),
                      K.clamp(min=1.0) ** ((slope - (dim - 1)) / 2.0), torch.zeros_like(K))
    out = torch.empty((ncomp, nz, ny, nx), dtype=torch.float64, device=dev)
    for c in range(ncomp):
        re = torch.randn(K.shape, generator=gen, dtype=torch.float64, device=dev)
        im = torch.randn(K.shape, generator=gen, dtype=torch.float64, device=dev)
        out[c] = torch.fft.irfftn(torch.complex(re, im) * amp, s=(nz, ny, nx))
    return out / out.square().mean().sqrt()


def _curl(A, dx):
    """Face field of an edge vector potential (periodic): discretely divergence free."""
    up = lambda a, d: torch.roll(a, -1, 2 - d)  # noqa: E731
    b = torch.empty_like(A)
    for d in range(3):
        a, c = (d + 1) % 3, (d + 2) % 3
        b[d] = (up(A[c], a) - A[c]) / dx[a] - (up(A[a], c) - A[a]) / dx[c]
    return b


def _faces_to_cells(b):
    return torch.stack([0.5 * (b[d] + torch.roll(b[d], -1, 2 - d)) for d in range(3)])


def _prims(case, n, gen, dev, b0=None):
    """Primitive state (9, nz, ny, nx), and the face field for constrained transport."""
    nx, ny, nz = n
    V = torch.zeros((9, nz, ny, nx), dtype=torch.float64, device=dev)
    r = torch.rand(8, generator=gen, dtype=torch.float64, device=dev).tolist()
    x, y, z = [((torch.arange(s, device=dev, dtype=torch.float64) + 0.5) / s).view(shape)
               for s, shape in ((nx, (1, 1, -1)), (ny, (1, -1, 1)), (nz, (-1, 1, 1)))]
    if case["ic"] == "shock":  # Brio & Wu (1988) with the two states varied
        left = (x < 0.5).expand(nz, ny, nx)
        pick = lambda a, b: torch.where(left, a, b)  # noqa: E731
        f = [torch.tensor(1.0 + 0.2 * (q - 0.5), dtype=torch.float64, device=dev) for q in r]
        V[RHO] = pick(f[0], 0.125 * f[1])
        V[PRS] = pick(f[2], 0.1 * f[3])
        V[BX + 1] = pick(f[4], -f[5])
        V[BX] = 0.75 * f[6]
        return V, None
    if case["ic"] == "vortex":  # Orszag-Tang with shifted origins and B0 varied
        b0 = 0.2 + 0.2 * r[0] if b0 is None else b0
        V[RHO] = 25.0 / (36.0 * math.pi)
        V[PRS] = 5.0 / (12.0 * math.pi)
        V[VX] = -torch.sin(TP * (y + r[1]))
        V[VX + 1] = torch.sin(TP * (x + r[2]))
        V[VX + 2] = 0.1 * torch.sin(TP * (z + r[3])) if nz > 1 else 0.0
        V[BX] = -b0 * torch.sin(TP * (y + r[4]))
        V[BX + 1] = b0 * torch.sin(2 * TP * (x + r[5]))
        if case["divb"] != "ct":
            return V, None
        A = _random_field(n, gen, 3, dev, kmax=4)
        b = _curl(A, [1.0 / s for s in n])
        b = V[BX:BX + 3] + b * (0.05 / b.square().mean().sqrt())
        V[BX:BX + 3] = _faces_to_cells(b)
        return V, b
    V[RHO] = 1.0  # a turbulent box: rms |v| 0.5, mean field plus a solenoidal one
    V[PRS] = 0.6
    V[VX:VX + 3] = _random_field(n, gen, 3, dev) * (0.5 / math.sqrt(3.0))
    b = _curl(_random_field(n, gen, 3, dev), [1.0 / s for s in n])
    if nz == 1:
        b[2] = 0.0
    V[BX:BX + 3] = _faces_to_cells(b) * (0.05 / b.square().sum(0).mean().sqrt())
    V[BX] += 0.2
    return V, None


def _to_cons(V, gamma):
    U = V.clone()
    U[1:4] *= V[0]
    U[PRS] = V[PRS] / (gamma - 1.0) + 0.5 * V[0] * V[1:4].square().sum(0) \
        + 0.5 * V[4:7].square().sum(0)
    return U


def _gamma(case):
    return 2.0 if case["ic"] == "shock" else 5.0 / 3.0


def _config(case, n):
    lim = {"mc": m.MHD_LIM_MC, "minmod": m.MHD_LIM_MINMOD, "wenoz": m.MHD_LIM_WENOZ}[case["lim"]]
    bc = m.MHD_BC_OUTFLOW if case["bc"] == "outflow" else m.MHD_BC_PERIODIC
    return m.Config(n=tuple(n), gamma=_gamma(case), limiter=lim, bc=(bc,) * 6,
                    precision=m.MHD_FP32 if case["prec"] == "fp32" else m.MHD_FP64,
                    flags=m.MHD_FLAG_ADJOINT if case["path"] == "adjoint" else 0,
                    rk_order=case["rk"],
                    divb=m.MHD_DIVB_CT if case["divb"] == "ct" else m.MHD_DIVB_GLM)


def _box_sizes(case):
    """An ensemble's box edges: the study's shapes come with the case, its fields with the seed."""
    rng = np.random.default_rng(case["shapes"])
    return [int(e) for e in rng.choice([32, 48, 64, 96, 128], size=case["boxes"])]


def _boxes(case, seed, dev):
    gen = torch.Generator(device=dev).manual_seed(seed)
    b0 = torch.rand(case["boxes"], generator=gen, dtype=torch.float64, device=dev).tolist()
    return [_to_cons(_prims(case, (e,) * 3, gen, dev, 0.1 + 0.4 * q)[0], _gamma(case))
            for e, q in zip(_box_sizes(case), b0)]


def _inputs(case, seed, dev):
    gen = torch.Generator(device=dev).manual_seed(seed)
    n = (case["nx"], case["ny"], case["nz"])
    V, b = _prims(case, n, gen, dev)
    w = None
    if case["path"] == "adjoint":
        # a perturbed start (every variable varies in every direction, so the
        # step is differentiable there) and a seeded smooth functional of U_N
        V += 0.02 * _random_field(n, gen, 9, dev, kmax=8) * V.square().mean().sqrt()
        w = _random_field(n, gen, 9, dev, kmax=8)
    return _to_cons(V, _gamma(case)), b, w


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["path"] == "ensemble":
        U = _boxes(case, seed, dev)
        return {"case": case, "ens": m.Ensemble([_config(case, (e,) * 3)
                                                 for e in _box_sizes(case)]), "U": U}
    U, b, w = _inputs(case, seed, dev)
    st = {"case": case, "U": U, "b": b, "w": w,
          "solver": m.MHD(_config(case, (case["nx"], case["ny"], case["nz"])))}
    if case["path"] == "host":  # page-locked host buffers
        st["host"] = [torch.empty(U.shape, dtype=torch.float64, pin_memory=True).numpy()
                      for _ in range(2)]
        st["host"][0][...] = U.cpu().numpy()
        del st["U"]
    else:
        st["out"] = torch.empty_like(U)
    return st


def _snapshot(case, U):
    return U.float() if case["prec"] == "fp32" else U


def run(st):
    case = st["case"]
    if case["path"] == "ensemble":
        ens = st["ens"]
        for i, U in enumerate(st["U"]):
            ens.set_state(i, U)
        ens.step(case["steps"])
        return [_snapshot(case, ens.get_state(i)) for i in range(len(ens))]
    s = st["solver"]
    if case["path"] == "host":
        s.step_host(*st["host"])
        return {"U": st["host"][1]}
    if case["path"] == "adjoint":
        U0 = st["U"].detach().requires_grad_(True)
        UN = MHDRollout.apply(U0, s, case["steps"], case["every"])
        (UN * st["w"]).sum().backward()
        return {"U": UN.detach(), "grad": U0.grad}
    s.set_state(st["U"])
    if st["b"] is not None:
        s.set_face_field(st["b"])
    if case["path"] == "graph":
        s.step_n(case["steps"])
    else:
        for _ in range(case["steps"]):
            s.step()
    out = {"U": _snapshot(case, s.get_state(st["out"]))}
    if st["b"] is not None:
        out["b"] = _snapshot(case, s.get_face_field())
    if case.get("sums"):
        out["sums"] = s.conserved_sums()
    return out


def work(case):
    """State in, state out, and the arithmetic of the scheme: per cell and
    stage about 35 operations for the conversion and the update, and per
    direction about 160 for HLLD + GLM and 6 (PLM) or 55 (WENO-Z) per variable for
    the reconstruction; the adjoint about three times the forward step."""
    if case["path"] == "ensemble":
        cells, ndim = sum(e ** 3 for e in _box_sizes(case)), 3
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
        ndim = sum(case[k] > 1 for k in ("nx", "ny", "nz"))
    words = 18 + (6 if case["divb"] == "ct" else 0)
    rec = 9 * (55 if case["lim"] == "wenoz" else 6)
    flops = cells * case["steps"] * case["rk"] * (35.0 + ndim * (160 + rec))
    size = 4 if case["prec"] == "fp32" else 8
    if case["path"] == "adjoint":
        return {"bytes": 27.0 * cells * size, "flops": 4.0 * flops}
    return {"bytes": float(words * cells * size), "flops": flops}


# ---------------------------------------------------- the method in float64 --
def _cons_to_prim(U, gamma):
    rho = U[0]
    v = U[1:4] / rho
    p = (gamma - 1.0) * (U[7] - 0.5 * (U[1:4] * v).sum(0) - 0.5 * (U[4:7] * U[4:7]).sum(0))
    return torch.cat([rho[None], v, U[4:7], p[None], U[8:9]])


def _root(x):
    return x.clamp(min=1e-300).sqrt()


def _fast2(rho, gp, b2, bn2):
    a = (gp + b2) / rho
    return 0.5 * (a + _root(a * a - 4.0 * gp * bn2 / (rho * rho)))


def _max_speed(U, gamma, dims):
    """max |v_d| + c_f,d over cells and active directions."""
    lam = 0.0
    for z in range(0, U.shape[1], 64):
        V = _cons_to_prim(U[:, z:z + 64], gamma)
        b2 = (V[4:7] * V[4:7]).sum(0)
        for d in dims:
            c = _fast2(V[0], gamma * V[7], b2, V[4 + d] ** 2).sqrt()
            lam = max(lam, float((V[1 + d].abs() + c).max()))
    return lam


def _hlld(l, r, d, ch, gamma):
    """GLM interface step, then HLLD along d; l, r: (9, ...) primitive face states."""
    t1, t2 = (d + 1) % 3, (d + 2) % 3
    bx = 0.5 * (l[4 + d] + r[4 + d]) - (r[8] - l[8]) / (2.0 * ch)
    psi = 0.5 * (l[8] + r[8]) - 0.5 * ch * (r[4 + d] - l[4 + d])
    side = []
    for q in (l, r):
        u, v, w, by, bz = q[1 + d], q[1 + t1], q[1 + t2], q[4 + t1], q[4 + t2]
        b2 = bx * bx + by * by + bz * bz
        pt = q[7] + 0.5 * b2
        e = q[7] / (gamma - 1.0) + 0.5 * q[0] * (u * u + v * v + w * w) + 0.5 * b2
        side.append({"r": q[0], "u": u, "v": v, "w": w, "by": by, "bz": bz, "pt": pt, "e": e,
                     "c2": _fast2(q[0], gamma * q[7], b2, bx * bx),
                     "vb": u * bx + v * by + w * bz})
    L, R = side
    c = torch.maximum(L["c2"], R["c2"]).sqrt()
    L["S"], R["S"] = torch.minimum(L["u"], R["u"]) - c, torch.maximum(L["u"], R["u"]) + c
    dl, dr = (L["S"] - L["u"]) * L["r"], (R["S"] - R["u"]) * R["r"]
    SM = (dr * R["u"] - dl * L["u"] - R["pt"] + L["pt"]) / (dr - dl)
    pts = (dr * L["pt"] - dl * R["pt"] + dl * dr * (R["u"] - L["u"])) / (dr - dl)
    for q in side:
        den = q["r"] * (q["S"] - q["u"]) * (q["S"] - SM) - bx * bx
        deg = den.abs() < 1e-8 * pts
        den = torch.where(deg, torch.ones_like(den), den)
        q["rs"] = q["r"] * (q["S"] - q["u"]) / (q["S"] - SM)
        fv = bx * (SM - q["u"]) / den
        fb = (q["r"] * (q["S"] - q["u"]) ** 2 - bx * bx) / den
        q["vs"] = torch.where(deg, q["v"], q["v"] - q["by"] * fv)
        q["ws"] = torch.where(deg, q["w"], q["w"] - q["bz"] * fv)
        q["bys"] = torch.where(deg, q["by"], q["by"] * fb)
        q["bzs"] = torch.where(deg, q["bz"], q["bz"] * fb)
        q["vbs"] = SM * bx + q["vs"] * q["bys"] + q["ws"] * q["bzs"]
        q["es"] = ((q["S"] - q["u"]) * q["e"] - q["pt"] * q["u"] + pts * SM
                   + bx * (q["vb"] - q["vbs"])) / (q["S"] - SM)
        q["sq"] = _root(q["rs"])
    sg = torch.where(bx >= 0, torch.ones_like(bx), -torch.ones_like(bx))
    i = 1.0 / (L["sq"] + R["sq"])
    lr = L["sq"] * R["sq"] * sg
    vss = (L["sq"] * L["vs"] + R["sq"] * R["vs"] + (R["bys"] - L["bys"]) * sg) * i
    wss = (L["sq"] * L["ws"] + R["sq"] * R["ws"] + (R["bzs"] - L["bzs"]) * sg) * i
    byss = (L["sq"] * R["bys"] + R["sq"] * L["bys"] + lr * (R["vs"] - L["vs"])) * i
    bzss = (L["sq"] * R["bzs"] + R["sq"] * L["bzs"] + lr * (R["ws"] - L["ws"])) * i
    vbss = SM * bx + vss * byss + wss * bzss
    for q, s in ((L, -1.0), (R, 1.0)):
        q["Ss"] = SM + s * bx.abs() / q["sq"]
        q["ess"] = q["es"] + s * q["sq"] * (q["vbs"] - vbss) * sg
        st = [q["rs"] - q["r"], q["rs"] * SM - q["r"] * q["u"],
              q["rs"] * q["vs"] - q["r"] * q["v"], q["rs"] * q["ws"] - q["r"] * q["w"],
              q["bys"] - q["by"], q["bzs"] - q["bz"], q["es"] - q["e"]]
        ss = [0.0, 0.0, q["rs"] * (vss - q["vs"]), q["rs"] * (wss - q["ws"]),
              byss - q["bys"], bzss - q["bzs"], q["ess"] - q["es"]]
        ru = q["r"] * q["u"]
        f = [ru, ru * q["u"] + q["pt"] - bx * bx, ru * q["v"] - bx * q["by"],
             ru * q["w"] - bx * q["bz"], q["by"] * q["u"] - bx * q["v"],
             q["bz"] * q["u"] - bx * q["w"], (q["e"] + q["pt"]) * q["u"] - bx * q["vb"]]
        out = q["S"] > 0 if s < 0 else q["S"] < 0
        inner = q["Ss"] <= 0 if s < 0 else q["Ss"] >= 0
        star = torch.where(out, torch.zeros_like(bx), q["S"])
        dbl = torch.where(inner & ~out, q["Ss"], torch.zeros_like(bx))
        q["F"] = [a + star * b + dbl * k for a, b, k in zip(f, st, ss)]
    left = (L["S"] > 0) | ((R["S"] >= 0) & (SM >= 0))
    f = [torch.where(left, a, b) for a, b in zip(L["F"], R["F"])]
    F = [None] * 9
    F[0], F[7], F[8] = f[0], f[6], ch * ch * bx
    F[1 + d], F[1 + t1], F[1 + t2] = f[1], f[2], f[3]
    F[4 + d], F[4 + t1], F[4 + t2] = psi, f[4], f[5]
    return torch.stack(F)


def _weno(f, eps):
    """WENO-Z value at the face after cell i from the five cells f = i-2 .. i+2."""
    q = [(2 * f[0] - 7 * f[1] + 11 * f[2]) / 6, (-f[1] + 5 * f[2] + 2 * f[3]) / 6,
         (2 * f[2] + 5 * f[3] - f[4]) / 6]
    b = [13 / 12 * (f[0] - 2 * f[1] + f[2]) ** 2 + 0.25 * (f[0] - 4 * f[1] + 3 * f[2]) ** 2,
         13 / 12 * (f[1] - 2 * f[2] + f[3]) ** 2 + 0.25 * (f[1] - f[3]) ** 2,
         13 / 12 * (f[2] - 2 * f[3] + f[4]) ** 2 + 0.25 * (3 * f[2] - 4 * f[3] + f[4]) ** 2]
    tau = (b[0] - b[2]).abs()
    a = [g * (1.0 + tau / (k + eps)) for g, k in zip((0.1, 0.6, 0.3), b)]
    return (a[0] * q[0] + a[1] * q[1] + a[2] * q[2]) / (a[0] + a[1] + a[2])


def _faces(V, ax, n, case):
    """Left and right states of the n + 1 faces along axis ax of V, which has
    2 (PLM) or 3 (WENO-Z) ghost cells there."""
    cut = lambda a, o, c: a.narrow(ax, o, c)  # noqa: E731
    if case["lim"] == "wenoz":
        eps = 1e-18 if case["prec"] == "fp32" else 1e-40
        mid = cut(V, 2, n + 2)
        cells = [cut(V, o, n + 2) for o in range(5)]
        plus, minus = _weno(cells, eps), _weno(cells[::-1], eps)
        ok = (plus[0] > 0) & (plus[7] > 0) & (minus[0] > 0) & (minus[7] > 0)
        plus, minus = torch.where(ok, plus, mid), torch.where(ok, minus, mid)
    else:
        mid = cut(V, 1, n + 2)
        dm, dp = mid - cut(V, 0, n + 2), cut(V, 2, n + 2) - mid
        mag = torch.minimum(dm.abs(), dp.abs())
        if case["lim"] == "mc":
            mag = torch.minimum(2.0 * mag, 0.5 * (dm + dp).abs())
        sl = torch.where(dm * dp > 0, torch.where(dm > 0, mag, -mag), torch.zeros_like(mag))
        ok = (mid[0] - 0.5 * sl[0].abs() > 0) & (mid[7] - 0.5 * sl[7].abs() > 0)
        sl = torch.where(ok, sl, torch.zeros_like(sl))
        plus, minus = mid + 0.5 * sl, mid - 0.5 * sl
    return cut(plus, 0, n + 1), cut(minus, 1, n + 1)


def _stage_rhs(W, bw, dims, dx, ch, case):
    """L(W), and for constrained transport each direction's lower-face fluxes."""
    gamma, g = _gamma(case), 3 if case["lim"] == "wenoz" else 2
    L, low = torch.zeros_like(W), []
    for d in dims:
        ax, n = 3 - d, W.shape[3 - d]
        at = torch.arange(-g, n + g, device=W.device)
        at = at % n if case["bc"] == "periodic" else at.clamp(0, n - 1)
        side = 2 if d == 2 else 1  # blocks along another axis bound the memory
        parts, lows = [], []
        size = W.shape[side] if W.requires_grad else max(1, min(W.shape[side], 2 ** 23 // (
            W[0].numel() // W.shape[side]) or 1))
        for o in range(0, W.shape[side], size):
            c = min(size, W.shape[side] - o)
            V = _cons_to_prim(W.narrow(side, o, c), gamma).index_select(ax, at)
            l, r = _faces(V, ax, n, case)
            if bw is not None:
                bn = bw[d].narrow(side - 1, o, c)
                bn = torch.cat([bn, bn.narrow(ax - 1, 0, 1)], ax - 1)
                l, r = l.clone(), r.clone()
                l[4 + d] = r[4 + d] = bn
                l[8] = r[8] = 0.0
            F = _hlld(l, r, d, ch, gamma)
            parts.append((F.narrow(ax, 0, n) - F.narrow(ax, 1, n)) / dx[d])
            if bw is not None:
                lows.append(F.narrow(ax, 0, n).clone())
        L = L + torch.cat(parts, side)
        if bw is not None:
            low.append(torch.cat(lows, side))
    return L, low


def _upwind(f, lo, hi):
    return torch.where(f > 0, lo, torch.where(f < 0, hi, 0.5 * (lo + hi)))


def _curl_e(W, low, dx, ch, case):
    """-curl E on the faces from the CT-contact edge average."""
    V = _cons_to_prim(W, _gamma(case))
    thr = (1e-4 if case["prec"] == "fp32" else 1e-12) * ch * V[0]
    fm = [torch.where(F[0].abs() > thr, F[0], torch.zeros_like(F[0])) for F in low]
    dn = lambda a, d: torch.roll(a, 1, 2 - d)  # noqa: E731
    E = []
    for e in range(3):
        a, b = (e + 1) % 3, (e + 2) % 3
        Ec = V[1 + b] * V[4 + a] - V[1 + a] * V[4 + b]
        Ea, Eb = -low[a][4 + b], low[b][4 + a]  # on the a-faces, on the b-faces
        ea0, ea1, fa0, fa1 = dn(Ea, b), Ea, dn(fm[a], b), fm[a]
        eb0, eb1, fb0, fb1 = dn(Eb, a), Eb, dn(fm[b], a), fm[b]
        c00, c01, c10, c11 = dn(dn(Ec, a), b), dn(Ec, a), dn(Ec, b), Ec
        E.append(0.25 * (ea0 + ea1 + eb0 + eb1)
                 + 0.25 * (_upwind(fa0, eb0 - c00, eb1 - c10) - _upwind(fa1, c01 - eb0, c11 - eb1))
                 + 0.25 * (_upwind(fb0, ea0 - c00, ea1 - c01) - _upwind(fb1, c10 - ea0, c11 - ea1)))
    up = lambda q, d: torch.roll(q, -1, 2 - d)  # noqa: E731
    return torch.stack([(up(E[(d + 1) % 3], (d + 2) % 3) - E[(d + 1) % 3]) / dx[(d + 2) % 3]
                        - (up(E[(d + 2) % 3], (d + 1) % 3) - E[(d + 2) % 3]) / dx[(d + 1) % 3]
                        for d in range(3)])


def _advance(U, b, case, steps):
    n = U.shape[:0:-1]
    dims = [d for d in range(3) if n[d] > 1]
    dx = [1.0 / s for s in n]
    stages = [(0.0, 1.0), (0.75, 0.25), (1 / 3, 2 / 3)] if case["rk"] == 3 else [(0.0, 1.0),
                                                                                (0.5, 0.5)]
    for _ in range(steps):
        ch = _max_speed(U.detach(), _gamma(case), dims)
        dt = 0.8 / (ch * sum(1.0 / dx[d] for d in dims))
        W, bw = U, b
        for an, aw in stages:
            L, low = _stage_rhs(W, bw, dims, dx, ch, case)
            N = aw * (W + dt * L) + an * U
            if b is not None:
                bw = aw * (bw + dt * _curl_e(W, low, dx, ch, case)) + an * b
                N[8] = 0.0
                N[4:7] = _faces_to_cells(bw)
            W = N
        if b is None:
            damp = math.exp(-0.1 * ch * dt / min(dx[d] for d in dims))
            W = torch.cat([W[:8], W[8:] * damp])
        U, b = W, bw
    return U, b


def exact(case, seed, dev=None):
    dev = dev or torch.device("cuda")
    if case["path"] == "ensemble":
        return [_advance(U, None, case, case["steps"])[0] for U in _boxes(case, seed, dev)]
    U, b, w = _inputs(case, seed, dev)
    if case["path"] == "adjoint":
        U.requires_grad_(True)
        UN, _ = _advance(U, None, case, case["steps"])
        (UN * w).sum().backward()
        return {"U": UN.detach(), "grad": U.grad}
    if b is not None:  # the library makes the cells' B the face means, the pressure kept
        U[PRS] += 0.5 * (_faces_to_cells(b).square() - U[4:7].square()).sum(0)
        U[4:7] = _faces_to_cells(b)
    U, b = _advance(U, b, case, case["steps"])
    out = {"U": U}
    if b is not None:
        out["b"] = b
    if case.get("sums"):
        vol = 1.0 / U[0].numel()
        out["sums"] = torch.stack([U[k].sum() for k in (0, 1, 2, 3, 7, 4, 5, 6)]) * vol
    return out
