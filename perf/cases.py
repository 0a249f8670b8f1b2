"""The measured work of the GKS library: what users of it have it do, through its public entry points.

Every case is a workload of the package (``workloads.py``) at one size, with inputs of its own seed:
steps of the 2-D TM and 3-D Maxwell systems on Cartesian grids (both precisions, open, periodic and
closed sides, the limiter, divergence cleaning), steps on tetrahedral meshes, and the whole gradient of
the inverse-design objective.  A step case restarts from a state kept on the device, advances it and
stores the new state, as a checkpointed run does.  Results of FP32 contexts are returned in FP32.

``exact`` restates the scheme in 64-bit torch (global components, moments of the D2Q4 / D3Q4 velocity
set) without the package.
"""
import math

import numpy as np
import torch

from paper_2412_16845_gb300 import gks as G
from paper_2412_16845_gb300 import workloads as wl
from paper_2412_16845_gb300.gks import GKSSolver, SolverSpec

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
BCS = {"n": "nrbc", "p": "periodic", "m": "pec"}      # per side, in the order -x +x -y +y [-z +z]


def _cart(name, nx, ny, nz, prec, steps, bc, cfl, kappa=0.0, mu=False, limiter=False, clean=False,
          source="none", medium="cylinders"):
    c = {"kind": "cart", "nx": nx, "ny": ny, "nz": nz, "prec": prec, "steps": steps, "bc": bc,
         "cfl": cfl, "kappa": kappa, "mu": mu, "limiter": limiter, "clean": clean, "source": source,
         "medium": medium}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the scheme's verification run: a small periodic grid in double precision, host fields in
        # and out; launches and latency are all of it
        {"name": "tm2d_periodic_64_fp64", "kind": "whole", "nx": 64, "ny": 64, "steps": 200},
        # the oscillating dipole on the paper's grid, its energy read every 100 steps
        {"name": "tm2d_dipole_100_fp32", "kind": "monitor", "nx": 100, "ny": 100, "steps": 600,
         "every": 100},
        # the large scattering run: dielectric cylinders, line source, open sides
        _cart("tm2d_cylinders_4096_fp32", 4096, 4096, 1, "fp32", 20, "nnnn", 0.5, source="line"),
        # the same in double precision on a grid that fits no tile
        _cart("tm2d_cylinders_1531_fp64", 1531, 1022, 1, "fp64", 20, "nnnn", 0.5, source="line"),
        # discontinuous fields need the limiter; an odd grid
        _cart("tm2d_limiter_1801_fp32", 1801, 1203, 1, "fp32", 20, "nnnn", 0.5, limiter=True),
        # 3-D scattering by a dielectric sphere at full size
        _cart("maxwell3d_sphere_256_fp32", 256, 256, 256, "fp32", 10, "nnnnnn", 0.4, medium="sphere"),
        # the same in double precision, a ragged grid
        _cart("maxwell3d_sphere_130_fp64", 130, 118, 97, "fp64", 4, "nnnnnn", 0.4, medium="sphere"),
        # a small 3-D run, periodic across
        _cart("maxwell3d_small_45_fp32", 45, 34, 27, "fp32", 60, "nnpppp", 0.4, medium="sphere"),
        # divergence cleaning in 3-D
        _cart("cleaning3d_150_fp32", 150, 139, 128, "fp32", 6, "nnnnnn", 0.3, clean=True,
              medium="sphere"),
        # the unstructured workload at full size
        {"name": "tets_sphere_64_fp32", "kind": "tet", "m": 64, "prec": "fp32", "steps": 20},
        # a small mesh in double precision
        {"name": "tets_sphere_21_fp64", "kind": "tet", "m": 21, "prec": "fp64", "steps": 10},
        # inverse design: objective and whole gradient by checkpointed forward and adjoint steps
        {"name": "design_2048_fp32", "kind": "design", "n": 2048, "steps": 2000, "every": 45},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["whole", "monitor", "tm", "tm", "tm64", "tmx", "m3", "m3", "m64", "c3", "tet",
                       "tet64", "design"])
    if kind == "whole":
        return {"kind": "whole", "nx": _log(rng, 16, 128), "ny": _log(rng, 16, 128),
                "steps": _log(rng, 40, 400)}
    if kind == "monitor":
        return {"kind": "monitor", "nx": _log(rng, 40, 400), "ny": _log(rng, 40, 400),
                "steps": 4 * _log(rng, 10, 150), "every": _log(rng, 10, 150)}
    if kind in ("tet", "tet64"):
        m = _log(rng, 5, 64) if kind == "tet" else _log(rng, 5, 28)
        return {"kind": "tet", "m": m, "prec": "fp32" if kind == "tet" else "fp64",
                "steps": max(2, min(100, int(2e7 / (6 * m ** 3))))}
    if kind == "design":
        n = _log(rng, 96, 900)
        return {"kind": "design", "n": n, "steps": int(n * rng.uniform(0.7, 1.0)),
                "every": rng.randint(5, 60)}
    axes = lambda d: "".join(rng.choice(["nn", "nn", "pp", "mm", "nm"]) for _ in range(d))  # noqa: E731
    if kind in ("tm", "tm64", "tmx"):
        top = 4096 if kind == "tm" else 1800
        nx, ny = _log(rng, 40, top), _log(rng, 40, top)
        prec = "fp64" if kind == "tm64" else "fp32"
        steps = max(2, min(200, int((3e8 if prec == "fp32" else 2e7) / (nx * ny))))
        kw = {"kappa": rng.choice([0.0, 0.0, 0.05]), "source": rng.choice(["none", "line"])}
        if kind == "tmx":                            # an option of the step
            kw.update(rng.choice([{"limiter": True}, {"mu": True}, {"clean": True, "source": "none"}]))
            prec = rng.choice(["fp32", "fp32", "fp64"])
            steps = max(2, min(100, int((1e8 if prec == "fp32" else 1e7) / (nx * ny))))
        return _cart(None, nx, ny, 1, prec, steps, axes(2), 0.4 if kw.get("clean") else 0.5, **kw)
    top = {"m3": 256, "m64": 140, "c3": 170}[kind]
    n = [_log(rng, 14, top) for _ in range(3)]
    cells = n[0] * n[1] * n[2]
    prec = "fp64" if kind == "m64" else "fp32"
    bc = "".join(rng.choice(["nn", "nn", "pp"]) for _ in range(3)) if rng.random() < 0.7 else axes(3)
    kw = {"clean": True} if kind == "c3" else rng.choice([{}, {}, {}, {"mu": True}, {"limiter": True}])
    budget = {"m3": 1e8, "m64": 6e6, "c3": 2e7}[kind] / (4 if kw and kind == "m3" else 1)
    return _cart(None, n[0], n[1], n[2], prec, max(2, min(100, int(budget / cells))), bc,
                 0.3 if kind == "c3" else 0.4, medium="sphere", **kw)


# ------------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) + 20241216)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _centres(n, h):
    """Cell centres per axis, broadcastable over [nz][ny][nx] (or [ny][nx])."""
    d = len(n)
    out = []
    for a in range(d):
        s = [1] * d
        s[d - 1 - a] = n[a]
        out.append(((torch.arange(n[a], device=DEV, dtype=F64) + 0.5) * h).view(*s))
    return out


def _noise(g, n, h, waves=10, least=16.0):
    """Smooth noise in [0, 1]: plane waves of at least `least` cells a period."""
    x = _centres(n, h)
    p = 0.0
    for _ in range(waves):
        k = (_rand(g, len(n)) - 0.5) * (4.0 * math.pi / (least * h))
        p = p + torch.cos(sum(float(k[a]) * x[a] for a in range(len(n))) + 6.3 * float(_rand(g, 1)))
    return 0.5 + 0.5 * p / waves


def _waves(g, n, L, h, dim, extra):
    """A superposition of plane waves, periodic on the box, plus a pulse: [ncomp][cells]."""
    x = _centres(n, h)
    V = 0.0
    for _ in range(6):
        m = torch.round((_rand(g, dim) - 0.5) * 2.0 * torch.tensor(
            [max(1.0, v / 14.0) for v in n], device=DEV, dtype=F64))
        m[0] += (m.abs().sum() == 0)
        k = 2.0 * math.pi * m / torch.tensor(L, device=DEV, dtype=F64)
        u = (k / k.norm()).tolist()
        w = torch.cos(sum(float(k[a]) * x[a] for a in range(dim)) + 6.3 * float(_rand(g, 1)))
        if dim == 2:
            amp = [1.0, u[1], -u[0]]
        else:
            p = (_rand(g, 3) - 0.5).tolist()
            e = np.cross(u, p)
            e = e / np.linalg.norm(e)
            amp = list(e) + list(np.cross(u, e))
        V = V + torch.stack([a * w for a in amp])
    c = [float(v) * L[a] for a, v in enumerate(_rand(g, dim))]
    V[0 if dim == 2 else 2] += torch.exp(-sum((x[a] - c[a]) ** 2 for a in range(dim)) / (12.0 * h) ** 2)
    V = V.reshape(V.shape[0], -1)
    return torch.cat([V, torch.zeros(extra, V.shape[1], device=DEV, dtype=F64)]) if extra else V


def _line(n, h, share):
    i = int(share * n[0])
    m = torch.zeros(n[1], n[0], device=DEV, dtype=F64)
    m[:, i] = 1.0 / h
    return m.reshape(-1)


def _cart_inputs(case, seed):
    """The workload of a Cartesian step case, as torch tensors on the device."""
    g = _gen(seed)
    dim = 2 if case["nz"] == 1 else 3
    n = (case["nx"], case["ny"], case["nz"])[:dim]
    h = 1.0 / max(n)
    L = [v * h for v in n]
    eps = 1.0 + 0.1 * _noise(g, n, h)
    x = _centres(n, h)
    if case["medium"] == "sphere":
        r = 0.2 * min(L)
        eps = torch.where(sum((x[a] - 0.5 * L[a]) ** 2 for a in range(dim)) <= r * r, 2.25 + 0 * eps, eps)
    else:
        eps = torch.ones_like(eps)
        for _ in range(16):
            c, r, e = _rand(g, 2).tolist(), 0.01 + 0.04 * float(_rand(g, 1)), 2.0 + 4.0 * float(_rand(g, 1))
            r *= min(L)
            eps[(x[0] - c[0] * L[0]) ** 2 + (x[1] - c[1] * L[1]) ** 2 <= r * r] = e
    mu = 1.0 + _noise(g, n, h).reshape(-1) if case["mu"] else None
    extra = (1 if dim == 2 else 2) if case["clean"] else 0
    f = _waves(g, n, L, h, dim, extra)
    if case["limiter"]:                              # a jump across the grid
        f = f * torch.where(x[0] < 0.4 * L[0], 1.0, -0.5).expand(tuple(n)[::-1]).reshape(-1)
    src = _line(n, h, 0.25) if case["source"] == "line" else None
    return {"dim": dim, "n": n, "h": h, "L": L, "eps": eps.reshape(-1).contiguous(), "mu": mu, "f": f,
            "src": src, "phm": (1.0, 1.0) if case["clean"] else None}


def _whole_inputs(case, seed):
    """Periodic unit-height box in vacuum: an oblique wave and a pulse at a seeded place."""
    n = (case["nx"], case["ny"])
    h = 1.0 / max(n)
    return {"dim": 2, "n": n, "h": h, "L": [v * h for v in n],
            "f": _waves(_gen(seed), n, [v * h for v in n], h, 2, 0)}


def _monitor_inputs(case, seed):
    """A dipole on 2 x 2 cells in vacuum, its place, period and strength from the seed."""
    g = _gen(seed)
    n = (case["nx"], case["ny"])
    h = 1.0 / max(n)
    u = _rand(g, 4).tolist()
    i, j = int(n[0] * (0.3 + 0.4 * u[0])), int(n[1] * (0.3 + 0.4 * u[1]))
    m = torch.zeros(n[1], n[0], device=DEV, dtype=F64)
    m[j - 1:j + 1, i - 1:i + 1] = 1.0
    return {"dim": 2, "n": n, "h": h, "L": [v * h for v in n], "src": m.reshape(-1),
            "cw": (0.5 + u[2], 1.0 / ((12.0 + 12.0 * u[3]) * h), 0.0),
            "f": torch.zeros(3, n[0] * n[1], device=DEV, dtype=F64)}


def _tet_inputs(case, seed):
    """The unit cube in m^3 hexes of six tetrahedra each, inner vertices jittered, a sphere inside."""
    m = case["m"]
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    n1 = m + 1
    i, j, k = (a.ravel() for a in np.meshgrid(*[np.arange(n1)] * 3, indexing="ij"))
    vert = np.stack([i, j, k], axis=1) / m
    inner = ((vert > 0) & (vert < 1)).all(axis=1)
    vert[inner] += rng.uniform(-0.1 / m, 0.1 / m, size=(int(inner.sum()), 3))
    hex_ = np.stack([a.ravel() for a in np.meshgrid(*[np.arange(m)] * 3, indexing="ij")], axis=1)
    tets = []
    for order in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        at = hex_.copy()
        ids = [(at[:, 0] * n1 + at[:, 1]) * n1 + at[:, 2]]
        for a in order:
            at[:, a] += 1
            ids.append((at[:, 0] * n1 + at[:, 1]) * n1 + at[:, 2])
        tets.append(np.stack(ids, axis=1))
    tet = np.stack(tets, axis=1).reshape(-1, 4).astype(np.int64)
    mid = vert[tet].mean(axis=1)
    eps = np.where(((mid - 0.5) ** 2).sum(axis=1) <= 0.25 ** 2, 4.0, 1.0)
    ez = np.exp(-((mid[:, 0] - rng.uniform(0.15, 0.5)) / 0.1) ** 2) + 0.3 * np.sin(9.0 * mid[:, 1] + rng.uniform(0, 6))
    f = np.zeros((6, tet.shape[0]))
    f[2], f[4] = ez, -ez
    f[1] = 0.5 * np.cos(7.0 * mid[:, 2] + rng.uniform(0, 6))
    return {"vert": vert, "tet": tet, "eps": eps, "f": f}


def _design_inputs(case, seed):
    """Line source, design square of smoothed noise, probe disc, open sides."""
    g = _gen(seed)
    n = (case["n"], case["n"])
    h = 1.0 / case["n"]
    i0, i1, j0, j1 = (int(round(v * case["n"])) for v in (0.3125, 0.5625, 0.375, 0.625))
    eps = torch.ones(n[1], n[0], device=DEV, dtype=F64)
    eps[j0:j1, i0:i1] = 1.0 + 3.0 * _noise(g, (i1 - i0, j1 - j0), h)
    ids = torch.arange(n[0] * n[1], device=DEV).view(n[1], n[0])
    x = _centres(n, h)
    r = max(0.02, 2.0 * h)
    return {"dim": 2, "n": n, "h": h, "L": [1.0, 1.0], "eps": eps.reshape(-1), "src": _line(n, h, 0.30),
            "design": ids[j0:j1, i0:i1].reshape(-1),
            "probe": ids[(x[0] - 0.5) ** 2 + (x[1] - 0.5) ** 2 <= r * r],
            "f": torch.zeros(3, n[0] * n[1], device=DEV, dtype=F64)}


# ------------------------------------------------------------------------------ prepare and run
def _host(t):
    return None if t is None else t.cpu().numpy()


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _state(s, n, prec):
    """The context's state now, and room for the state after a pass; the result seen per component."""
    count, _ = G.gks_state_layout(s.ctx)
    dt = F64 if prec == "fp64" else torch.float32
    init, out = (torch.zeros(count, dtype=dt, device="cuda") for _ in range(2))
    G.gks_copy_state(s.ctx, init.data_ptr())
    rows = tuple(n)[:0:-1]
    view = out.view(s.ncomp, *rows, count // (s.ncomp * int(np.prod(rows))))[..., :n[0]]
    return {"s": s, "init": init, "out": out, "view": view}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "design":
        from paper_2412_16845_gb300.adjoint import DesignProblem
        d = _design_inputs(case, seed)
        w = wl.CartWorkload(name="design", dim=2, n=d["n"], lo=(0.0, 0.0), hi=(1.0, 1.0), bc=("nrbc",) * 4,
                            cfl=0.5, steps=case["steps"], eps=_host(d["eps"]), mu=None,
                            fields0=_host(d["f"]), jz_mask=_host(d["src"]), probe=_host(d["probe"]),
                            design=_host(d["design"]))
        p = DesignProblem(w, precision="fp32", checkpoint_every=case["every"])
        return {"kind": kind, "p": p, "eps": d["eps"][d["design"]].float().requires_grad_(True)}
    if kind == "tet":
        d = _tet_inputs(case, seed)
        s = GKSSolver.from_tets(d["vert"], d["tet"], 0.4, precision=case["prec"], stream=_stream())
        s.set_materials(d["eps"])
        # the cells' order in the state buffers: the state of the fields 0, 1, 2, ... (two parts, so
        # that single precision holds them)
        ids = np.zeros_like(d["f"])
        ids[0], ids[1] = np.arange(s.ncell) % 4096, np.arange(s.ncell) // 4096
        s.write_fields(ids)
        st = _state(s, (s.ncell,), case["prec"])
        order = st["init"].view(6, -1)
        order = (order[0] + 4096.0 * order[1].double()).round().long()
        st["user"] = torch.empty_like(order)
        st["user"][order] = torch.arange(s.ncell, device="cuda")
        s.write_fields(d["f"])
        G.gks_copy_state(s.ctx, st["init"].data_ptr())
        torch.cuda.synchronize()
        return {"kind": kind, "steps": case["steps"], **st}
    d = {"whole": _whole_inputs, "monitor": _monitor_inputs, "cart": _cart_inputs}[kind](case, seed)
    n = d["n"]
    spec = SolverSpec(dim=d["dim"], n=n, lo=(0.0,) * d["dim"], hi=tuple(d["L"]),
                      bc=tuple(BCS[b] for b in {"whole": "pppp", "monitor": "nnnn"}.get(kind) or case["bc"]),
                      cfl=case.get("cfl", 0.5), kappa=case.get("kappa", 0.0), c_lattice=1.0,
                      precision={"whole": "fp64", "monitor": "fp32"}.get(kind) or case["prec"],
                      phm=d.get("phm"), limiter="vanleer" if case.get("limiter") else None)
    s = GKSSolver(spec, stream=_stream())
    ones = np.ones(s.ncell)
    s.set_materials(_host(d["eps"]) if "eps" in d else ones, _host(d.get("mu")))
    f = _host(d["f"])
    s.write_fields(f)
    if kind == "whole":
        return {"kind": kind, "s": s, "f": f, "steps": case["steps"], "out": np.empty_like(f)}
    if "cw" in d:
        s.set_source_cw(_host(d["src"]), *d["cw"])
    elif d["src"] is not None:
        s.set_source(_host(d["src"]), wl.SRC_A, wl.SRC_F0, wl.SRC_T0, wl.SRC_S)
    return {"kind": kind, "steps": case["steps"], "every": case.get("every"), **_state(s, n, spec.precision)}


def run(state):
    kind, s = state["kind"], state.get("s")
    if kind == "design":
        from paper_2412_16845_gb300.adjoint import GKSEnergyObjective
        eps = state["eps"]
        eps.grad = None
        loss = GKSEnergyObjective.apply(eps, state["p"]).to(eps.dtype)
        loss.backward()
        return {"J": loss.detach(), "grad": eps.grad}
    if kind == "whole":
        s.write_fields(state["f"])
        s.step(state["steps"])
        return s.read_fields(state["out"])
    G.gks_load_state(s.ctx, state["init"].data_ptr(), 0)
    if kind == "monitor":
        energy, done = [], 0
        while done < state["steps"]:
            k = min(state["every"], state["steps"] - done)
            s.step(k)
            done += k
            energy.append(s.energy())
        G.gks_copy_state(s.ctx, state["out"].data_ptr())
        return {"fields": state["view"], "energy": np.asarray(energy, dtype=np.float32)}
    s.step(state["steps"])
    G.gks_copy_state(s.ctx, state["out"].data_ptr())
    if kind == "tet":
        return state["view"].index_select(1, state["user"])
    return state["view"]


def work(case):
    """Per step and cell: the fields read and written once, the materials read; the operations of the
    face fluxes (each face once) and of the update."""
    kind, k = case["kind"], case["steps"]
    if kind == "design":                             # forward and adjoint step: fields, lambda, eps
        return {"bytes": 56.0 * k * case["n"] ** 2, "flops": 320.0 * k * case["n"] ** 2}
    if kind == "tet":                                # geometry, neighbours and fields in one pass
        cells = 6.0 * case["m"] ** 3
        return {"bytes": (229.0 if case["prec"] == "fp32" else 438.0) * k * cells, "flops": 1000.0 * k * cells}
    cells = float(case["nx"] * case["ny"] * case.get("nz", 1))
    dim = 3 if case.get("nz", 1) > 1 else 2
    nc = (3 if dim == 2 else 6) + (dim - 1 if case.get("clean") else 0)
    size = 8 if kind == "whole" or case.get("prec") == "fp64" else 4
    flops = (150.0 if dim == 2 else 500.0) * (nc / (3.0 if dim == 2 else 6.0)) ** 2
    return {"bytes": k * cells * size * (2 * nc + 1 + bool(case.get("mu"))), "flops": k * cells * flops}


# ------------------------------------------------------------------------------------- 64 bits
def _times(dt, tau):
    """The integrals over [0, dt] of 1 - e, (tau + t) e - tau, t + tau (e - 1), e and t e, e = exp(-t/tau)."""
    if tau == 0.0:
        return dt, 0.0, 0.5 * dt * dt, 0.0, 0.0
    e = math.exp(-dt / tau)
    c4, c5 = tau * (1.0 - e), tau * tau * (1.0 - e) - tau * dt * e
    return dt - c4, tau * c4 + c5 - tau * dt, 0.5 * dt * dt + tau * c4 - tau * dt, c4, c5


def _jacobians(nc, dim, phm):
    """F_j as matrices over the carried components, j = x, y, z."""
    full = np.zeros((3, 8, 8))
    for j in range(3):
        a, b = (j + 1) % 3, (j + 2) % 3
        full[j, a, 3 + b], full[j, b, 3 + a] = 1.0, -1.0          # the curl of H in the E rows
        full[j, 3 + b, a], full[j, 3 + a, b] = 1.0, -1.0          # minus the curl of E in the H rows
        chi, gam = phm or (0.0, 0.0)
        full[j, j, 6] = full[j, 6, j] = chi
        full[j, 3 + j, 7] = full[j, 7, 3 + j] = gam
    keep = ([2, 3, 4, 7] if dim == 2 else list(range(8)))[:nc]
    return torch.tensor(full[:, keep][:, :, keep], device=DEV, dtype=F64)


class _Faces:
    """The time-integrated flux through faces of one orientation; frame: the rows n, t, w."""

    def __init__(self, F, frame, dim, C, c=1.0):
        u = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], dtype=np.float64) * c
        if dim == 2:
            u[:, 2] = 0.0
        v = u @ np.asarray(frame, dtype=np.float64)
        t = lambda a: torch.tensor(a, device=DEV, dtype=F64)  # noqa: E731
        pos = u[:, 0] > 0
        self.F, self.C, self.c, self.n = F, C, c, t(frame[0])
        self.Fn = torch.einsum("i,iab->ab", self.n, F)
        mix = lambda q: torch.einsum("ij,iab->jab", t(q), F) / (4.0 * c * c)  # noqa: E731
        self.P = [mix(np.einsum("ki,kj->ij", v[s], v[s])) for s in (pos, ~pos)]
        self.Q = mix(np.einsum("k,ki,kj->ij", u[:, 0], v, v))

    def flux(self, Xl, ml, Xr, mr, ms):
        """X: the state at the face and its three derivatives, [4, ncomp, faces]; m: [ncomp, faces]."""
        c, (C1, C2, C3, C4, C5), Fn = self.c, self.C, self.Fn
        on = lambda A, x: torch.tensordot(A, x, dims=1)  # noqa: E731
        over = lambda A, x: sum(on(A[j], x[j]) for j in range(3) if bool(A[j].any()))  # noqa: E731
        W = [0.5 * (ml * a + mr * b) + on(Fn, a - b) / (2.0 * c) for a, b in zip(Xl, Xr)]
        V = [w / ms for w in W]
        along = lambda x: sum(float(self.n[j]) * x[j] for j in range(3) if float(self.n[j]))  # noqa: E731
        out = C1 * on(Fn, V[0]) - C3 * on(Fn, over(self.F, V[1:]) / ms)
        if C2 or C4 or C5:
            out = out + C2 * (c * c * along(W[1:]) + over(self.Q, V[1:]))
            out = out + C4 * (0.5 * c * (ml * Xl[0] - mr * Xr[0]) + 0.5 * on(Fn, Xl[0] + Xr[0]))
            out = out - C5 * (0.5 * c * c * along([ml * a + mr * b for a, b in zip(Xl[1:], Xr[1:])])
                              + c * (over(self.P[0], Xl[1:]) - over(self.P[1], Xr[1:])))
        return out


#: face frames of the grid's axes, interior (and high) sides, and the outward ones of the low sides
_HIGH = [[(1, 0, 0), (0, 1, 0), (0, 0, 1)], [(0, 1, 0), (-1, 0, 0), (0, 0, 1)], [(0, 0, 1), (0, 1, 0), (-1, 0, 0)]]
_LOW = [[(-1, 0, 0), (0, -1, 0), (0, 0, 1)], [(0, -1, 0), (1, 0, 0), (0, 0, 1)], [(0, 0, -1), (0, 1, 0), (1, 0, 0)]]


class _Grid:
    def __init__(self, d, bc, cfl, kappa=0.0, limiter=False):
        self.dim, self.n, self.h, self.bc, self.limiter = d["dim"], d["n"], d["h"], bc, limiter
        self.dt = cfl * self.h
        self.nc = d["f"].shape[0]
        C = _times(self.dt, kappa * self.dt)
        F = _jacobians(self.nc, self.dim, d.get("phm"))
        self.high = [_Faces(F, f, self.dim, C) for f in _HIGH[:self.dim]]
        self.low = [_Faces(F, f, self.dim, C) for f in _LOW[:self.dim]]
        names = (["Ez", "Hx", "Hy", "psi"] if self.dim == 2 else
                 ["Ex", "Ey", "Ez", "Hx", "Hy", "Hz", "phi", "psi"])[:self.nc]
        self.e = [v[0] == "E" for v in names]
        self.hh = [v[0] == "H" for v in names]
        odd = lambda a, v: (v[0] == "E") != (v[1:] == "xyz"[a]) if v[0] in "EH" else v == "phi"  # noqa: E731
        self.sign = [torch.tensor([-1.0 if odd(a, v) else 1.0 for v in names], device=DEV, dtype=F64)
                     for a in range(self.dim)]

    def mass(self, eps, mu=None):
        one = torch.ones_like(eps)
        rows = [eps if e else (mu if mu is not None and h else one) for e, h in zip(self.e, self.hh)]
        return torch.stack(rows).view(self.nc, *tuple(self.n)[::-1])

    def ghost(self, X, fields):
        """Two layers beyond every side: the wrapped cells, the edge cell, or the wall's mirror image."""
        for a in range(self.dim):
            ax, n = self.dim - a, self.n[a]
            at = torch.arange(-2, n + 2, device=DEV)
            lo, hi = self.bc[2 * a], self.bc[2 * a + 1]
            idx = at % n if lo == "p" else torch.where(
                at < 0, (-1 - at).clamp(max=n - 1) if lo == "m" else 0 * at,
                torch.where(at >= n, (2 * n - 1 - at).clamp(min=0) if hi == "m" else 0 * at + n - 1, at))
            X = X.index_select(ax, idx)
            if fields:
                for side, sl in ((lo, slice(0, 2)), (hi, slice(n + 2, n + 4))):
                    if side == "m":
                        s = torch.ones(self.nc, n + 4, device=DEV, dtype=F64)
                        s[:, sl] = self.sign[a][:, None]
                        shape = [self.nc] + [1] * self.dim
                        shape[ax] = n + 4
                        X = X * s.view(shape)
        return X

    def step(self, V, M, Mg, jz):
        """V, M [ncomp][nz][ny][nx]; Mg: M with its ghosts."""
        P = self.ghost(V, True)
        cut = lambda X, ax, lo, hi: X.narrow(ax, lo, X.shape[ax] - lo - hi)  # noqa: E731
        grads = []
        inner = P
        for a in range(self.dim):
            inner = cut(inner, self.dim - a, 1, 1)
        for a in range(self.dim):
            Q = P
            for b in range(self.dim):
                if b != a:
                    Q = cut(Q, self.dim - b, 1, 1)
            up, dn = cut(Q, self.dim - a, 2, 0), cut(Q, self.dim - a, 0, 2)
            if self.limiter:
                p, m = up - inner, inner - dn
                same = p * m > 0
                grads.append(torch.where(same, 2.0 * p * m / torch.where(same, p + m, 1.0), 0.0) / self.h)
            else:
                grads.append((up - dn) / (2.0 * self.h))
        while len(grads) < 3:
            grads.append(torch.zeros_like(inner))
        out = M * V
        for a in range(self.dim):
            ax = self.dim - a

            def strip(X):                            # the cells beside this axis' faces: no ghosts across
                for b in range(self.dim):
                    if b != a:
                        X = cut(X, self.dim - b, 1, 1)
                return X

            def strip2(X):
                for b in range(self.dim):
                    X = cut(X, self.dim - b, 1, 1) if b == a else cut(X, self.dim - b, 2, 2)
                return X

            C, D, m = strip(inner), [strip(g) for g in grads], strip2(Mg)
            L = [cut(C + 0.5 * self.h * D[a], ax, 0, 1)] + [cut(x, ax, 0, 1) for x in D]
            R = [cut(C - 0.5 * self.h * D[a], ax, 1, 0)] + [cut(x, ax, 1, 0) for x in D]
            ml, mr = cut(m, ax, 0, 1), cut(m, ax, 1, 0)
            F = self.high[a].flux(L, ml, R, mr, 0.5 * (ml + mr))
            k = self.n[a]
            lowf, highf = F.narrow(ax, 0, 1), F.narrow(ax, k, 1)
            if self.bc[2 * a + 1] == "n":
                one = [x.narrow(ax, k, 1) for x in L]
                z = [torch.zeros_like(one[0])] * 4
                w = ml.narrow(ax, k, 1)
                highf = self.high[a].flux(one, w, z, torch.zeros_like(w), w)
            if self.bc[2 * a] == "n":
                one = [x.narrow(ax, 0, 1) for x in R]
                z = [torch.zeros_like(one[0])] * 4
                w = mr.narrow(ax, 0, 1)
                lowf = -self.low[a].flux(one, w, z, torch.zeros_like(w), w)
            F = torch.cat([lowf, F.narrow(ax, 1, k - 1), highf], dim=ax)
            out = out - (F.narrow(ax, 1, k) - F.narrow(ax, 0, k)) / self.h
        if jz is not None:
            e = self.e.index(True) if self.dim == 2 else 2
            out = torch.cat([out[:e], out[e:e + 1] - self.dt * jz, out[e + 1:]])
        return out / M


def _gauss(t):
    """The line source of the 2-D workloads."""
    return math.exp(-((t - 0.075) / 0.025) ** 2) * math.sin(40.0 * math.pi * (t - 0.075))


def exact(case, seed):
    kind, k = case["kind"], case["steps"]
    if kind == "tet":
        return _exact_tet(case, seed)
    if kind == "design":
        return _exact_design(case, seed) if case["n"] ** 2 * k <= 4.5e8 else None
    d = {"whole": _whole_inputs, "monitor": _monitor_inputs, "cart": _cart_inputs}[kind](case, seed)
    shape = tuple(d["n"])[::-1]
    g = _Grid(d, {"whole": "pppp", "monitor": "nnnn"}.get(kind) or case["bc"], case.get("cfl", 0.5),
              case.get("kappa", 0.0), case.get("limiter", False))
    cells = int(np.prod(shape))
    one = torch.ones(cells, device=DEV, dtype=F64)
    M = g.mass(d.get("eps", one), d.get("mu"))
    Mg = g.ghost(M, False)
    V = d["f"].view(-1, *shape)
    src = d.get("src")
    src = None if src is None else src.view(shape)
    energy = []
    for s in range(k):
        jz = None
        if src is not None:
            t = s * g.dt
            jz = src * (d["cw"][0] * math.cos(2.0 * math.pi * d["cw"][1] * t) if "cw" in d else _gauss(t))
        V = g.step(V, M, Mg, jz)
        if kind == "monitor" and ((s + 1) % case["every"] == 0 or s + 1 == k):
            energy.append(0.5 * g.h ** 2 * float((M * V * V).sum()))
    if kind == "whole":
        return V.reshape(V.shape[0], -1).cpu().numpy()
    return {"fields": V, "energy": np.asarray(energy)} if kind == "monitor" else V


def _exact_design(case, seed):
    from torch.utils.checkpoint import checkpoint
    d = _design_inputs(case, seed)
    g = _Grid(d, "nnnn", 0.5)
    shape = tuple(d["n"])[::-1]
    e = d["eps"][d["design"]].float().double().requires_grad_(True)     # as the design is handed over
    src = d["src"].view(shape)

    def one(V, e, t):
        M = g.mass(d["eps"].clone().index_put((d["design"],), e))
        return g.step(V, M, g.ghost(M, False), src * _gauss(t))

    V, J = d["f"].view(-1, *shape), 0.0
    for s in range(case["steps"]):
        V = checkpoint(one, V, e, s * g.dt, use_reentrant=False)
        J = J + g.dt * g.h ** 2 * (V[0].reshape(-1)[d["probe"]] ** 2).sum()
    J.backward()
    return {"J": J.detach(), "grad": e.grad}


def _exact_tet(case, seed):
    d = _tet_inputs(case, seed)
    t = lambda a, dt=F64: torch.tensor(a, device=DEV, dtype=dt)  # noqa: E731
    vert, tet = t(d["vert"]), t(d["tet"], torch.long)
    nt, nv = tet.shape[0], vert.shape[0]
    p = vert[tet]
    mid = p.mean(1)
    vol = (torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]) * (p[:, 3] - p[:, 0])).sum(1).abs() / 6.0
    tri = torch.cat([tet[:, list(o)] for o in ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))]).sort(1).values
    own = torch.arange(nt, device=DEV).repeat(4)
    key, order = ((tri[:, 0] * nv + tri[:, 1]) * nv + tri[:, 2]).sort(stable=True)
    pair = torch.zeros(key.numel(), dtype=torch.bool, device=DEV)
    pair[:-1] = key[1:] == key[:-1]
    second = torch.zeros_like(pair)
    second[1:] = pair[:-1]
    first = (~second).nonzero().view(-1)
    a = own[order[first]]
    b = torch.where(pair[first], own[order[(first + 1).clamp(max=key.numel() - 1)]], -1)
    L = torch.where(b >= 0, torch.minimum(a, b), a)
    R = torch.where(b >= 0, torch.maximum(a, b), -1)
    q = vert[tri[order[first]]]
    cr = torch.linalg.cross(q[:, 1] - q[:, 0], q[:, 2] - q[:, 0])
    xs = q.mean(1)
    cr = cr * torch.where((cr * (xs - mid[L])).sum(1) < 0, -1.0, 1.0)[:, None]
    area = 0.5 * cr.norm(dim=1)
    n = cr / (2.0 * area)[:, None]
    inside = (R >= 0).double()
    Rc = R.clamp(min=0)
    h = torch.zeros(nt, device=DEV, dtype=F64).index_add_(0, L, area).index_add_(0, Rc, area * inside)
    dt = 0.4 * float((6.0 * vol / h).min())
    F = _jacobians(6, 3, None)
    m = torch.ones(6, nt, device=DEV, dtype=F64)
    m[:3] = t(d["eps"])
    V = t(d["f"])
    nT = n.T                                         # [3, faces]
    Fn = lambda x: torch.stack([sum(float(F[j, r, s]) * nT[j] * x[s] for j in range(3) for s in range(6)  # noqa: E731
                                    if float(F[j, r, s])) for r in range(6)])
    Fj = lambda x: sum(torch.tensordot(F[j], x[j], dims=1) for j in range(3))  # noqa: E731
    ml, mr = m[:, L], m[:, Rc] * inside
    ms = torch.where(inside > 0, 0.5 * (ml + mr), ml)
    dl, dr = (xs - mid[L]).T, (xs - mid[Rc]).T

    def sides(x, at, dx, w):
        y = [g[:, at] for g in x[1]]
        return [(x[0][:, at] + sum(dx[j] * y[j] for j in range(3))) * w] + [v * w for v in y]

    for _ in range(case["steps"]):
        face = torch.where(inside > 0, 0.5 * (V[:, L] + V[:, Rc]), V[:, L])
        grad = []
        for j in range(3):
            w = face * (nT[j] * area)
            grad.append((torch.zeros_like(V).index_add_(1, L, w).index_add_(1, Rc, -w * inside)) / vol)
        Xl, Xr = sides((V, grad), L, dl, 1.0), sides((V, grad), Rc, dr, inside)
        V0 = [(0.5 * (ml * x + mr * y) + 0.5 * Fn(x - y)) / ms for x, y in zip(Xl, Xr)]
        flux = (dt * Fn(V0[0]) - 0.5 * dt * dt * Fn(Fj(V0[1:]) / ms)) * area
        net = torch.zeros_like(V).index_add_(1, L, flux).index_add_(1, Rc, -flux * inside)
        V = V - net / vol / m
    return V
