"""The calls that users of this library make, as cases to be timed.

A case is a dict of plain values; ``prepare`` makes what a program has in hand
before the call (a handle with its fields loaded, or its own state buffers),
``run`` makes one pass through the public entry points and returns the updated
state, and ``exact`` is the same pass in 64-bit torch arithmetic, written here
from the scheme (arXiv 2403.16122, Section 3) without the library.

Kinds of pass:
  handle      lbm_step(n) on a handle over one lattice, or over a batch;
              with "observe", lbm_observables_all after it, as a program does
              that follows volume and solid fraction in time
  noalloc     steps of lbm_step_noalloc between the caller's two state buffers
  checkpoint  lbm_set_state and lbm_get_state of one lattice through host
              arrays (a restart, then a checkpoint)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2403_16122_gb300 import lbm

STORAGE = {"fp32": lbm.LBM_STORE_FP32, "fp16": lbm.LBM_STORE_FP16, "bf16": lbm.LBM_STORE_BF16}
POP_TYPE = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
# Bytes a lattice update reads and writes: 27 populations and 5 carried fields
# in FP32, or 24 16-bit populations and 10 FP32 values. Arithmetic operations
# of one update (stencils 60, closure and forces 110, nine directions of three
# sets 400), rounded.
BYTES_LU = {"fp32": 256, "fp16": 176, "bf16": 176}
FLOPS_LU = 570
# Lattices of a batch whose whole state a pass returns (two arrays each); the
# records of all of them are returned.
STATES = 24
LARGEST = 2501 * 2501 * 10  # lattice updates of the largest listed case


def listed():
    return [
        # Section 4.1's Stefan problem, the smallest lattice of all, walls in x,
        # advanced in calls of 100 steps: 2048 sites, latency and launches
        {"name": "stefan_256x8", "kind": "handle", "problem": "stefan", "nx": 256, "ny": 8,
         "storage": "fp32", "steps": 100},
        # Section 4.3's column with bubbles and buoyancy at the default l = 32
        {"name": "column_128x96", "kind": "handle", "problem": "column", "nx": 128, "ny": 96,
         "storage": "fp32", "steps": 50},
        # the sessile drop at 256 x 256, the observables read after every step
        {"name": "sessile_256_each_step", "kind": "handle", "problem": "sessile", "nx": 256,
         "ny": 256, "storage": "fp32", "steps": 1, "observe": True},
        # a closed box (walls on all four sides, corners, wetting, per-phase
        # thermal properties) of odd sizes
        {"name": "closed_203x151", "kind": "handle", "problem": "closed", "nx": 203, "ny": 151,
         "storage": "fp32", "steps": 20},
        # four allocation-free steps on the caller's own buffers
        {"name": "noalloc_512", "kind": "noalloc", "problem": "sessile", "nx": 512, "ny": 512,
         "storage": "fp32", "steps": 4},
        # the drop with bubbles at 1024 x 1024, observables every 20 steps, in
        # FP32 and in 16-bit storage
        {"name": "drop_1024_fp32", "kind": "handle", "problem": "bubbles", "nx": 1024, "ny": 1024,
         "storage": "fp32", "steps": 20, "observe": True},
        {"name": "drop_1024_fp16", "kind": "handle", "problem": "bubbles", "nx": 1024, "ny": 1024,
         "storage": "fp16", "steps": 20, "observe": True},
        # larger lattices of ragged sizes: BF16 storage, and the largest in FP32
        {"name": "drop_1900x1701_bf16", "kind": "handle", "problem": "bubbles", "nx": 1900,
         "ny": 1701, "storage": "bf16", "steps": 10},
        {"name": "drop_2501_fp32", "kind": "handle", "problem": "bubbles", "nx": 2501, "ny": 2501,
         "storage": "fp32", "steps": 10},
        # a parametric sweep: independent sessile drops on square grids of
        # 128 .. 512, the steps in one persistent launch replayed from a graph
        {"name": "sweep_48_fp32", "kind": "handle", "problem": "sweep", "lattices": 48,
         "lo": 128, "hi": 512, "storage": "fp32", "steps": 21, "exec": "persistent", "chunk": 20,
         "observe": True},
        # drops with 0-4 bubbles on uneven grids of 64 .. 256 per side, FP16
        {"name": "batch_256_fp16", "kind": "handle", "problem": "batch", "lattices": 256,
         "lo": 64, "hi": 256, "storage": "fp16", "steps": 21, "observe": True},
        # restart from a checkpoint and write one
        {"name": "checkpoint_384x300", "kind": "checkpoint", "problem": "sessile", "nx": 384,
         "ny": 300, "storage": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stefan", "closed", "column", "sessile", "sessile", "bubbles", "bubbles",
                       "bubbles", "sweep", "batch", "noalloc", "checkpoint"])
    if kind == "checkpoint":
        return {"kind": "checkpoint", "problem": "sessile", "nx": _log(rng, 64, 700),
                "ny": _log(rng, 64, 700), "storage": "fp32"}
    if kind == "noalloc":
        return {"kind": "noalloc", "problem": rng.choice(["sessile", "closed"]),
                "nx": _log(rng, 64, 1400), "ny": _log(rng, 64, 1400), "storage": "fp32",
                "steps": rng.choice([2, 4])}
    if kind in ("sweep", "batch"):
        sweep = kind == "sweep"
        mode = rng.choice(["launch", "graph", "persistent"])
        case = {"kind": "handle", "problem": kind, "lattices": rng.randint(8, 48 if sweep else 256),
                "lo": 128 if sweep else 64, "hi": 512 if sweep else 256,
                "storage": rng.choice(["fp32", "fp16"]), "steps": rng.randint(11, 25),
                "observe": True}
        if mode != "launch":
            case.update(exec=mode, chunk=10)
        return case
    nx, ny = {"stefan": lambda: (_log(rng, 64, 800), rng.randint(4, 40)),
              "closed": lambda: (_log(rng, 48, 600), _log(rng, 48, 600)),
              "column": lambda: (lambda l: (4 * l, 3 * l))(_log(rng, 16, 150)),
              "sessile": lambda: (_log(rng, 64, 700), _log(rng, 64, 700)),
              "bubbles": lambda: (_log(rng, 96, 2500), _log(rng, 96, 2500))}[kind]()
    periodic_x = kind not in ("stefan", "closed")
    steps = rng.choice([1, 5, 20, 50, 100])
    steps = max(1, min(steps, LARGEST // (2 * nx * ny)))
    return {"kind": "handle", "problem": kind, "nx": nx, "ny": ny,
            "storage": rng.choice(["fp32", "fp32", "fp16", "bf16"]) if periodic_x else "fp32",
            "steps": steps, "observe": rng.random() < 0.5}


# ----------------------------------------------------------------------------
# Problem statements: parameters and initial fields, from the seed alone
# ----------------------------------------------------------------------------

BASE = dict(
    nx=64, ny=64, periodic_x=1, periodic_y=0,
    dirichlet_x_lo=0, dirichlet_x_hi=0, dirichlet_y_lo=1, dirichlet_y_hi=0, st_mask_liquid=0,
    W=4.0, sigma=0.01, mobility=0.02, tau_f_liquid=0.8, tau_h=0.8,
    rho_l=1.0, rho_ratio_lg=10.0, rho_ratio_sl=0.9, mu_ratio_lg=10.0, Ste=0.1,
    Cp=1.0, Cp_ref=1.0, T_m=0.0, T_w=-1.0, theta_deg=90.0, pc_ramp=0.2, normal_eps=1e-3,
    gx=0.0, gy=0.0, beta_T=0.0, T_ref=0.0, rho_0=1.0,
    Cp_ratio_sl=1.0, Cp_ratio_gl=1.0, k_ratio_sl=1.0, k_ratio_gl=1.0,
)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _disk(p, xc, yc, r, inside=True):
    """tanh profile of width W: 1 inside a circle and 0 outside, or reversed."""
    y = torch.arange(p["ny"], dtype=torch.float64, device=_device())[:, None]
    x = torch.arange(p["nx"], dtype=torch.float64, device=_device())[None, :]
    d = r - torch.sqrt((x - xc) ** 2 + (y - yc) ** 2)
    return 0.5 + 0.5 * torch.tanh((2.0 if inside else -2.0) * d / p["W"])


def _drop(p, rng, r, n_bub, r_lo, r_hi):
    """Drop of radius r on the wall at y = -1/2, meeting it at the contact
    angle, with n_bub bubbles inside that touch neither its surface, the wall
    nor each other."""
    xc, yc = 0.5 * (p["nx"] - 1), -0.5 - r * math.cos(math.radians(p["theta_deg"]))
    phi = _disk(p, xc, yc, r)
    placed = []
    for _ in range(400):
        if len(placed) >= n_bub:
            break
        b = rng.uniform(r_lo, r_hi)
        x, y = rng.uniform(xc - r, xc + r), rng.uniform(-0.5, yc + r)
        if math.hypot(x - xc, y - yc) > r - b - p["W"] or y - b - p["W"] < -0.5:
            continue
        if any(math.hypot(x - q[0], y - q[1]) < b + q[2] + p["W"] for q in placed):
            continue
        placed.append((x, y, b))
        phi = phi * _disk(p, x, y, b, inside=False)
    return phi


def _problem(problem, nx, ny, rng):
    """(parameters, phi0, T0), the fields as FP64 tensors [ny, nx]."""
    p = dict(BASE, nx=int(nx), ny=int(ny))
    T = 0.0
    n = min(nx, ny)
    if problem == "stefan":  # cold wall at x = -1/2, liquid on the first half
        p.update(periodic_x=0, periodic_y=1, dirichlet_x_lo=1, dirichlet_y_lo=0,
                 Ste=rng.uniform(0.1, 0.2))
        x = torch.arange(nx, dtype=torch.float64, device=_device())
        h0 = nx * rng.uniform(0.45, 0.55)
        phi = (0.5 + 0.5 * torch.tanh(2.0 * (h0 - 0.5 - x) / p["W"])).expand(ny, nx).contiguous()
        T = rng.uniform(0.0, 0.1)
    elif problem == "column":  # liquid column with three bubbles under buoyancy
        p.update(st_mask_liquid=1, gy=-1e-4, beta_T=1.0, Ste=rng.uniform(0.08, 0.2))
        l = nx / 4.0
        y = torch.arange(ny, dtype=torch.float64, device=_device())[:, None]
        phi = (0.5 + 0.5 * torch.tanh(2.0 * (1.8 * l - 0.5 - y) / p["W"])).expand(ny, nx)
        for cx, cy, r in ((1.0, 0.3, 0.2), (2.0, 1.0, 0.24), (3.0, 0.4, 0.3)):
            phi = phi * _disk(p, l * (cx + rng.uniform(-0.05, 0.05)), l * cy, l * r, inside=False)
    elif problem in ("sessile", "sweep"):
        p.update(rho_ratio_lg=1000.0, mu_ratio_lg=100.0, theta_deg=rng.uniform(30.0, 150.0),
                 rho_ratio_sl=rng.uniform(0.88, 0.95), Ste=rng.uniform(0.05, 0.2))
        phi = _drop(p, rng, rng.uniform(0.15, 0.3) * n, 0, 0, 0)
    elif problem == "closed":  # walls everywhere, two of them cold
        p.update(periodic_x=0, dirichlet_x_hi=1, theta_deg=rng.uniform(45.0, 135.0),
                 Cp_ratio_sl=0.5, k_ratio_sl=3.8, k_ratio_gl=0.04)
        phi = _drop(p, rng, rng.uniform(0.2, 0.3) * n, 0, 0, 0)
    else:  # "bubbles", "batch"
        p.update(st_mask_liquid=1, theta_deg=rng.uniform(60.0, 120.0))
        if problem == "batch":
            phi = _drop(p, rng, rng.uniform(0.15, 0.3) * n, int(rng.integers(0, 5)), 3.0, 10.0)
        else:
            phi = _drop(p, rng, rng.uniform(0.28, 0.32) * n, 8, 4.0, 12.0)
    return p, phi, torch.full((ny, nx), T, dtype=torch.float64, device=_device())


def _problems(case, seed):
    rng = np.random.default_rng([int(seed), 20240324])
    if "lattices" not in case:
        return [_problem(case["problem"], case["nx"], case["ny"], rng)]
    # the grids of a batch belong to the case, the drops on them to the seed
    sizes = np.random.default_rng(1000 * case["lattices"] + case["lo"])
    out = []
    for _ in range(case["lattices"]):
        if case["problem"] == "sweep":
            nx = ny = int(sizes.choice([q for q in (128, 192, 256, 384, 512)
                                        if case["lo"] <= q <= case["hi"]]))
        else:
            nx, ny = (int(v) for v in sizes.integers(case["lo"], case["hi"] + 1, 2))
        out.append(_problem(case["problem"], nx, ny, rng))
    return out


def _sites(case):
    if "lattices" not in case:
        return case["nx"] * case["ny"]
    sizes = np.random.default_rng(1000 * case["lattices"] + case["lo"])
    total = 0
    for _ in range(case["lattices"]):
        if case["problem"] == "sweep":
            total += int(sizes.choice([q for q in (128, 192, 256, 384, 512)
                                       if case["lo"] <= q <= case["hi"]])) ** 2
        else:
            nx, ny = (int(v) for v in sizes.integers(case["lo"], case["hi"] + 1, 2))
            total += nx * ny
    return total


def work(case):
    n = _sites(case)
    if case["kind"] == "checkpoint":  # 32 doubles a site in, 32 out
        return {"bytes": 2 * 32 * 8 * n, "flops": 0}
    steps = case["steps"]
    return {"bytes": BYTES_LU[case["storage"]] * n * steps, "flops": FLOPS_LU * n * steps}


# ----------------------------------------------------------------------------
# The passes
# ----------------------------------------------------------------------------

# The state layout that include/lbm.h documents: row blocks of 32 sites, 768
# population values a block (chunk, place in it and its directions) and 320
# own-site floats.
CHUNK = {2: (0, 0, 3), 5: (0, 1, 3), 6: (0, 2, 3), 1: (288, 0, 2), 3: (288, 1, 2),
         4: (480, 0, 3), 7: (480, 1, 3), 8: (480, 2, 3)}


def _blocks(p):
    return p["ny"] * ((p["nx"] + 31) // 32)


def _state_views(lat, storage):
    """The state buffers of a handle as tensors: [lattice][buffer] = (pops,
    aux). They are the tail of the workspace that the caller owns, two buffers
    of populations and own-site values per lattice."""
    elem = 4 if storage == "fp32" else 2
    end = lat.workspace.numel()
    at = end - sum(2 * _blocks(p) * (768 * elem + 320 * 4) for p in lat.params)
    out = []
    for p in lat.params:
        pair = []
        for _ in range(2):
            n = _blocks(p) * 768 * elem
            m = _blocks(p) * 320 * 4
            pair.append((lat.workspace[at:at + n].view(POP_TYPE[storage]),
                         lat.workspace[at + n:at + n + m].view(torch.float32)))
            at += n + m
        out.append(pair)
    return out


def prepare(case, seed):
    probs = _problems(case, seed)
    if case["kind"] == "noalloc":
        p, phi, T = probs[0]
        dev = torch.device("cuda")
        pops, aux, _ = _start(p, phi, T)
        P, A = (v.float() for v in _blocked(p, pops, aux))
        return {"case": case, "params": p, "bufs": [(P, A), (torch.zeros_like(P), torch.zeros_like(A))],
                "d_obs": torch.zeros(lbm.LBM_OBS_COUNT, dtype=torch.float64, device=dev),
                "pitch": (p["nx"] + 31) // 32 * 32, "at": 0}
    if case["kind"] == "checkpoint":
        p, phi, T = probs[0]
        lat = lbm.Lattice([p])
        lat.init(phi.cpu().numpy(), T.cpu().numpy())
        pops, aux = _checkpoint(p, phi, T, seed)
        return {"case": case, "lat": lat, "pops": pops, "aux": aux}
    lat = lbm.Lattice([p for p, _, _ in probs], storage=STORAGE[case["storage"]])
    views = _state_views(lat, case["storage"])
    for pair in views:  # the columns that pad a row to whole blocks are never written
        for pops, aux in pair:
            pops.zero_()
            aux.zero_()
    for k, (_, phi, T) in enumerate(probs):
        lat.init(phi.cpu().numpy(), T.cpu().numpy(), inst=k)
    if case.get("exec"):
        lat.set_exec({"graph": lbm.LBM_EXEC_GRAPH, "persistent": lbm.LBM_EXEC_PERSISTENT}[case["exec"]],
                     case["chunk"])
    return {"case": case, "lat": lat, "views": views[:STATES], "at": 0}


def run(state):
    case = state["case"]
    if case["kind"] == "noalloc":
        stream = torch.cuda.current_stream().cuda_stream
        for _ in range(case["steps"]):
            (Pi, Ai), (Po, Ao) = state["bufs"][state["at"]], state["bufs"][state["at"] ^ 1]
            lbm.lbm_step_noalloc(state["params"], Pi.data_ptr(), Ai.data_ptr(), Po.data_ptr(),
                                 Ao.data_ptr(), state["pitch"], state["d_obs"].data_ptr(), stream)
            state["at"] ^= 1
        # the record is kept in the precision of the fields it sums
        return [*state["bufs"][state["at"]], state["d_obs"].float()]
    lat = state["lat"]
    if case["kind"] == "checkpoint":
        lat.set_state(state["pops"], state["aux"])
        return list(lat.get_state())
    lat.step(case["steps"])
    out = []
    if case.get("observe"):  # a time series in the precision of the fields it sums
        out.append(lat.observables_all(check=False).astype(np.float32))
    state["at"] ^= case["steps"] & 1
    for pair in state["views"]:
        out += pair[state["at"]]
    return out


# ----------------------------------------------------------------------------
# The same in 64 bits (Section 3 of the paper, with plain torch operations)
# ----------------------------------------------------------------------------

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _mix(fs, phi, zs, zl, zg):
    ph = phi.clamp(0.0, 1.0)
    return fs * zs + (1.0 - fs) * (ph * zl + (1.0 - ph) * zg)


def _closure(p, H, phihat, phi):
    """Liquid fraction, solid fraction, temperature and the ramp of H and phi."""
    L = p["Cp"] * (p["T_m"] - p["T_w"]) / p["Ste"]
    Hs = p["Cp"] * p["T_m"]
    fl = ((H - Hs) / L).clamp(0.0, 1.0)
    chi = ((phihat - 0.5) / p["pc_ramp"] + 0.5).clamp(0.0, 1.0)
    fs = chi * (1.0 - fl)
    cp = _mix(fs, phi, p["Cp"] * p["Cp_ratio_sl"], p["Cp"], p["Cp"] * p["Cp_ratio_gl"])
    return fl, fs, p["T_m"] + (H - Hs - L * fl) / cp, chi, cp


def _start(p, phi, T0):
    """Equilibrium at rest: (populations [27], carried fields [5], (phi, T))."""
    L = p["Cp"] * (p["T_m"] - p["T_w"]) / p["Ste"]
    cp0 = _mix(torch.zeros_like(phi), phi, 0.0, p["Cp"], p["Cp"] * p["Cp_ratio_gl"])
    H = p["Cp"] * p["T_m"] + L + cp0 * (T0 - p["T_m"])
    fl, _, T, _, _ = _closure(p, H, phi, phi)
    pops = torch.zeros((27,) + phi.shape, dtype=torch.float64, device=phi.device)
    for i in range(9):
        pops[i] = WT[i] * phi
        pops[9 + i] = WT[i] * p["Cp_ref"] * T
    pops[9] += H - p["Cp_ref"] * T
    aux = torch.zeros((5,) + phi.shape, dtype=torch.float64, device=phi.device)
    aux[0] = fl
    return pops, aux, (phi, T)


def _wall(p, i, like):
    """Sites whose link along c_i starts behind a wall, and those of them at a
    wall held at T_w."""
    wall = torch.zeros(like.shape, dtype=torch.bool, device=like.device)
    held = wall.clone()
    if not p["periodic_x"] and CX[i]:
        col = 0 if CX[i] > 0 else p["nx"] - 1
        wall[:, col] = True
        if p["dirichlet_x_lo" if CX[i] > 0 else "dirichlet_x_hi"]:
            held[:, col] = True
    if not p["periodic_y"] and CY[i]:
        row = 0 if CY[i] > 0 else p["ny"] - 1
        wall[row] = True
        if p["dirichlet_y_lo" if CY[i] > 0 else "dirichlet_y_hi"]:
            held[row] = True
    return wall, held


def _padded(p, Z, wet):
    """Z with one ghost layer: periodic wrap, or the wall rule (a copy of the
    adjacent value; wet: Eqs. 39-41)."""
    tan = math.tan(math.pi / 2 - math.radians(p["theta_deg"]))

    def ghost(a, b, periodic):  # a: the layer at the wall, b: the next one
        if not wet:
            return a

        def d(v):
            lo = torch.roll(v, 1) if periodic else torch.cat([v[:1], v[:-1]])
            hi = torch.roll(v, -1) if periodic else torch.cat([v[1:], v[-1:]])
            return 0.5 * (hi - lo)
        return a + tan * (1.5 * d(a) - 0.5 * d(b)).abs()

    px, py = p["periodic_x"], p["periodic_y"]
    lo = Z[-1] if py else ghost(Z[0], Z[1], px)
    hi = Z[0] if py else ghost(Z[-1], Z[-2], px)
    le = Z[:, -1] if px else ghost(Z[:, 0], Z[:, 1], py)
    ri = Z[:, 0] if px else ghost(Z[:, -1], Z[:, -2], py)
    out = torch.empty((p["ny"] + 2, p["nx"] + 2), dtype=Z.dtype, device=Z.device)
    out[1:-1, 1:-1] = Z
    out[0, 1:-1], out[-1, 1:-1], out[1:-1, 0], out[1:-1, -1] = lo, hi, le, ri
    for r, row in ((0, lo), (-1, hi)):
        for c, col in ((0, le), (-1, ri)):
            if px:      # the ghost row, wrapped
                out[r, c] = row[-1 if c == 0 else 0]
            elif py:    # the ghost column, wrapped
                out[r, c] = col[-1 if r == 0 else 0]
            else:       # the corner site
                out[r, c] = Z[r, c]
    return out


def _stencil(p, Z, wet=False, lap=False):
    q = _padded(p, Z, wet)
    ny, nx = Z.shape
    gx, gy, lp = torch.zeros_like(Z), torch.zeros_like(Z), torch.zeros_like(Z)
    for i in range(1, 9):
        z = q[1 + CY[i]:1 + CY[i] + ny, 1 + CX[i]:1 + CX[i] + nx]
        if CX[i]:
            gx += (3 * WT[i] * CX[i]) * z
        if CY[i]:
            gy += (3 * WT[i] * CY[i]) * z
        if lap:
            lp += (6 * WT[i]) * (z - Z)
    return (gx, gy, lp) if lap else (gx, gy)


def _steps(p, phi, T0, n):
    """n steps from the equilibrium start: (pops, aux, (phi, T), record)."""
    pops, aux, refs = _start(p, phi, T0)
    L = p["Cp"] * (p["T_m"] - p["T_w"]) / p["Ste"]
    tau_g = 3 * p["mobility"] + 0.5
    rho_l, rho_g, rho_s = p["rho_l"], p["rho_l"] / p["rho_ratio_lg"], p["rho_l"] * p["rho_ratio_sl"]
    mu_l = rho_l * (p["tau_f_liquid"] - 0.5) / 3
    mu_g, mu_s = mu_l / p["mu_ratio_lg"], mu_l * p["rho_ratio_sl"]
    kappa, beta = 1.5 * p["sigma"] * p["W"], 12 * p["sigma"] / p["W"]
    walls = [_wall(p, i, phi) for i in range(9)]
    rec = None
    for _ in range(n):
        pre = torch.empty_like(pops)
        for s in range(3):
            pre[9 * s] = pops[9 * s]
            for i in range(1, 9):
                v = torch.roll(pops[9 * s + i], (CY[i], CX[i]), (0, 1))
                wall, held = walls[i]
                back = pops[9 * s + OPP[i]]
                if s == 1:
                    back = torch.where(held, -back + 2 * WT[i] * p["Cp_ref"] * p["T_w"], back)
                pre[9 * s + i] = torch.where(wall, back, v)
        g, h, f = pre[:9], pre[9:18], pre[18:]
        phihat, H = g.sum(0), h.sum(0)
        fl, fs, _, chi, _ = _closure(p, H, phihat, phihat)
        mdot = (1 - rho_s / rho_l) * chi * (aux[0] - fl)
        ph = phihat / (1 - 0.5 * mdot)
        _, _, T, _, cp = _closure(p, H, phihat, ph)
        rho = _mix(fs, ph, rho_s, rho_l, rho_g)
        gpx, gpy, lph = _stencil(p, ph, wet=True, lap=True)
        grx, gry = _stencil(p, rho)
        gqx, gqy = _stencil(p, aux[3])
        gsx, gsy = _stencil(p, aux[4])
        mu_phi = 4 * beta * (ph - 1) * ph * (ph - 0.5) - kappa * lph
        if p["st_mask_liquid"]:
            mu_phi = mu_phi * (1 - fs)
        buoy = -p["rho_0"] * p["beta_T"] * (T - p["T_ref"])
        Fx, Fy = mu_phi * gpx + buoy * p["gx"], mu_phi * gpy + buoy * p["gy"]
        mx = sum(CX[i] * f[i] for i in range(9) if CX[i])
        my = sum(CY[i] * f[i] for i in range(9) if CY[i])
        usx, usy = (mx + 0.5 * Fx) / rho, (my + 0.5 * Fy) / rho
        ffx, ffy = -fs * usx, -fs * usy
        ux, uy = usx + 0.5 * ffx, usy + 0.5 * ffy
        uu = ux * ux + uy * uy
        S = rho * mdot + ux * grx + uy * gry
        Ftx, Fty = Fx - gqx + (grx + gsx) / 3, Fy - gqy + (gry + gsy) / 3
        uF = ux * Ftx + uy * Fty
        tau_f = 3 * _mix(fs, ph, mu_s, mu_l, mu_g) / rho + 0.5
        F0 = WT[0] * (S - 3 * uF)
        pn = (f[1:].sum(0) + 0.5 * S + (tau_f - 0.5) * F0 - rho * WT[0] * 1.5 * uu) / (3 * (1 - WT[0]))
        gm = torch.sqrt(gpx * gpx + gpy * gpy + p["normal_eps"] ** 2)
        lam = 4 * ph * (1 - ph) / p["W"]
        ax = ph * ux - aux[1] + lam * gpx / gm / 3
        ay = ph * uy - aux[2] + lam * gpy / gm / 3
        tau_h = _mix(fs, ph, p["k_ratio_sl"], 1.0, p["k_ratio_gl"]) * (p["tau_h"] - 0.5) + 0.5
        new = torch.empty_like(pops)
        for i in range(9):
            w, cu = WT[i], CX[i] * ux + CY[i] * uy
            si = w * (3 * cu + 4.5 * cu * cu - 1.5 * uu)
            Gi = 3 * w * (CX[i] * ax + CY[i] * ay) + w * ph * mdot
            new[i] = g[i] - (g[i] - w * ph * (1 + 3 * cu)) / tau_g + (1 - 0.5 / tau_g) * Gi
            heq = w * p["Cp_ref"] * T + cp * T * si
            if i == 0:
                heq = heq + H - p["Cp_ref"] * T
            new[9 + i] = h[i] - (h[i] - heq) / tau_h
            feq = 3 * pn * (w - (1.0 if i == 0 else 0.0)) + rho * si
            Fi = w * (S + 3 * (CX[i] * (Fx + rho * ffx) + CY[i] * (Fy + rho * ffy))
                      + 9 * cu * (CX[i] * Ftx + CY[i] * Fty) - 3 * uF)
            new[18 + i] = f[i] - (f[i] - feq) / tau_f + (1 - 0.5 / tau_f) * Fi
        pops, aux, refs = new, torch.stack([fl, ph * ux, ph * uy, pn, S]), (ph, T)
        bad = ~(torch.isfinite(ph) & torch.isfinite(H) & torch.isfinite(ux) & torch.isfinite(pn))
        rec = (ph, fs, H, rho, fs * rho_s + (1 - fs) * ph.clamp(0, 1) * rho_l, mdot, ph * mdot, uu, bad)
    ph, fs, H, rho, cond, mdot, pmd, uu, bad = rec
    record = torch.stack([ph.sum(), fs.sum(), H.sum(), rho.sum(), cond.sum(), mdot.sum(), pmd.sum(),
                          fs[:, p["nx"] // 2].sum(), fs[p["ny"] // 2].sum(), uu.max().sqrt(),
                          bad.sum().double()])
    return pops, aux, refs, record


def _blocked(p, pops, aux, refs=None):
    """Populations and carried fields in the library's blocked layout (FP64);
    refs: in the form that 16-bit storage keeps, deviations from the rest
    equilibria of the site each link ends at (g, h) or starts from (f)."""
    ny, nx, nb = p["ny"], p["nx"], (p["nx"] + 31) // 32
    L = p["Cp"] * (p["T_m"] - p["T_w"]) / p["Ste"]

    def wide(a):
        w = torch.zeros((ny, nb * 32), dtype=torch.float64, device=a.device)
        w[:, :nx] = a
        return w.view(ny, nb, 32)

    P = torch.zeros((ny, nb, 768), dtype=torch.float64, device=pops.device)
    A = torch.zeros((ny, nb, 320), dtype=torch.float64, device=pops.device)
    for i, (c, k, n) in CHUNK.items():
        g, h, f = pops[i], pops[9 + i], pops[18 + i]
        if refs is not None:
            wall, _ = _wall(p, OPP[i], g)  # the link along c_i ends behind a wall
            ph, T = (torch.where(wall, r, torch.roll(r, (-CY[i], -CX[i]), (0, 1))) for r in refs)
            g, h = g - WT[i] * ph, h - WT[i] * p["Cp_ref"] * T
            f = 4096 * (f - 3 * WT[i] * aux[3])
        at = c + 64 * k
        P[:, :, at:at + 64:2], P[:, :, at + 1:at + 64:2] = wide(g), wide(h)
        at = c + 64 * n + 32 * k
        P[:, :, at:at + 32] = wide(f)
    for c, v in enumerate((pops[0], pops[9] - L * aux[0], pops[18], aux[0])):
        A[:, :, c:128:4] = wide(v)
        A[:, :, 128 + c:256:4] = wide(aux[1 + c])
    if refs is not None:
        for c in range(2):
            A[:, :, 256 + c:320:2] = wide(refs[c])
    return P.reshape(-1), A.reshape(-1)


def _checkpoint(p, phi, T, seed):
    """Host arrays of a checkpoint: the equilibrium start with a little noise."""
    pops, aux, _ = _start(p, phi, T)
    rng = np.random.default_rng([int(seed), 7])
    pops, aux = pops.cpu().numpy(), aux.cpu().numpy()
    pops += 1e-3 * rng.standard_normal(pops.shape)
    aux[1:] += 1e-3 * rng.standard_normal(aux[1:].shape)
    return pops, aux


def exact(case, seed):
    probs = _problems(case, seed)
    if case["kind"] == "checkpoint":
        return list(_checkpoint(*probs[0], seed))
    out, records = [], []
    for k, (p, phi, T) in enumerate(probs):
        if k >= STATES:
            break
        pops, aux, refs, record = _steps(p, phi, T, case["steps"])
        records.append(record)
        out += _blocked(p, pops, aux, None if case["storage"] == "fp32" else refs)
    if case["kind"] == "noalloc":
        return [*out, records[0]]
    if not case.get("observe"):
        return out
    # the records of a batch are compared only where every lattice was followed
    return [torch.stack(records) if len(probs) <= STATES else None] + out
