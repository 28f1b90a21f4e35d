"""Workloads of the overlapping Schwarz FOM / OpInf hot path as a user's program calls them.

Each case is one call (or the two or three calls that belong together) of the public entry points:
the element-level force and its gradient, one controller step of a coupled problem (explicit and
implicit FOMs, quadratic ROMs, every precision), a batch of instances, the adjoint of an explicit
rollout, and the offline operator fit.  Sizes are those of `workloads.py`, the tests and `bench.py`.

A controller step advances its state, so `run` puts the start state back first (device to device) and
reads the new state at the end, as a program does that exchanges the state with its own code every
controller step.  The Schwarz iterations are capped (the coupling goes on after its cap, as in the
paper's capped runs), so that the work of a pass is fixed.  ROM bases are smooth orthonormalised
modes, ROM operators seeded stand-ins of the trained sizes.
"""
import math

import numpy as np
import torch

from paper_2511_20687_gb300 import autograd, osam
from paper_2511_20687_gb300 import workloads as W

DEV = "cuda:0"
F64 = torch.float64
PRECISION = {"fp64": osam.FP64, "fp32_force": osam.FP32_FORCE, "f32x2_force": osam.F32X2_FORCE,
             "fp64_tangent32": osam.FP64_TANGENT32}


def listed():
    return [
        # one internal force of the smallest mesh: launches and latency
        {"name": "force_le_6x6x12", "kind": "force", "material": "le", "nx": 6, "ny": 6, "nz": 12,
         "per_element": False, "grad": False},
        # force and gradient through autograd on the adjoint bar's mesh, per-element Lame parameters
        {"name": "force_grad_nh_20x20x40", "kind": "force", "material": "nh", "nx": 20, "ny": 20, "nz": 40,
         "per_element": True, "grad": True},
        # the plain FOM-FOM coupling: the smallest controller step
        {"name": "step_fom_fom_le_6x6x12", "kind": "step", "layout": "ff", "material": "le", "n": 6, "nz": 12,
         "r": 0, "precision": "fp64", "implicit": False, "substeps": 20, "iters": 5, "dt": 1e-6},
        # the headline hybrid: FOM 40x40x80 with an r = 64 ROM
        {"name": "step_hybrid_nh_40x40x80", "kind": "step", "layout": "fr", "material": "nh", "n": 40, "nz": 80,
         "r": 64, "precision": "fp64", "implicit": False, "substeps": 20, "iters": 4, "dt": 1e-6},
        # the same with the double-float force (training runs)
        {"name": "step_hybrid_f32x2_40x40x80", "kind": "step", "layout": "fr", "material": "nh", "n": 40, "nz": 80,
         "r": 64, "precision": "f32x2_force", "implicit": False, "substeps": 20, "iters": 4, "dt": 1e-6},
        # the large chain FOM - OpInf r = 128 - FOM
        {"name": "step_chain_nh_96x96x192", "kind": "step", "layout": "frf", "material": "nh", "n": 96, "nz": 192,
         "r": 128, "precision": "fp64", "implicit": False, "substeps": 20, "iters": 2, "dt": 5e-7},
        # a chain of odd sizes with the FP32 force
        {"name": "step_chain_fp32_75x75x149", "kind": "step", "layout": "frf", "material": "nh", "n": 75, "nz": 149,
         "r": 48, "precision": "fp32_force", "implicit": False, "substeps": 20, "iters": 3, "dt": 5e-7},
        # a parameter sweep: FOM / OpInf pairs of uneven meshes in one context
        {"name": "batch_nh_64_samples", "kind": "batch", "samples": 64, "n_min": 8, "n_max": 32, "r": 32,
         "substeps": 20, "iters": 4},
        # implicit Newmark FOMs (Newton-CG) with the FP64 and the FP32 tangent
        {"name": "step_implicit_nh_20x20x40", "kind": "step", "layout": "ff", "material": "nh", "n": 20, "nz": 40,
         "r": 0, "precision": "fp64", "implicit": True, "substeps": 4, "iters": 2, "dt": 1e-5},
        {"name": "step_implicit_t32_40x40x80", "kind": "step", "layout": "fr", "material": "nh", "n": 40, "nz": 80,
         "r": 64, "precision": "fp64_tangent32", "implicit": True, "substeps": 4, "iters": 2, "dt": 5e-6},
        # gradient of a tip displacement through an explicit rollout, checkpoints every 50 steps
        {"name": "adjoint_nh_20x20x40", "kind": "adjoint", "material": "nh", "nx": 20, "ny": 20, "nz": 40,
         "steps": 200, "every": 50},
        # the headline ROM's fit: 500 snapshots of the 40x40x80 mesh's free dofs
        {"name": "fit_quadratic_403440x500", "kind": "fit", "n_dof": 403440, "n_sdof": 5043, "snaps": 500, "r": 64,
         "r_s": 41, "model": "quadratic"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["force", "force", "step", "step", "step", "batch", "adjoint", "fit"])
    if kind == "force":
        n = [_log_int(rng, 3, 110) for _ in range(3)]
        mat = rng.choice(["le", "nh", "nh", "svk"])
        return {"kind": kind, "material": mat, "nx": n[0], "ny": n[1], "nz": n[2], "per_element": rng.random() < 0.5,
                "grad": mat != "svk" and rng.random() < 0.5}
    if kind == "step":
        layout = rng.choice(["ff", "fr", "frf"])
        implicit = layout != "frf" and rng.random() < 0.3
        n = _log_int(rng, 6, 36 if implicit else 80)
        nz = int(n * rng.uniform(1.5, 2.2))
        prec = rng.choice(["fp64", "fp64_tangent32"] if implicit else ["fp64", "fp64", "fp32_force", "f32x2_force"])
        return {"kind": kind, "layout": layout, "material": rng.choice(["nh", "nh", "nh", "le", "svk"]), "n": n,
                "nz": nz, "r": 0 if layout == "ff" else _log_int(rng, 8, 128), "precision": prec,
                "implicit": implicit, "substeps": rng.randint(2, 4) if implicit else rng.randint(10, 24),
                "iters": 2 if implicit else rng.randint(2, 4), "dt": 5e-6 if implicit else 1e-6}
    if kind == "batch":
        lo = rng.randint(6, 12)
        return {"kind": kind, "samples": _log_int(rng, 2, 60), "n_min": lo, "n_max": lo + rng.randint(2, 16),
                "r": _log_int(rng, 6, 40), "substeps": rng.randint(10, 20), "iters": rng.randint(2, 4)}
    if kind == "adjoint":
        return {"kind": kind, "material": rng.choice(["nh", "nh", "le"]), "nx": _log_int(rng, 4, 20),
                "ny": _log_int(rng, 4, 20), "nz": _log_int(rng, 8, 40), "steps": rng.randint(40, 160),
                "every": rng.choice([20, 50, 64])}
    model = rng.choice(["linear", "quadratic", "quadratic", "cubic"])
    return {"kind": "fit", "n_dof": _log_int(rng, 4000, 400000), "n_sdof": _log_int(rng, 200, 5000),
            "snaps": rng.randint(120, 480), "r": rng.randint(4, 14) if model == "cubic" else rng.randint(6, 60),
            "r_s": rng.randint(4, 36), "model": model}


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _orthonormal(A):
    """Cholesky-QR, twice (the columns are well conditioned)."""
    for _ in range(2):
        L = torch.linalg.cholesky(A.T @ A)
        A = A @ torch.linalg.solve_triangular(L, torch.eye(len(L), device=DEV, dtype=F64), upper=False).T
    return A.contiguous()


def _modes(xyz, comp, r, seed):
    """r smooth orthonormal fields on the dofs at xyz [m, 3] (unit box) of components comp [m]: axial modes
    of u_z (most of them) and transverse ones, with a small seeded roughness."""
    g = _gen(seed, 11)
    x, y, z = xyz.T
    A = 1e-3 * torch.randn(len(comp), r, generator=g, device=DEV, dtype=F64)
    for k in range(r):
        c = (2, 2, 0, 2, 1)[k % 5]
        m = (k + 5) // 5 + (2 * k) % 5
        w = torch.cos(math.pi * (k % 3) * x) * torch.cos(math.pi * ((k // 3) % 2) * y)
        A[:, k] += (comp == c) * torch.sin(math.pi * (m + 0.5) * z + 0.3 * k) * w
    return _orthonormal(A)


def _rom_operators(spec, i, r, seed):
    sd = spec.subdomains[i]
    free, schwarz = W.subdomain_dof_masks(spec, i)
    ext = np.array(sd.dims, float) * sd.h
    xyz = torch.from_numpy(((sd.node_coords() - np.array(sd.origin)) / ext).repeat(3, axis=0)).to(DEV)
    comp = torch.arange(3 * sd.n_nodes, device=DEV) % 3
    free, schwarz = torch.from_numpy(free).to(DEV), torch.from_numpy(schwarz).to(DEV)
    r = min(r, int(free.sum()) // 4)
    rs = max(1, min(r // 2 + 1, int(schwarz.sum()) // 2))
    rng = np.random.default_rng(seed + 17)
    omega = np.sort(rng.uniform(1e4, 1e5, r))
    return {"Phi": _modes(xyz[free], comp[free], r, seed), "Phi_S": _modes(xyz[schwarz], comp[schwarz], rs, seed + 1),
            "K": -np.diag(omega ** 2), "H": 1e6 * rng.standard_normal((r, r * (r + 1) // 2)) / r,
            "B": 1e8 * rng.standard_normal((r, rs)) / rs, "c": np.zeros(r)}


def _step_problem(case, seed):
    """(spec, rom_ops) of a coupled bar; Young's modulus, Poisson's ratio and the pulse from the seed."""
    rng = np.random.default_rng(seed)
    E, nu, amp = rng.uniform(0.5e9, 1.2e9), rng.uniform(0.2, 0.33), rng.uniform(0.5e-3, 1e-3)
    kinds = [{"f": "fom", "r": "rom"}[c] for c in case["layout"]]
    spec = W.bar_chain("case", case["n"], [case["nz"]] * len(kinds), kinds, case["material"], E, nu, 1000.0, amp,
                       case["dt"], case["substeps"], max_iters=case["iters"])
    ops = {}
    for i, sd in enumerate(spec.subdomains):
        if sd.kind == "rom":
            ops[i] = _rom_operators(spec, i, case["r"], seed + 31 * i)
        elif case["implicit"]:
            sd.integrator = "implicit"
    return spec, ops


def _batch_problems(case, seed):
    specs = W.batched_samples(case["samples"], n_min=case["n_min"], n_max=case["n_max"])
    rng = np.random.default_rng(seed)
    for s in specs:
        s.n_substeps, s.max_iters = case["substeps"], case["iters"]
        scale = rng.uniform(0.5, 1.0)
        for sd in s.subdomains:
            sd.u0 *= scale
    return specs, [{1: _rom_operators(s, 1, case["r"], seed + k)} for k, s in enumerate(specs)]


def _force_inputs(case, seed):
    nx, ny, nz = dims = case["nx"], case["ny"], case["nz"]
    g = _gen(seed, 1)
    h = W.H_DEFAULT
    z = torch.arange(nz + 1, device=DEV, dtype=F64) / nz
    u = 1e-4 * torch.randn(nz + 1, ny + 1, nx + 1, 3, generator=g, device=DEV, dtype=F64)
    u[..., 2] += 1e-3 * torch.exp(-((z - 0.5) ** 2) / 0.02)[:, None, None]
    u = u.reshape(-1, 3).contiguous()
    lam, mu = W.lame(1e9 * (1.0 + (seed % 7) / 10), 0.25)
    ne = nx * ny * nz
    lam_e = lam * (1.0 + 0.1 * (2.0 * torch.rand(ne, generator=g, device=DEV, dtype=F64) - 1.0))
    mu_e = mu * (1.0 + 0.1 * (2.0 * torch.rand(ne, generator=g, device=DEV, dtype=F64) - 1.0))
    ybar = torch.randn(u.shape, generator=g, device=DEV, dtype=F64)
    return dims, h, u, lam, mu, lam_e, mu_e, ybar


def _adjoint_inputs(case, seed):
    nz = case["nz"]
    rng = np.random.default_rng(seed)
    lam, mu = W.lame(1e9, 0.25)
    p = W.single_bar("case", 1, nz, case["material"], 1e9, 0.25, 1000.0, rng.uniform(0.5e-3, 1e-3), 1e-6, 1)
    sd = p.subdomains[0]
    sd.dims = dims = (case["nx"], case["ny"], nz)
    ne = sd.n_elements
    _, _, kk = sd.node_grid()
    u0 = W.gaussian_z(sd.node_coords(), p.info["amplitude"], p.info["z_c"], p.info["s"])
    w = np.zeros_like(u0)
    w[kk == nz, 2] = 1.0 / np.sum(kk == nz)
    dirichlet = np.where(kk == 0, 7, 0).astype(np.uint8)
    return {"dims": dims, "h": sd.h, "lam_e": lam * (1 + 0.1 * rng.uniform(-1, 1, ne)),
            "mu_e": mu * (1 + 0.1 * rng.uniform(-1, 1, ne)), "dirichlet": dirichlet, "u0": u0, "w": w}


def _snapshots(rows, cols, decay, seed, salt, weights):
    """Snapshot matrices [rows, cols] sharing their modes, one per entry of weights: localised fields with
    geometrically decaying amplitudes above a noise floor of 1e-3."""
    g = _gen(seed, salt)
    z = torch.linspace(0.0, 1.0, cols, device=DEV, dtype=F64)
    modes = torch.randn(rows, cols, generator=g, device=DEV, dtype=F64)
    modes *= torch.exp(-((z - 0.5) ** 2) / 0.02) / math.sqrt(0.125 * cols)
    V = torch.linalg.qr(torch.randn(rows, rows, generator=g, device=DEV, dtype=F64))[0]
    k = torch.arange(rows, device=DEV, dtype=F64)
    amp = torch.clamp(decay ** k, min=1e-3)
    return [((V * (amp * f(k))) @ modes).contiguous() for f in weights]


def _fit_inputs(case, seed):
    U, A = _snapshots(case["snaps"], case["n_dof"], 0.93, seed, 5,
                      [lambda k: torch.ones_like(k), lambda k: -(1.0 + 0.1 * k)])
    S, = _snapshots(case["snaps"], case["n_sdof"], 0.85, seed, 6, [lambda k: torch.ones_like(k)])
    return U, A, S


# ------------------------------------------------------------------------------------------------
# the calls
# ------------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "force":
        dims, h, u, lam, mu, lam_e, mu_e, ybar = _force_inputs(case, seed)
        if case["grad"]:
            for t in (u, lam_e, mu_e):
                t.requires_grad_(True)
        if not case["per_element"] and case["grad"]:
            with torch.no_grad():
                lam_e.fill_(lam)
                mu_e.fill_(mu)
        return {"case": case, "dims": dims, "h": h, "u": u, "lam": lam, "mu": mu, "lam_e": lam_e, "mu_e": mu_e,
                "ybar": ybar, "f": torch.empty_like(ybar)}
    if kind in ("step", "batch"):
        if kind == "step":
            spec, ops = _step_problem(case, seed)
            specs, p = [spec], osam.Problem(spec, ops, precision=PRECISION[case["precision"]])
        else:
            specs, ops = _batch_problems(case, seed)
            p = osam.Batch(specs, ops)
        # the nodal fields of all FOMs of a subdomain index in one buffer each, one slice per instance
        start, fields = [], []
        for i in range(len(specs[0].subdomains)):
            at = np.cumsum([0] + [s.subdomains[i].n_nodes for s in specs])
            fom = specs[0].subdomains[i].kind == "fom"
            if fom:
                first, out = (torch.empty(3, at[-1], 3, device=DEV, dtype=F64) for _ in range(2))
                fields.append(out)
            for n in range(len(specs)):
                if fom:
                    cut = [f[:, at[n]:at[n + 1]] for f in (first, out)]
                    p.state(i, out=cut[0], inst=n)
                    start.append((n, i, cut[0], cut[1]))
                else:
                    start.append((n, i, p.reduced_state(i, n), None))
        return {"case": case, "problem": p, "start": start, "fields": fields}
    if kind == "adjoint":
        return {"case": case, "inputs": _adjoint_inputs(case, seed)}
    return {"case": case, "snapshots": _fit_inputs(case, seed)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "force":
        if case["grad"]:
            u, lam_e, mu_e = state["u"], state["lam_e"], state["mu_e"]
            f = autograd.hex8_force(u, lam_e, mu_e, state["dims"], state["h"], case["material"])
            return (f.detach(),) + torch.autograd.grad(f, (u, lam_e, mu_e), state["ybar"])
        per = case["per_element"]
        osam.hex8_force(state["dims"], state["h"], case["material"], state["lam"], state["mu"], state["u"], state["f"],
                        lam_e=state["lam_e"] if per else None, mu_e=state["mu_e"] if per else None,
                        stream=torch.cuda.current_stream())
        return state["f"]
    if kind in ("step", "batch"):
        p = state["problem"]
        for n, i, first, out in state["start"]:
            if out is None:
                p.set_reduced_state(i, *first, inst=n)
            else:
                p.set_state(i, *first, inst=n)
        p.step()
        reduced = []
        for n, i, first, out in state["start"]:
            if out is None:
                reduced.append(p.reduced_state(i, n))
            else:
                p.state(i, out=out, inst=n)
        return [list(f) for f in state["fields"]] + [[np.concatenate(q) for q in zip(*reduced)]]
    if kind == "adjoint":
        q = state["inputs"]
        r = osam.adjoint(q["dims"], q["h"], case["material"], q["lam_e"], q["mu_e"], 1000.0, q["dirichlet"], q["u0"],
                         None, 1e-6, case["steps"], q["w"], checkpoint_every=case["every"])
        return [r[k] for k in ("J", "grad_u0", "grad_v0", "grad_lambda", "grad_mu")]
    U, A, S = state["snapshots"]
    # lambda from the upper half of the usual candidates, where the operators are well determined
    return _with_signs(osam.opinf_fit(U, A, S, case["r"], 1e-2, r_s=case["r_s"], r_s_max=case["r_s"],
                                      quadratic=case["model"] != "linear", cubic=case["model"] == "cubic"))


def _with_signs(o):
    """The fitted model with every mode's entry of largest magnitude made positive (a POD basis is unique up
    to the signs of its modes), as a program that compares two fits has it."""
    def signs(P):
        return np.sign(P[np.abs(P).argmax(axis=0), np.arange(P.shape[1])])

    s, ss = signs(o["Phi"]), signs(o["Phi_S"])
    r = len(s)
    i, j = np.triu_indices(r)
    out = {"Phi": o["Phi"] * s, "Phi_S": o["Phi_S"] * ss, "K": o["K"] * s[:, None] * s, "H": o["H"] * s[:, None] * (s[i] * s[j]),
           "B": o["B"] * s[:, None] * ss, "c": o["c"] * s, "sigma": o["sigma"], "sigma_s": o["sigma_s"]}
    if o.get("C") is not None:
        t = np.array([s[a] * s[b] * s[c] for a in range(r) for b in range(a, r) for c in range(b, r)])
        out["C"] = o["C"] * s[:, None] * t
    return out


# ------------------------------------------------------------------------------------------------
# work
# ------------------------------------------------------------------------------------------------
# FP64 operations of one element's internal force (interpolation, constitutive law, transposed
# interpolation; FMA = 2), of its vector-Jacobian product and of one tangent action, and of one node's update
FORCE_FLOPS = {"le": 632, "nh": 1232, "svk": 1500}
VJP_FLOPS = {"le": 1264, "nh": 3000}
TANGENT_FLOPS, NODE_FLOPS = 1832, 45


def _sizes(case):
    n, nz = case["n"], case["nz"]
    return n * n * nz, (n + 1) ** 2 * (nz + 1)


def work(case):
    kind = case["kind"]
    if kind in ("force", "adjoint"):
        ne = case["nx"] * case["ny"] * case["nz"]
        nn = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        f = FORCE_FLOPS[case["material"]]
    if kind == "force":
        el = 16 * ne if case["per_element"] or case["grad"] else 0
        if not case["grad"]:
            return {"bytes": 48 * nn + el, "flops": f * ne}
        return {"bytes": 48 * nn + el + 72 * nn + 2 * el, "flops": (f + VJP_FLOPS[case["material"]]) * ne}
    if kind == "adjoint":
        # a forward sweep, its recomputation from the checkpoints and the reverse sweep
        flops = case["steps"] * (ne * (2 * f + VJP_FLOPS[case["material"]]) + 3 * NODE_FLOPS * nn)
        return {"bytes": 2 * 72 * nn + 32 * ne + 48 * nn, "flops": flops}
    if kind == "step":
        ne, nn = _sizes(case)
        foms, sweeps = case["layout"].count("f"), case["substeps"] * case["iters"]
        flops = foms * sweeps * (ne * FORCE_FLOPS[case["material"]] + nn * NODE_FLOPS)
        if case["implicit"]:   # at least two Newton solves of a few CG iterations each
            flops += foms * sweeps * 10 * ne * TANGENT_FLOPS
        # the start state in, the end state out; the state is read and written once per substep
        return {"bytes": foms * nn * (144 + 144 * sweeps) + 8 * case["r"] ** 2 * (case["r"] + 3) // 2, "flops": flops}
    if kind == "batch":
        n = 0.5 * (case["n_min"] + case["n_max"])
        ne = 2 * n ** 3 * case["samples"]
        sweeps = case["substeps"] * case["iters"]
        return {"bytes": 1.2 * ne * (144 + 144 * sweeps), "flops": ne * sweeps * (FORCE_FLOPS["nh"] + NODE_FLOPS)}
    n, s, r = case["n_dof"], case["snaps"], case["r"]
    d = {"linear": r, "quadratic": r + r * (r + 1) // 2, "cubic": r + r * (r + 1) // 2 + r * (r + 1) * (r + 2) // 6}
    d = d[case["model"]] + case["r_s"] + 1
    flops = n * s * (s + 1) + 6 * n * s * r + 4 * n * r * r + case["n_sdof"] * s * (s + 4 * case["r_s"])
    flops += (s * (s + 1) * d + s ** 3 / 3 if d > s else d * (d + 1) * s + d ** 3 / 3) + 4 * s * d * r + 9 * s ** 3
    return {"bytes": 8 * (2 * n * s + case["n_sdof"] * s + n * r), "flops": flops}


# ------------------------------------------------------------------------------------------------
# the same results in plain torch, 64 bits
# ------------------------------------------------------------------------------------------------
class _Mesh:
    """Internal force of a structured hex8 mesh by 2x2x2 Gauss quadrature, element by element."""

    def __init__(self, dims, h, material, lam, mu):
        nx, ny, nz = dims
        i, j, k = torch.meshgrid(*(torch.arange(n, device=DEV) for n in (nz, ny, nx)), indexing="ij")
        n0 = (k + (nx + 1) * (j + (ny + 1) * i)).reshape(-1)
        corner = [(a, b, c) for c in (0, 1) for b in (0, 1) for a in (0, 1)]
        off = torch.tensor([a + (nx + 1) * (b + (ny + 1) * c) for a, b, c in corner], device=DEV)
        self.conn = n0[:, None] + off
        self.nn = (nx + 1) * (ny + 1) * (nz + 1)
        self.material, self.h, self.lam, self.mu = material, h, lam, mu
        q = [(1 - 1 / math.sqrt(3)) / 2, (1 + 1 / math.sqrt(3)) / 2]
        B = torch.zeros(8, 8, 3, dtype=F64)
        for g, p in enumerate((a, b, c) for c in q for b in q for a in q):
            for n, s in enumerate(corner):
                l = [p[d] if s[d] else 1 - p[d] for d in range(3)]
                dl = [1 if s[d] else -1 for d in range(3)]
                B[g, n] = torch.tensor([dl[0] * l[1] * l[2], l[0] * dl[1] * l[2], l[0] * l[1] * dl[2]], dtype=F64)
        self.B = (B / h).to(DEV)
        self.w = h ** 3 / 8

    def stress(self, H, lam, mu):
        eye = torch.eye(3, device=DEV, dtype=F64)
        tr = lambda A: A.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None]  # noqa: E731
        if self.material == "le":
            return lam * tr(H) * eye + mu * (H + H.mT)
        Fg = H + eye
        if self.material == "svk":
            E = 0.5 * (H + H.mT + H.mT @ H)
            return Fg @ (lam * tr(E) * eye + 2 * mu * E)
        r = [Fg[..., k, :] for k in range(3)]
        cof = torch.stack([torch.linalg.cross(r[1], r[2]), torch.linalg.cross(r[2], r[0]),
                           torch.linalg.cross(r[0], r[1])], -2)
        J = (r[0] * cof[..., 0, :]).sum(-1)[..., None, None]
        kappa = lam + 2 / 3 * mu
        jm = J.pow(-2 / 3)
        return mu * jm * Fg + (0.5 * kappa * (J * J - 1) - mu / 3 * jm * (Fg * Fg).sum((-2, -1), keepdim=True)) / J * cof

    def force(self, u, lam=None, mu=None, at=None):
        """f(u); lam, mu: per-element values in place of the mesh's."""
        lam = self.lam if lam is None else lam[:, None, None, None]
        mu = self.mu if mu is None else mu[:, None, None, None]
        f = torch.zeros(self.nn, 3, device=DEV, dtype=F64)
        for e in range(0, len(self.conn), 1 << 18):
            s = slice(e, e + (1 << 18))
            conn = self.conn[s]
            H = torch.einsum("eac,gak->egck", u[conn], self.B)
            cut = lambda v: v[s] if torch.is_tensor(v) else v  # noqa: E731
            P = self.stress(H, cut(lam), cut(mu))
            f = f.index_add(0, conn.reshape(-1), self.w * torch.einsum("egck,gak->eac", P, self.B).reshape(-1, 3))
        return f


class _Fom:
    def __init__(self, spec, i):
        sd = spec.subdomains[i]
        self.mesh = _Mesh(sd.dims, sd.h, sd.material, sd.lam, sd.mu)
        self.plane, self.layers = (sd.dims[0] + 1) * (sd.dims[1] + 1), sd.dims[2]
        m = torch.zeros(self.mesh.nn, device=DEV, dtype=F64)
        self.mass = m.index_add(0, self.mesh.conn.reshape(-1), torch.full((self.mesh.conn.numel(),), sd.rho * sd.h ** 3 / 8,
                                                                          device=DEV, dtype=F64))[:, None]
        clamped = torch.from_numpy(sd.dirichlet).to(DEV) != 0
        self.live = (~clamped).to(F64)[:, None]
        self.implicit = sd.integrator == "implicit"
        self.u = torch.from_numpy(sd.u0).to(DEV) * self.live
        self.v = torch.zeros_like(self.u)
        self.faces = {}
        fixed = clamped.clone()
        for c in spec.couplings:
            if c.dst == i:
                self.faces[c.src] = torch.from_numpy(c.nodes.astype(bool)).to(DEV)
                fixed |= self.faces[c.src]
        self.free = (~fixed).to(F64)[:, None]
        self.a = -self.mesh.force(self.u) / self.mass * self.live

    def save(self):
        self.saved = self.u, self.v, self.a

    def restore(self):
        self.u, self.v, self.a = self.saved

    def substep(self, dt, data):
        """data: {src: (u, v, a) on the face fed by src} at the new level."""
        imp = self.implicit
        up = self.u + dt * self.v + (0.25 if imp else 0.5) * dt * dt * self.a
        up = up * self.live
        for src, d in data.items():
            up[self.faces[src]] = d[0]
        if imp:
            un = self.newton(up, 4 / (dt * dt))
            an = 4 / (dt * dt) * (un - up)
        else:
            un = up
            an = -self.mesh.force(un) / self.mass
        self.v = (self.v + 0.5 * dt * (self.a + an)) * self.free
        self.u, self.a = un, an * self.free
        for src, d in data.items():
            self.v[self.faces[src]], self.a[self.faces[src]] = d[1], d[2]

    def newton(self, up, c0):
        u = up.clone()
        first = None
        for _ in range(25):
            R = (c0 * self.mass * (u - up) + self.mesh.force(u)) * self.free
            first = R.norm() if first is None else first
            if R.norm() <= 1e-14 * first or _ > 8:
                break
            x, r = torch.zeros_like(u), -R
            M = c0 * self.mass
            z = r / M
            p, rz = z, (r * z).sum()
            end = 1e-26 * rz
            for _k in range(1000):
                Ap = (M * p + torch.func.jvp(self.mesh.force, (u,), (p,))[1]) * self.free
                al = rz / (p * Ap).sum()
                x, r = x + al * p, r - al * Ap
                z = r / M
                rz, old = (r * z).sum(), rz
                if rz <= end:
                    break
                p = z + rz / old * p
            u = u + x
            if x.norm() <= 1e-16 * u.norm():
                break
        return u

    def at_layer(self, k):
        s = slice(k * self.plane, (k + 1) * self.plane)
        return self.u[s], self.v[s], self.a[s]

    def result(self):
        return torch.stack([self.u, self.v, self.a])


class _Rom:
    def __init__(self, spec, i, ops):
        sd = spec.subdomains[i]
        free, schwarz = (torch.from_numpy(m).to(DEV) for m in W.subdomain_dof_masks(spec, i))
        self.plane, self.layers, self.n = (sd.dims[0] + 1) * (sd.dims[1] + 1), sd.dims[2], sd.n_nodes
        self.Phi, self.Phi_S, self.K, self.H, self.Bm = (torch.as_tensor(ops[k], device=DEV) for k in
                                                         ("Phi", "Phi_S", "K", "H", "B"))
        self.iu = torch.triu_indices(*self.K.shape, device=DEV)
        self.free, self.schwarz = free, schwarz
        u0 = torch.from_numpy(sd.u0).to(DEV).reshape(-1)
        self.q = self.Phi.T @ u0[free]
        self.qd = torch.zeros_like(self.q)
        self.faces = {c.src: torch.from_numpy(c.nodes.astype(bool)).to(DEV).repeat_interleave(3) for c in spec.couplings
                      if c.dst == i}
        self.qdd = None

    def rhs(self, data):
        s = torch.zeros(3 * self.n, device=DEV, dtype=F64)
        for src, d in data.items():
            s[self.faces[src]] = d[0].reshape(-1)
        return self.K @ self.q + self.H @ (self.q[self.iu[0]] * self.q[self.iu[1]]) + self.Bm @ (self.Phi_S.T @ s[self.schwarz])

    def save(self):
        self.saved = self.q, self.qd, self.qdd

    def restore(self):
        self.q, self.qd, self.qdd = self.saved

    def substep(self, dt, data):
        self.q = self.q + dt * self.qd + 0.5 * dt * dt * self.qdd
        new = self.rhs(data)
        self.qd = self.qd + 0.5 * dt * (self.qdd + new)
        self.qdd = new

    def at_layer(self, k):
        full = torch.zeros(3 * self.n, 3, device=DEV, dtype=F64)
        lo, hi = 3 * k * self.plane, 3 * (k + 1) * self.plane
        at = torch.nonzero(self.free[:lo]).numel(), torch.nonzero(self.free[:hi]).numel()
        rows = torch.nonzero(self.free[lo:hi]).reshape(-1) + lo
        zero = torch.zeros_like(self.q) if self.qdd is None else self.qdd
        full[rows] = self.Phi[at[0]:at[1]] @ torch.stack([self.q, self.qd, zero], 1)
        return tuple(full[lo:hi, f].reshape(-1, 3) for f in range(3))

    def result(self):
        return [self.q, self.qd, self.qdd]


def _exact_step(spec, ops):
    """One controller step of the bar chain (conforming 2-layer overlaps: a face takes its neighbour's
    node layer two above or below), multiplicative sweeps at the iteration cap."""
    subs = [_Fom(spec, i) if sd.kind == "fom" else _Rom(spec, i, ops[i]) for i, sd in enumerate(spec.subdomains)]
    layer = lambda src, dst: subs[src].layers - 2 if src < dst else 2  # noqa: E731
    hold = {(c.src, c.dst): subs[c.src].at_layer(layer(c.src, c.dst)) for c in spec.couplings}
    for i, s in enumerate(subs):
        if isinstance(s, _Rom):
            s.qdd = s.rhs({src: hold[src, i] for src in s.faces})
    n = spec.n_substeps
    hist = {(c.src, c.dst): [subs[c.src].at_layer(layer(c.src, c.dst))] * (n + 1) for c in spec.couplings}
    for s in subs:
        s.save()
    for it in range(spec.max_iters):
        for i, s in enumerate(subs):
            if it:
                s.restore()
            told = {k: [None] for k in hist if k[0] == i}
            for j in range(1, n + 1):
                s.substep(spec.dt, {src: hist[src, i][j] for src in s.faces})
                for k in told:
                    told[k].append(s.at_layer(layer(*k)))
            hist.update(told)
    return [s.result() for s in subs]


def _as_run(results, spec):
    """The results of each instance in the layout of run(): (u, v, a) of every FOM index, then (q, q', q'')
    of every ROM."""
    kinds = [sd.kind for sd in spec.subdomains]
    out = [list(torch.cat([r[i] for r in results], 1)) for i, k in enumerate(kinds) if k == "fom"]
    rom = [r[i] for i, k in enumerate(kinds) if k == "rom" for r in results]
    return out + [[torch.cat(q) for q in zip(*rom)]]


def _exact_adjoint(case, q):
    mesh = _Mesh(q["dims"], q["h"], case["material"], None, None)
    leaf = lambda a: torch.from_numpy(a).to(DEV).requires_grad_(True)  # noqa: E731
    u0, lam, mu = leaf(q["u0"]), leaf(q["lam_e"]), leaf(q["mu_e"])
    v0 = torch.zeros_like(u0).requires_grad_(True)
    live = torch.from_numpy(q["dirichlet"] == 0).to(DEV, F64)[:, None]
    ones = torch.full((mesh.conn.numel(),), 1000.0 * q["h"] ** 3 / 8, device=DEV, dtype=F64)
    mass = torch.zeros(mesh.nn, device=DEV, dtype=F64).index_add(0, mesh.conn.reshape(-1), ones)[:, None]
    dt = 1e-6
    u, v = u0 * live, v0 * live
    a = -mesh.force(u, lam, mu) / mass * live
    for _ in range(case["steps"]):
        u = u + dt * v + 0.5 * dt * dt * a
        new = -mesh.force(u, lam, mu) / mass * live
        v = v + 0.5 * dt * (a + new)
        a = new
    J = (torch.from_numpy(q["w"]).to(DEV) * u).sum()
    return [float(J.detach())] + [g.cpu().numpy() for g in torch.autograd.grad(J, (u0, v0, lam, mu))]


def _exact_fit(case, U, A, S):
    def pod(X, r):
        w, V = torch.linalg.eigh(X @ X.T)
        w, V = w.flip(0), V.flip(1)
        return _orthonormal(X.T @ (V[:, :r] / w[:r].sqrt())), w.clamp(min=0).sqrt()

    r, rs = case["r"], case["r_s"]
    Phi, sigma = pod(U, r)
    Phi_S, sigma_s = pod(S, rs)
    Ub = U @ Phi
    cols = [Ub]
    i, j = torch.triu_indices(r, r, device=DEV)
    if case["model"] != "linear":
        cols.append(Ub[:, i] * Ub[:, j])
    if case["model"] == "cubic":
        t = torch.tensor([(a, b, c) for a in range(r) for b in range(a, r) for c in range(b, r)], device=DEV).T
        cols.append(Ub[:, t[0]] * Ub[:, t[1]] * Ub[:, t[2]])
    D = torch.cat(cols + [S @ Phi_S, torch.ones(len(U), 1, device=DEV, dtype=F64)], 1)
    Y = A @ Phi
    if D.shape[1] > len(D):
        O = D.T @ torch.cholesky_solve(Y, torch.linalg.cholesky(D @ D.T + 1e-2 * torch.eye(len(D), device=DEV, dtype=F64)))
    else:
        O = torch.cholesky_solve(D.T @ Y, torch.linalg.cholesky(D.T @ D + 1e-2 * torch.eye(D.shape[1], device=DEV, dtype=F64)))
    O = O.T.cpu().numpy()
    nq = r * (r + 1) // 2
    at = r if case["model"] == "linear" else r + nq
    out = {"Phi": Phi, "Phi_S": Phi_S, "sigma": sigma, "sigma_s": sigma_s}
    out = {k: v.cpu().numpy() for k, v in out.items()}
    out.update(K=O[:, :r], H=O[:, r:r + nq] if at > r else np.zeros((r, nq)), c=O[:, -1], B=O[:, -1 - rs:-1])
    if case["model"] == "cubic":
        out["C"] = O[:, at:-1 - rs]
    return _with_signs(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "force":
        dims, h, u, lam, mu, lam_e, mu_e, ybar = _force_inputs(case, seed)
        if not case["grad"]:
            mesh = _Mesh(dims, h, case["material"], lam, mu)
            return mesh.force(u, lam_e, mu_e) if case["per_element"] else mesh.force(u)
        if not case["per_element"]:
            lam_e, mu_e = torch.full_like(lam_e, lam), torch.full_like(mu_e, mu)
        args = [t.requires_grad_(True) for t in (u, lam_e, mu_e)]
        f = _Mesh(dims, h, case["material"], None, None).force(*args)
        return (f.detach(),) + torch.autograd.grad(f, args, ybar)
    if kind == "step":
        ne, _ = _sizes(case)
        if case["implicit"] and ne > 20000:
            return None
        spec, ops = _step_problem(case, seed)
        return _as_run([_exact_step(spec, ops)], spec)
    if kind == "batch":
        if case["samples"] * case["n_max"] ** 3 > 1e5:
            return None
        specs, ops = _batch_problems(case, seed)
        return _as_run([_exact_step(spec, o) for spec, o in zip(specs, ops)], specs[0])
    if kind == "adjoint":
        return _exact_adjoint(case, _adjoint_inputs(case, seed))
    return _exact_fit(case, *_fit_inputs(case, seed))
