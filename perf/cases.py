"""The calls a user of the library makes, at the sizes they make them: what performance work measures.

``listed`` gives one case per kind of call; ``draw`` gives more cases of the same kinds over the
ranges those stand for (grids from a few patches to a quarter million DOF and more, odd and
unequal sides, open and periodic, both precisions, both Hessians, both assemblies). ``prepare``
builds the shell, batch or network that a program keeps and one call's inputs; ``run`` makes the
call through the Python binding; ``exact`` restates the element, mass and network formulas in
plain 64-bit torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_14839_gb300 import bhem
from paper_2312_14839_gb300 import scenes as S

SHEET = S.SHEET_MATERIAL


def listed():
    return [
        # Elastic energy and gradient of a small sheet without a shell object: a plug-in or an
        # outer optimiser calling it in a loop, where the call's latency is all that counts.
        {"name": "energy_grad_10", "kind": "energy_grad", "nu": 10, "nv": 10, "shape": "sheet"},
        # Per-patch energies, gradients and 48 x 48 Hessians of the large throughput sheet, for a
        # program that assembles them itself.
        {"name": "element_256", "kind": "element", "nu": 256, "nv": 256, "shape": "sheet",
         "precision": "mixed", "hessian": "exact"},
        # Assembled energy, gradient and K + M / dt^2 of the parasol strip, handed to another solver.
        {"name": "assemble_annulus_280x5", "kind": "assemble", "nu": 280, "nv": 5, "shape": "annulus",
         "precision": "mixed", "hessian": "exact", "assembly": "atomic"},
        # One Newton iteration of the large sheet with a fixed budget of 50 PCG iterations: the
        # throughput form of the implicit step, bound by the matrix's passes over memory.
        {"name": "newton_256_pcg50", "kind": "newton", "scene": "sinusoid", "nu": 256, "nv": 256,
         "shape": "sheet", "precision": "mixed", "hessian": "exact", "assembly": "atomic", "pcg_fixed": 50},
        # An implicit-Euler step to 1e-8 of the 30 x 30 sheet whose centre is twisted: the paper's
        # usual scene size, many short kernels.
        {"name": "newton_twist_30", "kind": "newton", "scene": "twist", "nu": 30, "nv": 30, "shape": "sheet",
         "precision": "mixed", "hessian": "exact", "assembly": "atomic", "pcg_fixed": 0},
        # The same of the periodic parasol strip falling from a rough state.
        {"name": "newton_annulus_280x5", "kind": "newton", "scene": "noisy", "nu": 280, "nv": 5,
         "shape": "annulus", "precision": "mixed", "hessian": "exact", "assembly": "atomic", "pcg_fixed": 0},
        # A step of the 10 x 10 sheet, everything in FP64: the validation runs of the method.
        {"name": "newton_fp64_10", "kind": "newton", "scene": "noisy", "nu": 10, "nv": 10, "shape": "sheet",
         "precision": "fp64", "hessian": "exact", "assembly": "atomic", "pcg_fixed": 0},
        # A step of the 64 x 64 sheet from the network's warm start, inference included.
        {"name": "warm_newton_64", "kind": "newton", "scene": "warm", "nu": 64, "nv": 64, "shape": "sheet",
         "precision": "mixed", "hessian": "exact", "assembly": "atomic", "pcg_fixed": 0},
        # One step of 512 independent sheets of uneven sizes and materials: data generation.
        {"name": "batch_512", "kind": "batch", "shells": 512, "n_min": 4, "n_max": 40},
        # A depth frame of the draped sheet: one ray per pixel.
        {"name": "rays_drape_1024x768", "kind": "rays", "scene": "drape", "width": 1024, "height": 768,
         "variant": "newton"},
        # Contacts of a moving point cloud with the moving drape over one step.
        {"name": "ccd_drape_262144", "kind": "ccd", "scene": "drape", "points": 262144, "variant": "newton"},
        # Loss and weight gradients of one training minibatch, read back as a logger or an outer
        # optimiser does.
        {"name": "mlp_gradients_16384", "kind": "mlp", "rows": 16384, "data_rows": 262144},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _grid_sides(rng, lo, hi):
    """Two sides between lo and hi, their product spread over its logarithm."""
    nu = _log_int(rng, lo, hi)
    return nu, max(lo, min(hi, _log_int(rng, max(lo, nu // 4), min(hi, nu * 4))))


def draw(rng):
    kind = rng.choice(["energy_grad", "element", "assemble", "newton_pcg50", "newton_twist", "newton_noisy",
                       "newton_fp64", "newton_warm", "batch", "rays", "ccd", "mlp"])
    hessian = "pseudo" if rng.random() < 0.25 else "exact"
    assembly = "color" if rng.random() < 0.25 else "atomic"
    if kind == "energy_grad":
        nu, nv = _grid_sides(rng, 4, 200)
        return {"kind": "energy_grad", "nu": nu, "nv": nv, "shape": rng.choice(["sheet", "annulus"])}
    if kind == "element":
        nu, nv = _grid_sides(rng, 6, 256)
        return {"kind": "element", "nu": nu, "nv": nv, "shape": rng.choice(["sheet", "annulus"]),
                "precision": "mixed", "hessian": hessian}
    if kind == "assemble":
        nu, nv = _grid_sides(rng, 6, 256)
        return {"kind": "assemble", "nu": nu, "nv": nv, "shape": rng.choice(["sheet", "annulus", "cylinder"]),
                "precision": "mixed", "hessian": hessian, "assembly": assembly}
    if kind == "newton_pcg50":
        nu, nv = _grid_sides(rng, 16, 256)
        return {"kind": "newton", "scene": "sinusoid", "nu": nu, "nv": nv, "shape": rng.choice(["sheet", "annulus"]),
                "precision": "mixed", "hessian": "exact", "assembly": assembly, "pcg_fixed": 50}
    if kind == "newton_twist":
        n = rng.randint(10, 64)
        return {"kind": "newton", "scene": "twist", "nu": n, "nv": n, "shape": "sheet", "precision": "mixed",
                "hessian": hessian, "assembly": assembly, "pcg_fixed": 0}
    if kind == "newton_noisy":
        nu, nv = _grid_sides(rng, 6, 128)
        return {"kind": "newton", "scene": "noisy", "nu": nu, "nv": nv,
                "shape": rng.choice(["sheet", "annulus"]), "precision": "mixed", "hessian": "exact", "assembly": assembly, "pcg_fixed": 0}
    if kind == "newton_fp64":
        nu, nv = _grid_sides(rng, 4, 32)
        return {"kind": "newton", "scene": "noisy", "nu": nu, "nv": nv, "shape": "sheet", "precision": "fp64",
                "hessian": "exact", "assembly": assembly, "pcg_fixed": 0}
    if kind == "newton_warm":
        n = rng.randint(24, 96)
        return {"kind": "newton", "scene": "warm", "nu": n, "nv": n, "shape": "sheet", "precision": "mixed",
                "hessian": "exact", "assembly": "atomic", "pcg_fixed": 0}
    if kind == "batch":
        return {"kind": "batch", "shells": _log_int(rng, 8, 400), "n_min": 4, "n_max": rng.randint(12, 40)}
    if kind == "rays":
        w = _log_int(rng, 64, 960)
        return {"kind": "rays", "scene": rng.choice(["drape", "cylinder", "plane"]), "width": w,
                "height": max(48, int(w * 0.72)), "variant": rng.choice(["newton", "midpoint"])}
    if kind == "ccd":
        return {"kind": "ccd", "scene": rng.choice(["drape", "plane", "cylinder"]),
                "points": _log_int(rng, 1000, 262144), "variant": rng.choice(["newton", "midpoint"])}
    return {"kind": "mlp", "rows": _log_int(rng, 1000, 65536), "data_rows": 262144}


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
def _rest(case):
    if case["shape"] == "annulus":
        return S.annulus(case["nu"], case["nv"])
    if case["shape"] == "cylinder":
        return S.cylinder(case["nu"], case["nv"])
    # square patches of the unit sheet's size, so that a long sheet is longer, not finer
    side = max(case["nu"], case["nv"])
    return S.flat_sheet(case["nu"], case["nv"], case["nu"] / side, case["nv"] / side)


def _normalised_params(case, g):
    """xi mapped to one period per unit length, and the slopes of that map."""
    x1, x2 = S.node_params(g)
    l1, l2 = g.nu * g.dxi1, g.nv * g.dxi2
    return x1 / l1, x2 / l2, 1.0 / l1, 1.0 / l2


def _sinusoid(case, g, rest, seed, amplitude):
    return rest + S.sinusoid_displacement(*_normalised_params(case, g), seed, amplitude)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a).reshape(-1), device="cuda")


def _mlp_norm():
    """Column statistics of the size that recorded sheet trajectories have (metres, metres per second)."""
    in_std = np.concatenate([np.full(12, 1e-2), np.full(12, 0.1), np.full(3, 1e-3), np.full(1, 0.1)])
    return np.zeros(28), in_std, np.zeros(12), np.full(12, 1e-6)


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind in ("energy_grad", "element", "assemble"):
        g, rest = _rest(case)
        q = _sinusoid(case, g, rest, seed, 0.02)
        state.update(grid=g, rest=_dev(rest), q=_dev(q))
        if kind == "energy_grad":
            state["energy"] = torch.empty(1, dtype=torch.float64, device="cuda")
            state["grad"] = torch.empty(g.n_dof, dtype=torch.float64, device="cuda")
        else:
            state["shell"] = bhem.Shell(g, SHEET, state["rest"], precision=case["precision"],
                                        hessian=case["hessian"], assembly=case.get("assembly", "atomic"))
        return state
    if kind == "newton":
        g, rest = _rest(case)
        rng = np.random.Generator(np.random.PCG64(seed))
        scene, mask, q_fixed, v0, gravity, dt, tau = case["scene"], None, None, None, (0.0, 0.0, -9.81), 1e-3, 0.0
        if scene == "sinusoid":
            q0, tau = _sinusoid(case, g, rest, seed, 0.05), 1.0   # the level that a rollout of it carries
        elif scene == "noisy":
            # noise of a hundredth of the smallest patch side (1 mm on the 10 x 10 sheet of one metre)
            side = min(g.dxi1 * (0.2 if case["shape"] == "annulus" else 1.0), g.dxi2)
            q0 = S.noisy(rest, 1e-2 * side, seed)
            nodes = [0, g.n_nodes - 1]
            mask = S.pinned_mask(g, nodes)
            q_fixed = q0
        elif scene == "twist":
            gravity, dt = (0.0, 0.0, 0.0), 2e-3
            q0 = S.noisy(rest, 1e-6, seed)
            mask, q_fixed = S.twist_prescription(g, rest, 1, rng.uniform(1.5, 2.5))
        else:
            amp = 1e-4
            q0 = _sinusoid(case, g, rest, seed, amp)
            v0 = (_sinusoid(case, g, rest, seed + 1, 10 * amp) - rest).reshape(-1)
            rates = S.corner_twist_rates(seed)[0]
            mask, q_fixed = S.corner_twist_prescription(g, rest, 1, rates)
            net = bhem.Mlp(g.n_nodes)
            params, norm = S.mlp_init_params(seed), _mlp_norm()
            net.set_params(params)
            net.set_normalization(*norm)
            state.update(net=net, warm=torch.empty(g.n_dof, dtype=torch.float64, device="cuda"))
        q0_d = _dev(q0)
        v0_d = torch.zeros_like(q0_d) if v0 is None else _dev(v0)
        fixed = case["pcg_fixed"]
        state.update(
            shell=bhem.Shell(g, SHEET, _dev(rest), precision=case["precision"], hessian=case["hessian"],
                             assembly=case["assembly"]),
            q0=q0_d, v0=v0_d, q=q0_d.clone(), v=v0_d.clone(), dt=dt,
            mask=None if mask is None else _dev(mask), q_fixed=None if q_fixed is None else _dev(q_fixed),
            params=bhem.step_params(dt=dt, gravity=gravity, newton_max=1 if fixed else 200, pcg_max=2000,
                                    pcg_fixed_iters=fixed, tau_carry=tau))
        return state
    if kind == "batch":
        sheets = S.batch_sheets(case["shells"], seed=4, n_min=case["n_min"], n_max=case["n_max"])
        q0 = _dev(np.concatenate([S.noisy(r, 1e-3, [seed, k]).reshape(-1) for k, (_, _, r, _) in enumerate(sheets)]))
        masks = []
        for g, _, _, _ in sheets:
            c = S.corner_nodes(g)
            masks.append(S.pinned_mask(g, [c[0], c[3]]))
        state.update(batch=bhem.Batch([(g, m, r) for g, m, r, _ in sheets], stream=torch.cuda.current_stream()),
                     q0=q0, q=q0.clone(), v=torch.zeros_like(q0), mask=_dev(np.concatenate(masks)),
                     params=bhem.step_params(dt=1e-3))
        return state
    if kind == "rays":
        rng = np.random.Generator(np.random.PCG64(seed))
        g, q, eye, target = S.ray_scenes()[case["scene"]]
        if case["scene"] == "drape":
            q = S.sheet_sinusoid(30, seed, 0.05)[2]
        eye = tuple(float(e + rng.uniform(-0.02, 0.02)) for e in eye)
        o, d = S.camera_rays(case["width"], case["height"], eye, target)
        n = o.shape[0]
        state.update(shell=bhem.Shell(g, SHEET, _dev(q), precision="mixed"), q=_dev(q),
                     o=torch.as_tensor(o, device="cuda"), d=torch.as_tensor(d, device="cuda"),
                     variant=case["variant"], out=_hits(n, "tau"))
        return state
    if kind == "ccd":
        g, q, dq, x0, dx = S.ccd_scene(case["scene"], case["points"], seed)
        state.update(shell=bhem.Shell(g, SHEET, _dev(q), precision="mixed"), q=_dev(q), dq=_dev(dq),
                     x0=torch.as_tensor(x0, device="cuda"), dx=torch.as_tensor(dx, device="cuda"),
                     variant=case["variant"], out=_hits(case["points"], "s"))
        return state
    X, T, idx = _mlp_data(case, seed)
    net = bhem.Mlp(case["rows"])
    net.set_params(S.mlp_init_params(seed, 1.0))
    net.set_normalization(*_mlp_norm())
    state.update(net=net, X=X, T=T, idx=idx)
    return state


def _hits(n, key):
    return {key: torch.empty(n, dtype=torch.float64, device="cuda"),
            "patch": torch.empty(n, dtype=torch.int32, device="cuda"),
            "uv": torch.empty((n, 2), dtype=torch.float64, device="cuda"),
            "flags": torch.empty(n, dtype=torch.int32, device="cuda")}


def _mlp_data(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    _, in_std, _, out_std = _mlp_norm()
    X = torch.randn(case["data_rows"], 28, generator=gen, device="cuda") * torch.as_tensor(in_std, dtype=torch.float32, device="cuda")
    T = torch.randn(case["data_rows"], 12, generator=gen, device="cuda") * torch.as_tensor(out_std, dtype=torch.float32, device="cuda")
    idx = torch.randint(0, case["data_rows"], (case["rows"],), generator=gen, device="cuda", dtype=torch.int32)
    return X, T, idx


# ---------------------------------------------------------------------------------------------
# The calls
# ---------------------------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "energy_grad":
        bhem.energy_grad_noalloc(state["grid"], SHEET, state["rest"], state["q"], state["energy"], state["grad"])
        return {"energy": state["energy"], "grad": state["grad"]}
    if kind == "element":
        E, G, H = state["shell"].element_egh(state["q"])
        return {"energy": E, "grad": G, "hessian": H}
    if kind == "assemble":
        E, G = state["shell"].energy_grad_hess(state["q"], mass_scale=1e6)
        rp, col, val = state["shell"].bsr()
        return {"energy": E, "grad": G, "row_ptr": rp, "col": col, "values": val}
    if kind == "newton":
        q, v, warm = state["q"], state["v"], state.get("warm")
        q.copy_(state["q0"])
        v.copy_(state["v0"])
        if warm is not None:
            state["net"].warm_start(state["shell"], q, v, state["dt"], warm)
        st = state["shell"].newton_step(q, v, state["params"], mask=state["mask"], q_fixed=state["q_fixed"], warm=warm)
        out = {"q": q, "v": v, "status": st["status"]}
        if warm is not None:
            out["warm"] = warm
        return out
    if kind == "batch":
        q, v = state["q"], state["v"]
        q.copy_(state["q0"])
        v.zero_()
        st = state["batch"].newton_step(q, v, state["params"], mask=state["mask"], q_fixed=state["q0"])
        return {"q": q, "v": v, "status": np.array([s["status"] for s in st])}
    if kind == "rays":
        return state["shell"].trace_rays(state["q"], state["o"], state["d"], variant=state["variant"], out=state["out"])
    if kind == "ccd":
        return state["shell"].ccd_points(state["q"], state["dq"], state["x0"], state["dx"], variant=state["variant"],
                                         out=state["out"])
    loss = state["net"].gradients(state["X"], state["T"], idx=state["idx"])
    return {"loss": loss, "grads": state["net"].get_grads()}


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------
# Per patch: 16 Gauss points x (interpolation of 5 kinds x 3 components by sum factorisation, the
# energy and its gradient, and the gradient's way back); with the Hessian, 16 matrices of 15 x 15
# and their contraction (T = Phi^T M, K = T Phi, symmetric half).
_EG_FLOPS = 2.0 * (1536 + 1536 + 16 * 190)
_HESS_FLOPS = 2.0 * (16 * 15 * 48 * 5 + 1176 * 80 + 16 * 1200)
# Newton iterations and PCG iterations per Newton iteration that the scenes take to 1e-8.
_NEWTON = {"noisy": (4, 25), "twist": (3, 26), "warm": (2, 28)}


def _n_blocks(g):
    """Blocks of the 12 x 12 matrix: node pairs that share a patch."""
    a = 3 * g.n1 - (0 if g.periodic_u else 2)
    b = 3 * g.n2 - (0 if g.periodic_v else 2)
    return a * b


def work(case):
    kind = case["kind"]
    if kind in ("energy_grad", "element", "assemble", "newton"):
        g, _ = _rest(case)
        np_, nd, nb = g.n_patches, g.n_dof, _n_blocks(g)
        if kind == "energy_grad":
            return {"bytes": 3 * 8 * nd, "flops": np_ * _EG_FLOPS}
        if kind == "element":
            return {"bytes": 2 * 8 * nd + np_ * (8 + 48 * 8 + 2304 * 4), "flops": np_ * (_EG_FLOPS + _HESS_FLOPS)}
        if kind == "assemble":
            return {"bytes": 3 * 8 * nd + nb * 576 + nb * 8 + 8 * nd, "flops": np_ * (_EG_FLOPS + _HESS_FLOPS)}
        size = 8 if case["precision"] == "fp64" else 4
        newton, pcg = (1, case["pcg_fixed"]) if case["pcg_fixed"] else _NEWTON[case["scene"]]
        # inputs and outputs once; per PCG iteration a matrix and a block-diagonal product
        return {"bytes": 8 * nd * 6 + nb * 144 * size,
                "flops": newton * (np_ * (2 * _EG_FLOPS + _HESS_FLOPS) + pcg * (2.0 * 144 * nb + 2.0 * 12 * nd + 10.0 * nd))}
    if kind == "batch":
        mean = (case["n_min"] + case["n_max"]) / 2.0
        patches = case["shells"] * (mean * mean + (case["n_max"] - case["n_min"]) ** 2 / 12.0)
        nodes = case["shells"] * ((mean + 1) ** 2 + (case["n_max"] - case["n_min"]) ** 2 / 12.0)
        return {"bytes": nodes * (12 * 8 * 6 + 9 * 576),
                "flops": 4.4 * (patches * (2 * _EG_FLOPS + _HESS_FLOPS) + 60 * nodes * (2.0 * 144 * 9 + 34 * 12))}
    if kind == "rays":
        n = case["width"] * case["height"]
        return {"bytes": n * (48 + 32), "flops": n * 1324.0 * 4}
    if kind == "ccd":
        return {"bytes": case["points"] * (48 + 32), "flops": case["points"] * 2950.0 * 4}
    per_row = 2.0 * (28 * 256 + 2 * 256 * 256 + 256 * 12)
    return {"bytes": case["rows"] * 4 * 41 + 2 * 4 * 142092, "flops": case["rows"] * (3 * per_row - 2.0 * 28 * 256)}


# ---------------------------------------------------------------------------------------------
# The same numbers in plain 64-bit torch
# ---------------------------------------------------------------------------------------------
def _basis(t):
    """Cubic Hermite factors [d, p, r] of theta: derivative d, end p, value or slope r."""
    f = [2 * t ** 3 - 3 * t * t + 1, 6 * t * t - 6 * t, 12 * t - 6]
    h = [t ** 3 - 2 * t * t + t, 3 * t * t - 4 * t + 1, 6 * t - 4]
    u = 1 - t
    f1 = [2 * u ** 3 - 3 * u * u + 1, -(6 * u * u - 6 * u), 12 * u - 6]
    h1 = [-(u ** 3 - 2 * u * u + u), 3 * u * u - 4 * u + 1, -(6 * u - 4)]
    return [[[f[d], h[d]], [f1[d], h1[d]]] for d in range(3)]


def _shape_table(g):
    """phi [16 Gauss points, 6 kinds (value, 1, 2, 11, 22, 12), 16 shape functions] and weights [16]."""
    xi, xo = math.sqrt(3 / 7 - 2 / 7 * math.sqrt(1.2)), math.sqrt(3 / 7 + 2 / 7 * math.sqrt(1.2))
    wi, wo = (18 + math.sqrt(30)) / 36, (18 - math.sqrt(30)) / 36
    x, w = [-xo, -xi, xi, xo], [wo, wi, wi, wo]
    phi, wt = np.zeros((16, 6, 16)), np.zeros(16)
    kinds = [(0, 0), (1, 0), (0, 1), (2, 0), (0, 2), (1, 1)]
    for j in range(4):
        for i in range(4):
            b1, b2 = _basis(0.5 * (1 + x[i])), _basis(0.5 * (1 + x[j]))
            wt[4 * j + i] = 0.25 * g.dxi1 * g.dxi2 * w[i] * w[j]
            for k, (d1, d2) in enumerate(kinds):
                for p2 in range(2):
                    for p1 in range(2):
                        for s in range(2):
                            for r in range(2):
                                phi[4 * j + i, k, (p1 + 2 * p2) * 4 + r + 2 * s] = (
                                    b1[d1][p1][r] * b2[d2][p2][s] * g.dxi1 ** (r - d1) * g.dxi2 ** (s - d2))
    return torch.as_tensor(phi, device="cuda"), torch.as_tensor(wt, device="cuda")


def _patch_nodes(g):
    pv, pu = np.meshgrid(np.arange(g.nv), np.arange(g.nu), indexing="ij")
    pu, pv = pu.reshape(-1), pv.reshape(-1)
    n = [((pv + b) % g.n2) * g.n1 + (pu + a) % g.n1 for b in range(2) for a in range(2)]
    return torch.as_tensor(np.stack(n, axis=1), device="cuda")


def _forms(d):
    """First and second fundamental forms of [..., 5, 3] derivatives."""
    a1, a2 = d[..., 0, :], d[..., 1, :]
    n = torch.linalg.cross(a1, a2)
    sq = torch.sqrt((n * n).sum(-1))
    b = (d[..., 2:, :] * n.unsqueeze(-2)).sum(-1) / sq.unsqueeze(-1)
    return (a1 * a1).sum(-1), (a2 * a2).sum(-1), (a1 * a2).sum(-1), b, sq


def _density(d, rest, mat, b=None):
    """Energy per parameter area at derivatives d [15] against rest derivatives [15] (b: the second
    fundamental form, where it is not that of d)."""
    lam = mat.young * mat.poisson / (1 - mat.poisson ** 2)
    mu, h = mat.young / (2 * (1 + mat.poisson)), mat.thickness
    a11, a22, a12, own, _ = _forms(d.view(5, 3))
    r11, r22, r12, rb, rsq = _forms(rest.view(5, 3))
    b = own if b is None else b
    det = r11 * r22 - r12 * r12
    i11, i22, i12 = r22 / det, r11 / det, -r12 / det

    def quad(e11, e22, e12):
        tr = i11 * e11 + i22 * e22 + 2 * i12 * e12
        m11, m12 = i11 * e11 + i12 * e12, i11 * e12 + i12 * e22
        m21, m22 = i12 * e11 + i22 * e12, i12 * e12 + i22 * e22
        return 0.5 * lam * tr * tr + mu * (m11 * m11 + 2 * m12 * m21 + m22 * m22)

    A = [0.5 * (a11 - r11), 0.5 * (a22 - r22), 0.5 * (a12 - r12)]
    B = [0.5 * (b[i] - rb[i]) for i in range(3)]
    return rsq * (h * quad(*A) + h ** 3 / 3 * quad(*B))


def _element_exact(g, rest, q, mat, hessian, pseudo):
    """Energies [np], gradients [np, 48] and, if asked, Hessians [np, 48, 48]."""
    phi, wt = _shape_table(g)
    nodes = _patch_nodes(g)
    ders = phi[:, 1:, :]

    def energy(d, r):
        return _density(d, r, mat)

    def pseudo_energy(d, d0, r):   # the bending strain linearised at d0
        b0, db = torch.func.jvp(lambda x: _forms(x.view(5, 3))[3], (d0,), (d - d0,))
        return _density(d, r, mat, b0 + db)

    E, G, H = [], [], []
    for k in range(0, nodes.shape[0], 4096):
        nd = nodes[k:k + 4096]
        dq = torch.einsum("gki,pic->pgkc", ders, q.view(-1, 12)[nd].reshape(-1, 16, 3)).reshape(-1, 15)
        dr = torch.einsum("gki,pic->pgkc", ders, rest.view(-1, 12)[nd].reshape(-1, 16, 3)).reshape(-1, 15)
        e = torch.func.vmap(energy)(dq, dr).view(-1, 16)
        gr = torch.func.vmap(torch.func.grad(energy))(dq, dr).view(-1, 16, 5, 3)
        E.append((e * wt).sum(1))
        G.append(torch.einsum("g,gki,pgkc->pic", wt, ders, gr).reshape(-1, 48))
        if hessian:
            if pseudo:
                M = torch.func.vmap(torch.func.jacfwd(torch.func.jacrev(pseudo_energy)))(dq, dq, dr)
            else:
                M = torch.func.vmap(torch.func.jacfwd(torch.func.jacrev(energy)))(dq, dr)
            M = M.view(-1, 16, 5, 3, 5, 3)
            T = torch.einsum("g,gki,pgkcld->pgicld", wt, ders, M)
            H.append(torch.einsum("pgicld,glj->picjd", T, ders).reshape(-1, 48, 48))
    return torch.cat(E), torch.cat(G), torch.cat(H) if hessian else None


def _mlp_exact(params, norm, X, T):
    """Network output [rows, 12], loss and packed gradients in 64 bits (exact GELU)."""
    p = torch.as_tensor(params, dtype=torch.float64, device="cuda").requires_grad_(T is not None)
    im, isd, om, osd = (torch.as_tensor(np.asarray(a, dtype=np.float32), device="cuda").double() for a in norm)
    a, off = (X.double() - im) / isd, 0
    for l, (fi, fo) in enumerate(S.MLP_LAYERS):
        W, b = p[off:off + fi * fo].view(fo, fi), p[off + fi * fo:off + fi * fo + fo]
        off += fi * fo + fo
        a = a @ W.T + b
        if l < len(S.MLP_LAYERS) - 1:
            a = torch.nn.functional.gelu(a)
    if T is None:
        return a * osd + om
    loss = ((a - (T.double() - om) / osd) ** 2).mean()
    return loss.item(), torch.autograd.grad(loss, p)[0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("energy_grad", "element", "assemble"):
        g, rest = _rest(case)
        q = _dev(_sinusoid(case, g, rest, seed, 0.02))
        rest = _dev(rest)
        pseudo = case.get("hessian") == "pseudo"
        E, G, H = _element_exact(g, rest, q, SHEET, kind != "energy_grad", pseudo)
        if kind == "element":
            return {"energy": E, "grad": G, "hessian": H}
        nodes = _patch_nodes(g)
        grad = torch.zeros(g.n_nodes, 12, dtype=torch.float64, device="cuda")
        grad.index_add_(0, nodes.reshape(-1), G.view(-1, 12))
        if kind == "energy_grad":
            return {"energy": E.sum().view(1), "grad": grad.view(-1)}
        # K + 1e6 M on the sorted node pairs
        phi, wt = _shape_table(g)
        dr = torch.einsum("gki,pic->pgkc", phi[:, 1:, :], rest.view(-1, 12)[nodes].reshape(-1, 16, 3))
        m = torch.einsum("pg,gi,gj->pij", SHEET.density * SHEET.thickness * wt * _forms(dr)[4], phi[:, 0], phi[:, 0])
        H = H + 1e6 * torch.einsum("pij,cd->picjd", m, torch.eye(3, dtype=torch.float64, device="cuda")).reshape(-1, 48, 48)
        key = (nodes.unsqueeze(2) * g.n_nodes + nodes.unsqueeze(1)).reshape(-1)
        pairs, at = torch.unique(key, return_inverse=True)
        val = torch.zeros(pairs.numel(), 12, 12, dtype=torch.float64, device="cuda")
        val.index_add_(0, at, H.view(-1, 4, 12, 4, 12).permute(0, 1, 3, 2, 4).reshape(-1, 12, 12))
        return {"energy": E.sum().view(1), "grad": grad.view(-1), "row_ptr": None, "col": None, "values": val}
    if kind == "mlp":
        X, T, idx = _mlp_data(case, seed)
        i = idx.long()
        loss, grads = _mlp_exact(S.mlp_init_params(seed, 1.0), _mlp_norm(), X[i], T[i])
        return {"loss": loss, "grads": grads.cpu().numpy()}
    # A Newton step to a tolerance and a subdivision search have no value of their own beside where
    # they stop.
    return None
