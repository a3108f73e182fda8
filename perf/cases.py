"""Workloads for timing the library through its Python entry points.

``listed()`` are the calls that its users make, from one airfoil on a designer's
screen to a thousand finely panelled ones; ``draw(rng)`` gives others of the same
ranges.  A case is a plain dict:

  kind    'step'   PanelBatch.run(with_grad=True), mixed precision: strengths,
                   forces and dCl/dnodes (a gradient-refined generation)
          'solve'  PanelBatch.run(with_grad=False): strengths and forces
          'fp64'   PanelBatch.run(with_grad=True) of the plain FP64 path
          'replay' PanelBatch.step() of a captured step with gradients
          'polar'  PanelBatch.polar: Cl at `angles` angles per airfoil
          'cl'     PanelCl forward and backward (loss on the lift)
          'vjp'    PanelSolve forward and backward (loss on u, Cp and Cl)
          'ga'     GeneticOptimizer.evaluate: genome -> nodes -> solve -> drag
  batch   airfoils, and n_min, n_max: their panels, drawn from the case's own
          sizes (not from the seed), uniformly in between
  angles  of a polar

Airfoils are NACA 4-digit sections (camber 0-6 %, position 20-60 %, thickness
8-18 %, angle of attack -4 to 10 degrees) with cosine-spaced panels; with
``perturbed`` they carry eight smooth cosine modes of camber and thickness
(N(0, 0.005) chord), as a genetic algorithm's population does.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1511_02166_gb300.ga import GeneticOptimizer, default_bounds, default_control_x
from paper_1511_02166_gb300.solver import PanelBatch, PanelCl, PanelSolve

DEVICE = "cuda"


def _case(kind, batch, n_min, n_max, angles=0, perturbed=False):
    return {"kind": kind, "batch": batch, "n_min": n_min, "n_max": n_max, "angles": angles,
            "perturbed": perturbed}


def listed():
    return [
        # one section on a designer's screen: lift, pressures and gradient, latency only
        dict(_case("step", 1, 160, 160), name="one_airfoil_n160"),
        # the reference precision a small study is checked with: 64 sections, all FP64
        dict(_case("fp64", 64, 100, 100), name="fp64_b64_n100"),
        # a gradient step on a small population inside an optimisation loop (graph replay)
        dict(_case("replay", 64, 100, 100), name="replay_b64_n100"),
        # one generation of the genetic optimiser at the usual panel count, no gradient
        dict(_case("ga", 4096, 200, 200), name="ga_b4096_n200"),
        # the same population with gradients (gradient-refined generation)
        dict(_case("step", 4096, 200, 200), name="step_b4096_n200"),
        # lift gradients at 256 panels through autograd
        dict(_case("cl", 4096, 256, 256), name="autograd_cl_b4096_n256"),
        # a population of uneven panel counts
        dict(_case("step", 10000, 64, 512, perturbed=True), name="uneven_b10000_n64_512"),
        # an inverse-design loss on pressures: odd batch, odd sizes, autograd
        dict(_case("vjp", 777, 121, 333, perturbed=True), name="autograd_cp_b777_n121_333"),
        # lift curves: 16 angles from one factorisation
        dict(_case("polar", 1500, 150, 250, angles=16), name="polar_b1500_n150_250"),
        # a panel-count convergence study: few airfoils of very different size
        dict(_case("solve", 24, 50, 2047), name="study_b24_n50_2047"),
        # finely panelled sections with gradients
        dict(_case("step", 1024, 1024, 2048), name="large_b1024_n1024_2048"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "solve", "replay", "fp64", "polar", "cl", "vjp", "ga"])

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    n_max = log_int(20, 240 if kind == "fp64" else 400 if kind == "ga" else 2048)
    n_min = n_max if kind == "ga" or rng.random() < 0.3 else max(16, int(n_max * rng.uniform(0.3, 1)))
    # at most the pairs of 1024 airfoils of 1400 panels; the FP64 path is some 20 times slower
    cap = (1e8 if kind == "fp64" else 2.0e9) / n_max**2
    batch = max(1, min(log_int(1, 10000), int(cap)))
    if kind == "ga":
        batch += batch % 2
    return _case(kind, batch, min(n_min, n_max), n_max,
                 angles=rng.randint(2, 32) if kind == "polar" else 0,
                 perturbed=kind != "ga" and rng.random() < 0.4)


# -- inputs -------------------------------------------------------------------

def _sizes(case):
    """Panel counts of the case's airfoils (the same for every seed)."""
    rng = random.Random(1511 + 7 * case["batch"] + case["n_max"])
    n = [rng.randint(case["n_min"], case["n_max"]) for _ in range(case["batch"])]
    if len(n) > 1:
        n[rng.randrange(len(n))] = case["n_max"]
    return np.asarray(n, dtype=np.int64)


def _offsets(case):
    return np.concatenate([[0], np.cumsum(_sizes(case))]).astype(np.int64)


def _population(case, seed):
    """nodes [sum n][2] and alpha [B] in radians, float64 on the device."""
    gen = torch.Generator().manual_seed(int(seed) * 1000003 + case["batch"])
    B = case["batch"]

    def uniform(lo, hi):
        return (lo + (hi - lo) * torch.rand(B, generator=gen, dtype=torch.float64)).to(DEVICE)

    camber, pos, thick = uniform(0.0, 0.06), uniform(0.2, 0.6), uniform(0.08, 0.18)
    alpha = torch.deg2rad(uniform(-4.0, 10.0))
    sizes = torch.as_tensor(_sizes(case), device=DEVICE)
    b = torch.repeat_interleave(torch.arange(B, device=DEVICE), sizes)
    start = torch.as_tensor(_offsets(case)[:-1], device=DEVICE)
    k = torch.arange(len(b), device=DEVICE) - start[b]
    nu, nl = (sizes[b] + 1) // 2, sizes[b] // 2
    upper = k <= nu
    # cosine stations: trailing edge -> leading edge on top, back underneath
    beta = torch.where(upper, math.pi - math.pi * k / nu, math.pi * (k - nu) / nl)
    x = 0.5 * (1.0 - torch.cos(beta))
    x = torch.where(k == 0, torch.ones_like(x), x)
    sign = torch.where(upper, 1.0, -1.0).double()
    t, m, p = thick[b], camber[b], pos[b]
    yt = 5.0 * t * (0.2969 * torch.sqrt(x) - 0.1260 * x - 0.3516 * x**2 + 0.2843 * x**3 - 0.1036 * x**4)
    fore = x < p
    yc = torch.where(fore, m / p**2 * (2 * p * x - x**2),
                     m / (1 - p)**2 * ((1 - 2 * p) + 2 * p * x - x**2))
    slope = torch.where(fore, 2 * m / p**2 * (p - x), 2 * m / (1 - p)**2 * (p - x))
    cos, sin = 1.0 / torch.sqrt(1 + slope**2), slope / torch.sqrt(1 + slope**2)
    X, Y = x - sign * yt * sin, yc + sign * yt * cos
    if case["perturbed"]:
        amp = (0.005 * torch.randn(B, 8, generator=gen, dtype=torch.float64)).to(DEVICE)
        modes = torch.sin(beta[:, None] * torch.arange(1, 5, device=DEVICE))
        inner = (x > 0) & (x < 1)
        dyt = (amp[b, 4:] * modes).sum(1) * torch.sin(beta)
        # the thickness modes are scaled down where they would take more than
        # half of the section's own thickness away
        ratio = torch.where(inner, -dyt / (0.5 * yt.clamp_min(1e-12)), torch.zeros_like(x))
        worst = torch.zeros(B, dtype=torch.float64, device=DEVICE).scatter_reduce(
            0, b, ratio, "amax").clamp_min(1.0)
        Y = Y + torch.where(inner, (amp[b, :4] * modes).sum(1) + sign * dyt / worst[b],
                            torch.zeros_like(x))
    return torch.stack([X, Y], dim=1).contiguous(), alpha


def _upstream(case, seed):
    """Weights of a loss on u, Cp and Cl."""
    gen = torch.Generator().manual_seed(int(seed) * 1000003 + 1)
    total, B = int(_offsets(case)[-1]), case["batch"]
    return [torch.randn(n, generator=gen, dtype=torch.float64).to(DEVICE)
            for n in (total + B, total, B)]


def _angles(case, seed):
    gen = torch.Generator().manual_seed(int(seed) * 1000003 + 2)
    a = -4.0 + 14.0 * torch.rand(case["batch"], case["angles"], generator=gen, dtype=torch.float64)
    return torch.deg2rad(a).to(DEVICE)


def _bounds():
    """Genome bounds of a population of closed, reasonably thick sections: the
    outer 60 % of the optimiser's default band on either side."""
    lo, hi = default_bounds(default_control_x())
    half = len(lo) // 2
    lo2, hi2 = lo.copy(), hi.copy()
    lo2[:half] = lo[:half] + 0.4 * (hi - lo)[:half]
    hi2[half:] = hi[half:] - 0.4 * (hi - lo)[half:]
    return lo2, hi2


GA_ALPHA = math.radians(4.0)


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "ga":
        lo, hi = _bounds()
        state["ga"] = GeneticOptimizer(case["batch"], case["n_max"], GA_ALPHA, lo=lo, hi=hi,
                                       seed=int(seed), device=DEVICE)
        return state
    nodes, alpha = _population(case, seed)
    if kind in ("cl", "vjp"):
        w_u, w_cp, w_cl = _upstream(case, seed)
        state.update(nodes=nodes.requires_grad_(), offsets=_offsets(case), alpha=alpha, w_u=w_u,
                     w_cp=w_cp, w_cl=w_cl)
        return state
    pb = PanelBatch(nodes, _offsets(case), alpha, mode="fp64" if kind == "fp64" else "mixed",
                    device=DEVICE)
    if kind == "replay":
        pb.capture(with_grad=True)
    state["pb"] = pb
    if kind == "polar":
        state["alphas"] = _angles(case, seed)
    return state


def _forces(pb):
    return {"u": pb.u, "cp": pb.cp, "cl": pb.cl, "cl_p": pb.cl_p, "cd_p": pb.cd_p, "info": pb.info}


def run(state):
    kind = state["kind"]
    if kind == "ga":
        ga = state["ga"]
        ga.evaluate()
        pb = ga.pb
        return dict(_forces(pb), nodes=pb.nodes, ld=pb.ld, cd=pb.cd, cd_f=pb.cd_f, theta=pb.theta,
                    cf=pb.cf, sep=pb.sep)
    if kind == "cl":
        cl = PanelCl.apply(state["nodes"], state["offsets"], state["alpha"])
        (grad,) = torch.autograd.grad((state["w_cl"] * cl).sum(), state["nodes"])
        return {"cl": cl.detach(), "grad": grad}
    if kind == "vjp":
        u, cp, cl = PanelSolve.apply(state["nodes"], state["offsets"], state["alpha"])
        loss = (state["w_u"] * u).sum() + (state["w_cp"] * cp).sum() + (state["w_cl"] * cl).sum()
        (grad,) = torch.autograd.grad(loss, state["nodes"])
        return {"u": u.detach(), "cp": cp.detach(), "cl": cl.detach(), "grad": grad}
    pb = state["pb"]
    if kind == "polar":
        cl = pb.polar(state["alphas"])
        return {"cl": cl, "u_y": pb.u_y, "u_x": pb.u_x, "info": pb.info}
    if kind == "replay":
        pb.step()
    else:
        pb.run(with_grad=kind != "solve")
    out = _forces(pb)
    if kind != "solve":
        out.update(lam=pb.lam, grad=pb.grad)
    return out


def work(case):
    """Bytes: nodes and angles in, results out.  Operations: 90 per pair of panels
    for the matrix, 2/3 m^3 for the factor, 2 m^2 per system solved and two
    corrections with their residuals (4 m^2 each), 110 per pair for a gradient."""
    n = _sizes(case).astype(np.float64)
    m, kind = n + 1, case["kind"]
    grad = kind in ("step", "replay", "fp64", "cl", "vjp")
    systems = 2 if grad or kind == "polar" else 1
    passes = 2 if kind == "fp64" else 10
    flops = 90 * n**2 + 2 / 3 * m**3 + systems * passes * m**2 + (110 * n**2 if grad else 0)
    nbytes = 16 * n + 8
    if kind == "polar":
        nbytes = nbytes + 16 * m + 16 * case["angles"]
    elif kind == "cl":
        nbytes = nbytes + 16 + 16 * n
    elif kind == "vjp":
        nbytes = nbytes + 16 * m + 16 * n + 16 + 16 * n
    else:
        nbytes = nbytes + 8 * m + 8 * n + 28 + (8 * m + 16 * n if grad else 0)
        if kind == "ga":
            nbytes = nbytes + 144 + 16 * n + 32
    return {"bytes": float(nbytes.sum()), "flops": float(flops.sum())}


# -- the same results in 64 bits with plain torch -------------------------------

def _influence(z, nxt, n):
    """G [b][N][N] (row: control point, column: panel) of padded nodes z [b][N][2],
    nxt [b][N][2] the panels' ends, n [b] panel counts; 0 outside."""
    N = z.shape[1]
    p = 0.5 * (z + nxt)
    h = nxt - z
    L = torch.sqrt((h**2).sum(-1))
    t = h / L[..., None]
    d1 = p[:, :, None] - z[:, None]
    tx, ty = t[:, None, :, 0], t[:, None, :, 1]
    xi = d1[..., 0] * tx + d1[..., 1] * ty
    eta = d1[..., 1] * tx - d1[..., 0] * ty
    own = torch.eye(N, dtype=torch.bool, device=z.device)
    eta = eta.masked_fill(own, 0.0)
    xi2 = xi - L[:, None]
    theta = torch.atan2(eta * L[:, None], xi * xi2 + eta**2).masked_fill(own, 0.0)
    G = 0.5 * (xi * torch.log(xi**2 + eta**2) - xi2 * torch.log(xi2**2 + eta**2)) + eta * theta - L[:, None]
    k = torch.arange(N, device=z.device)
    ok = k[None] < n[:, None]
    return torch.where(ok[:, :, None] & ok[:, None], G / (2 * math.pi), torch.zeros_like(G))


def _pad(flat, idx, ok, fill):
    out = flat[idx.clamp_max(flat.shape[0] - 1)]
    return torch.where(ok[..., None] if out.dim() > ok.dim() else ok, out, fill)


def _exact_chunk(nodes, alpha, start, n, w):
    """Padded results of the airfoils at `start` with n panels: w the loss's weights
    (w_cl [b], w_u [b][N+1], w_cp [b][N]), or None for lambda and dCl/dnodes."""
    b, N = len(n), int(n.max())
    k = torch.arange(N, device=DEVICE)
    ok = k[None] < n[:, None]
    idx = start[:, None] + k[None]
    nxt = start[:, None] + (k[None] + 1) % n[:, None]
    far = torch.stack([10.0 + 2 * k, 10.0 + 0 * k], -1).double()[None].expand(b, N, 2)
    z = _pad(nodes, idx, ok, far).detach().requires_grad_()
    zn_far = far + torch.tensor([1.0, 0.0], dtype=torch.float64, device=DEVICE)

    def ends(zz):
        e = torch.gather(zz, 1, ((k[None] + 1) % n[:, None])[..., None].expand(b, N, 2))
        return torch.where(ok[..., None], e, zn_far)

    def system(zz):
        A = -_influence(zz, ends(zz), n)
        pc = 0.5 * (zz + ends(zz))
        rhs = pc[..., 1] * torch.cos(alpha)[:, None] - pc[..., 0] * torch.sin(alpha)[:, None]
        return A, torch.where(ok, rhs, torch.zeros_like(rhs))

    with torch.no_grad():
        A, rhs = system(z)
        M = torch.zeros(b, N + 1, N + 1, dtype=torch.float64, device=DEVICE)
        M[:, :N, :N] = A
        M[:, :N, N] = ok.double()
        M[:, N, 0] = 1.0
        M[torch.arange(b, device=DEVICE), N, n - 1] += 1.0
        pad = (~ok).nonzero(as_tuple=True)
        M[pad[0], pad[1], pad[1]] = 1.0
        full = torch.cat([rhs, torch.zeros_like(rhs[:, :1])], 1)
        basis = torch.cat([torch.where(ok, q, torch.zeros_like(q))[..., None] for q in
                           ((0.5 * (z + ends(z)))[..., 1], -(0.5 * (z + ends(z)))[..., 0])], -1)
        basis = torch.cat([basis, torch.zeros_like(basis[:, :1])], 1)
        LU, piv = torch.linalg.lu_factor(M)

        def solve(v, adjoint=False):
            x = torch.linalg.lu_solve(LU, piv, v, adjoint=adjoint)
            r = v - (M.mT if adjoint else M) @ x
            return x + torch.linalg.lu_solve(LU, piv, r, adjoint=adjoint)

        u = solve(full[..., None])[..., 0]
        bas = solve(basis)
        h = torch.where(ok[..., None], ends(z) - z, torch.zeros_like(z))
        L = torch.sqrt((h**2).sum(-1))
        g, cp = u[:, :N], torch.where(ok, 1 - u[:, :N]**2, torch.zeros_like(u[:, :N]))
        cl = 2 * (g * L).sum(1)
        fx, fy = -(cp * h[..., 1]).sum(1), (cp * h[..., 0]).sum(1)
        sa, ca = torch.sin(alpha), torch.cos(alpha)
        out = {"u": u, "cp": cp, "cl": cl, "cl_p": -fx * sa + fy * ca, "cd_p": fx * ca + fy * sa,
               "cl_yx": 2 * (bas[:, :N] * L[..., None]).sum(1), "u_y": bas[..., 0], "u_x": bas[..., 1]}
        du = torch.cat([2 * L, torch.zeros_like(L[:, :1])], 1)
        w_cl = torch.ones_like(cl) if w is None else w[0]
        if w is not None:
            du = du * w_cl[:, None] + w[1]
            du[:, :N] += torch.where(ok, -2 * w[2] * g, torch.zeros_like(g))
        lam = solve(du[..., None], adjoint=True)[..., 0]
        out["lam"] = lam
    # dJ/dnodes = explicit dCl + lambda^T (db - dM u) at fixed u and lambda
    A, rhs = system(z)
    hz = ends(z) - z
    Lz = torch.where(ok, torch.sqrt((hz**2).sum(-1)), torch.zeros_like(L))
    J = (2 * w_cl[:, None] * g * Lz).sum() + (lam[:, :N] * rhs).sum()
    J = J - torch.einsum("bj,bji,bi->", lam[:, :N], A, g)
    (out["grad"],) = torch.autograd.grad(J, z)
    return out


def exact(case, seed):
    kind = case["kind"]
    offs = _offsets(case)
    n = torch.as_tensor(_sizes(case), device=DEVICE)
    # a batched FP64 factorisation of more than ~10^11 operations per second is not to be had
    if float((n.double()**3).sum()) > 6e11:
        return None
    if kind == "ga":
        nodes, alpha = _spline(case, seed), torch.full((case["batch"],), GA_ALPHA,
                                                       dtype=torch.float64, device=DEVICE)
    else:
        nodes, alpha = _population(case, seed)
    w = _upstream(case, seed) if kind in ("cl", "vjp") else None
    B, total = case["batch"], int(offs[-1])
    start = torch.as_tensor(offs[:-1], device=DEVICE)
    res = {}

    def put(name, sel, val, off, m):
        if val.dim() == 1 or name == "cl_yx":
            res.setdefault(name, torch.zeros((B,) + tuple(val.shape[1:]), dtype=torch.float64,
                                             device=DEVICE))[sel] = val
            return
        k = torch.arange(val.shape[1], device=DEVICE)
        mask = k[None] < m[:, None]
        length = total + (B if off else 0)
        flat = res.setdefault(name, torch.zeros((length,) + tuple(val.shape[2:]),
                                                dtype=torch.float64, device=DEVICE))
        flat[((start[sel] + (sel if off else 0))[:, None] + k[None])[mask]] = val[mask]

    order = torch.argsort(n, descending=True)
    i = 0
    while i < B:
        N = int(n[order[i]])
        sel = order[i:i + max(1, int(1.5e7 / N**2))]
        i += len(sel)
        ws = None
        if w is not None:
            N1 = torch.arange(N + 1, device=DEVICE)
            mask = N1[None] < n[sel][:, None] + 1
            ws = [w[2][sel], torch.zeros(len(sel), N + 1, dtype=torch.float64, device=DEVICE),
                  torch.zeros(len(sel), N, dtype=torch.float64, device=DEVICE)]
            if kind == "vjp":
                ws[1][:, :N] = _pad(w[0], (start[sel] + sel)[:, None] + N1[None, :N],
                                    mask[:, :N], ws[2])
                ws[2] = _pad(w[1], start[sel][:, None] + N1[None, :N], mask[:, 1:], ws[2])
                # C follows an airfoil's last strength; padded, it sits in the last column
                last = w[0][start[sel] + sel + n[sel]]
                ws[1] = torch.where(N1[None] < n[sel][:, None], ws[1], torch.zeros_like(ws[1]))
                ws[1][:, N] = last
        part = _exact_chunk(nodes, alpha[sel], start[sel], n[sel], ws)
        for name, val in part.items():
            off = name in ("u", "lam", "u_y", "u_x")
            if off:  # C from the padded system's last column to its place after gamma
                val = val.clone()
                val[torch.arange(len(sel), device=DEVICE), n[sel]] = val[:, -1].clone()
            put(name, sel, val, off, n[sel] + (1 if off else 0))
    if kind == "cl":
        return {"cl": res["cl"], "grad": res["grad"]}
    if kind == "vjp":
        return {q: res[q] for q in ("u", "cp", "cl", "grad")}
    if kind == "polar":
        a = _angles(case, seed)
        cl = torch.cos(a) * res["cl_yx"][:, :1] + torch.sin(a) * res["cl_yx"][:, 1:]
        return {"cl": cl, "u_y": res["u_y"], "u_x": res["u_x"], "info": None}
    out = {q: res[q] for q in ("u", "cp", "cl", "cl_p", "cd_p")}
    out["info"] = None
    if kind == "ga":
        out["nodes"] = nodes
        out.update({q: None for q in ("ld", "cd", "cd_f", "theta", "cf", "sep")})
    elif kind != "solve":
        out.update(lam=res["lam"], grad=res["grad"])
    return out


def _spline(case, seed):
    """Nodes of the optimiser's first population: clamped uniform cubic B-splines
    of its genome, which a seeded generator draws uniformly within the bounds."""
    B, n = case["batch"], case["n_max"]
    cx = torch.as_tensor(default_control_x(), device=DEVICE)
    lo, hi = (torch.as_tensor(v, device=DEVICE) for v in _bounds())
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    P = len(cx)
    genome = lo + torch.rand(B, P, generator=gen, dtype=torch.float64, device=DEVICE) * (hi - lo)
    i = torch.arange(n, device=DEVICE, dtype=torch.float64)
    nu = (n + 1) // 2
    t = torch.where(i <= nu, 0.25 * (1 - torch.cos(math.pi * i / nu)),
                    0.5 + 0.25 * (1 - torch.cos(math.pi * (i - nu) / (n - nu))))
    knots = torch.cat([torch.zeros(3), torch.arange(P - 2) / (P - 3), torch.ones(3)]).double()
    knots[3:P + 1] = torch.arange(P - 2, dtype=torch.float64) / (P - 3)
    knots = knots.to(DEVICE)
    span = torch.clamp((t * (P - 3)).floor().long(), 0, P - 4) + 3
    N = torch.nn.functional.one_hot(span, P + 3).double()  # degree 0
    for d in range(1, 4):
        M = torch.zeros_like(N)
        for r in range(P + 3 - d):
            a, b = knots[r + d] - knots[r], knots[r + d + 1] - knots[r + 1]
            if a > 0:
                M[:, r] += (t - knots[r]) / a * N[:, r]
            if b > 0:
                M[:, r] += (knots[r + d + 1] - t) / b * N[:, r + 1]
        N = M
    N = N[:, :P]
    return torch.stack([(N @ cx)[None].expand(B, n), genome @ N.T], -1).reshape(B * n, 2)
