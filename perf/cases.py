"""Workloads whose speed is watched: what programs ask of this library, each
through its public entry points.

A "step" case is the time loop of a simulation: the state goes up, then `steps`
times the CFL time step and the full ADER-WENO-CT step, then the state comes
down.  A "gradient" case is one evaluation of the outer-shell objective and its
adjoint gradient through torch.autograd.  A "prism" case is the ADER-CG predictor
on triangular-prism zones.

States are device tensors made from the seed alone (density noise of 1 % and the
phase of the wave).  A FP32-bulk mesh computes the rates of change of the state in
32 bits (documented relative error 2e-5), so its results are handed on as 32-bit
tensors, which is all that they carry; the FP64 form's as 64-bit ones.
"""
import math

import torch

from paper_1905_02504_gb300 import autodiff, geomhd

CFL = 0.4
GAMMA = 5.0 / 3.0
PRISM_DT = 1e-3

# per order: nodes, time levels, Taylor terms, KKT inputs, face points of a zone,
# points per edge, nodes of a face, nodes of an edge, nonzeros of one D^alpha,
# zones of the central WENO stencil
HEX = {2: (8, 2, 3, 42, 24, 1, 4, 2, 16, 6), 3: (20, 3, 9, 60, 24, 2, 8, 3, 96, 26),
       4: (32, 4, 19, 108, 42, 3, 12, 4, 192, 32)}
# prism element: nodes and nonzeros of the three D^alpha
PRISM = {2: (6, 42), 3: (15, 247), 4: (26, 580)}


def _step(name, order, n, shells, fp32=False, problem="smooth", positivity=False, hlld=False, steps=1):
    return {"name": name, "kind": "step", "order": order, "subdiv": n, "shells": shells, "fp32": fp32,
            "problem": problem, "positivity": positivity, "hlld": hlld, "steps": steps}


def listed():
    return [
        # the smallest sensible run: one step on 162 zones, as a first check of an
        # installation makes it; launches and latency are all of it
        _step("first_step_p3", 3, 3, 3),
        # the coarse second-order run of ten steps on 3,072 zones
        _step("coarse_p2_10_steps", 2, 8, 8, steps=10),
        # second order as production runs use it for relaxation: many cheap zones
        _step("relax_p2_fp32", 2, 48, 96, fp32=True, steps=4),
        # the third-order blast wave in FP64, about 2e5 zones
        _step("blast_p3", 3, 24, 56, problem="blast", steps=1),
        # the same mesh in the reduced-precision form, smooth flow
        _step("smooth_p3_fp32", 3, 24, 56, fp32=True, steps=4),
        # the higher-fidelity face solver on a mesh of odd sizes
        _step("hlld_p3_odd_mesh", 3, 13, 37, problem="blast", hlld=True, steps=2),
        # fourth order in FP64, the headline form
        _step("smooth_p4", 4, 12, 128, steps=1),
        # fourth order in the reduced-precision form
        _step("smooth_p4_fp32", 4, 16, 96, fp32=True, steps=2),
        # the low-beta blast with the positivity scaling, a CFL reduction before every step
        _step("lowbeta_p4_fp32_positivity", 4, 12, 64, fp32=True, problem="lowbeta", positivity=True, steps=2),
        # one gradient of the outer-shell flux over a window of two steps
        {"name": "gradient_p3", "kind": "gradient", "order": 3, "subdiv": 16, "shells": 32, "steps": 2},
        # the predictor on prism zones of a geodesic mesh: fourth order ...
        {"name": "prism_p4", "kind": "prism", "order": 4, "zones": 262144},
        # ... and third order on a number of zones that fills no block evenly
        {"name": "prism_p3_odd", "kind": "prism", "order": 3, "zones": 100003},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["step", "gradient", "prism"], [10, 2, 2])[0]
    order = rng.choice([2, 3, 4])
    if kind == "prism":
        return {"kind": kind, "order": order, "zones": _log_int(rng, 500, 300000)}
    # columns are what a mesh costs to set up, shells are not
    n_max = {2: 40, 3: 20, 4: 11}[order]
    if kind == "gradient":
        return {"kind": kind, "order": order, "subdiv": _log_int(rng, 3, min(n_max, 12)),
                "shells": _log_int(rng, 4, 24), "steps": rng.choice([1, 2])}
    fp32 = rng.random() < 0.5
    problem = rng.choice(["smooth", "smooth", "blast"])
    c = _step("", order, _log_int(rng, 3, n_max), _log_int(rng, 4, 128 if fp32 else 72), fp32=fp32, problem=problem,
              positivity=problem == "blast", hlld=rng.random() < 0.25, steps=rng.choice([1, 2]))
    del c["name"]
    return c


# ------------------------------------------------------------------- inputs
def _magnetic(problem, x, wave):
    if problem == "smooth":
        k = 2.0 * math.pi
        return 0.1 * k * torch.stack([torch.cos(k * x[..., 1] + wave), torch.cos(k * x[..., 2] + wave),
                                      torch.cos(k * x[..., 0] + wave)], -1)
    return _uniform_b(problem, x).expand(x.shape)


def _uniform_b(problem, x):
    b = [0.0, 0.0, 10.0 / math.sqrt(4.0 * math.pi)] if problem == "blast" else \
        [math.sqrt(10.0), math.sqrt(10.0), 0.0]  # plasma beta 0.01 at p = 0.1
    return torch.tensor(b, dtype=x.dtype, device=x.device)


def _potential(problem, x, wave):
    if problem == "smooth":
        k = 2.0 * math.pi
        return 0.1 * torch.stack([torch.sin(k * x[..., 2] + wave), torch.sin(k * x[..., 0] + wave),
                                  torch.sin(k * x[..., 1] + wave)], -1)
    return 0.5 * torch.linalg.cross(_uniform_b(problem, x).expand(x.shape), x)


def _conserved(problem, x, wave):
    if problem == "smooth":
        rho = 1.0 + 0.1 * torch.sin(2.0 * math.pi * x.sum(-1) / math.sqrt(3.0) + wave)
        p = torch.ones_like(rho)
        v = torch.full_like(x, 0.5)
    else:
        rho = torch.ones_like(x[..., 0])
        r2 = x[..., 0] ** 2 + x[..., 1] ** 2 + (x[..., 2] - 1.5) ** 2
        p = torch.where(r2 < 0.01, 100.0, 0.1).to(x.dtype)
        v = torch.zeros_like(x)
    b = _magnetic(problem, x, wave)
    e = p / (GAMMA - 1.0) + 0.5 * rho * (v * v).sum(-1) + 0.5 * (b * b).sum(-1)
    return torch.cat([rho[..., None], rho[..., None] * v, e[..., None], b], -1)


def _initial_state(mesh, problem, seed):
    """Zone averages (8, Z) by cubature and face fluxes (F,) by edge circulation, on the device."""
    gen = torch.Generator().manual_seed(seed)
    wave = float(torch.rand((), generator=gen)) * 2.0 * math.pi
    noise = torch.rand(mesh.Z, generator=gen, dtype=torch.float64).mul_(2.0).sub_(1.0).cuda()
    pts, w = geomhd.geo_zone_cubature(mesh.h, 2)
    w = torch.from_numpy(w).cuda()
    U = (_conserved(problem, torch.from_numpy(pts).cuda(), wave) * w[..., None]).sum(1) / w.sum(1, keepdim=True)
    U = U.t().contiguous()
    fac = 1.0 + 0.01 * noise
    kinetic = 0.5 * (U[1:4] ** 2).sum(0) / U[0]
    U[4] += kinetic * (fac - 1.0)
    U[:4] *= fac
    pts, tw = geomhd.geo_edge_quadrature(mesh.h, 3)
    circ = (_potential(problem, torch.from_numpy(pts).cuda(), wave) * torch.from_numpy(tw).cuda()).sum((1, 2))
    phi = geomhd.geo_phi_from_edge_circulation(mesh.h, circ.cpu().numpy())
    return U, torch.from_numpy(phi).cuda()


def _prism_inputs(order, zones, seed, device):
    """Seeded affine prisms in a 1-2 shell with a smooth state and 1 % noise at the nodes."""
    gen = torch.Generator(device=device).manual_seed(seed)
    f64 = {"dtype": torch.float64, "device": device}
    xi = torch.from_numpy(geomhd.geo_prism_nodes(order)).to(device)
    n = len(xi)
    cen = torch.randn(3, zones, generator=gen, **f64)
    cen *= (1.0 + torch.rand(1, zones, generator=gen, **f64)) / cen.norm(dim=0, keepdim=True)
    a = 0.02 * (torch.eye(3, **f64)[:, :, None] + 0.1 * torch.randn(3, 3, zones, generator=gen, **f64))
    X = (cen[:, None, :] + torch.einsum("dez,ne->dnz", a, xi)).contiguous()
    U = torch.empty(8, n, zones, **f64)
    U[0] = 1.0 + 0.01 * (2.0 * torch.rand(n, zones, generator=gen, **f64) - 1.0)
    for k, (v, b) in enumerate(((0.3, 0.4), (-0.2, -0.3), (0.1, 0.2))):
        U[1 + k] = U[0] * v
        U[5 + k] = b + 0.05 * X[(k + 1) % 3]
    U[4] = 0.8 / (GAMMA - 1.0) + 0.5 * (U[1:4] ** 2).sum(0) / U[0] + 0.5 * (U[5:8] ** 2).sum(0)
    return X, U


def prepare(case, seed):
    if case["kind"] == "prism":
        X, U = _prism_inputs(case["order"], case["zones"], seed, "cuda")
        out = torch.empty((case["order"],) + tuple(U.shape), dtype=torch.float64, device="cuda")
        return {"case": case, "X": X, "U": U, "out": out}
    prec = geomhd.GEO_FP32_BULK if case.get("fp32") else geomhd.GEO_FP64
    mesh = geomhd.Mesh(case["subdiv"], case["shells"], 1.0, 2.0, case["order"], prec)
    if case.get("positivity"):
        geomhd.geo_set_positivity(mesh.h, 1)
    if case.get("hlld"):
        geomhd.geo_set_riemann(mesh.h, geomhd.GEO_RIEMANN_HLLD)
    U, phi = _initial_state(mesh, case.get("problem", "smooth"), seed)
    mesh.upload(U, phi)
    return {"case": case, "mesh": mesh, "U": U, "phi": phi, "U1": torch.empty_like(U), "phi1": torch.empty_like(phi),
            "dt": mesh.cfl_dt(CFL)}


# ------------------------------------------------------------------- one pass
def run(state):
    case = state["case"]
    if case["kind"] == "prism":
        geomhd.geo_prism_predictor(case["order"], state["X"], state["U"], PRISM_DT, GAMMA, state["out"])
        return state["out"]
    mesh = state["mesh"]
    if case["kind"] == "gradient":
        U = state["U"].detach().requires_grad_(True)
        phi = state["phi"].detach().requires_grad_(True)
        U1, phi1 = autodiff.step_window(mesh, U, phi, state["dt"], case["steps"])
        J = autodiff.outer_br2(mesh, phi1)
        J.backward()
        return {"U": U1.detach(), "phi": phi1.detach(), "J": J.detach(), "gU": U.grad, "gphi": phi.grad}
    mesh.upload(state["U"], state["phi"])
    for _ in range(case["steps"]):
        mesh.step(mesh.cfl_dt(CFL))
    geomhd.geo_state_download(mesh.h, state["U1"], state["phi1"])
    if case["fp32"]:
        return {"U": state["U1"].float(), "phi": state["phi1"].float()}
    return {"U": state["U1"], "phi": state["phi1"]}


# ------------------------------------------------------------------- its work
def _prim_flux(normals):
    """One recovery of the primitive state and its flux along some normals."""
    return 25.0 + 45.0 * normals


def work(case):
    """State in, state out; the scheme's own arithmetic (an FMA counts two)."""
    p = case["order"]
    if case["kind"] == "prism":
        n, nnz = PRISM[p]
        z, m = case["zones"], p
        level = n * _prim_flux(4) + 16.0 * nnz
        return {"bytes": 8.0 * z * n * (3 + 8 + 8 * m),
                "flops": z * (12.0 * nnz + 32 * n + (1 + (p - 1) * (m - 1)) * level + p * (m - 1) * 16.0 * m * n)}
    c, nr = 6 * case["subdiv"] ** 2, case["shells"]
    z = c * nr
    f = c * (nr + 1) + 2 * c * nr
    e = (c + 2) * nr + 2 * c * (nr + 1)
    n, m, nc1, nbin, nqt, ns, nfn, nen, nnz, st = HEX[p]
    weno = 8 * (st * (1 + 2 * nc1) + 2 * nc1 * nc1 + 248 + 144 + 4 * nc1)
    bperp = nqt / 6.0 * (12 * nc1 + 18)
    level = n * _prim_flux(4) + 48.0 * nnz
    ader = 2.0 * (3 + 3 * n) * nbin + 10.0 * n * nc1 + (1 + (p - 1) * (m - 1)) * level + p * (m - 1) * 16.0 * n * m + \
        (m - 1) * (nqt * (16 * nfn + 8) + 12 * ns * (16 * nen + 8))
    face = (m - 1) * nqt / 6.0 * 156.0
    edge = (m - 1) * ns * 508.0
    forward = z * (weno + ader + 104.0) + f * (bperp + face + 4.0) + e * edge
    state = 8.0 * (8 * z + f)
    k = case["steps"]
    if case["kind"] == "gradient":
        # the reverse of a step: its stages once more, and the transpose of each
        return {"bytes": 4.0 * state, "flops": k * 4.0 * forward}
    return {"bytes": 2.0 * state, "flops": k * forward}


# ------------------------------------------------------------------- in 64 bits
def _prism_basis(order, xi):
    """D [3][N][N]: derivatives at the nodes of the Lagrange basis on the prism's monomials."""
    lateral = [(a, d - a) for d in range(order) for a in range(d, -1, -1)]
    mono = [(a, b, c) for a, b in lateral for c in range(2)]
    mono += [(0, 0, c) for c in range(2, order)] + [(1, 0, c) for c in range(2, order)] + \
            [(0, 1, c) for c in range(2, order)]
    V = torch.stack([xi[:, 0] ** a * xi[:, 1] ** b * xi[:, 2] ** c for a, b, c in mono], 1)
    coef = torch.linalg.inv(V)                       # [monomial][node]
    D = []
    for ax in range(3):
        cols = []
        for ex in mono:
            if ex[ax] == 0:
                cols.append(torch.zeros_like(xi[:, 0]))
                continue
            q = list(ex)
            q[ax] -= 1
            cols.append(ex[ax] * xi[:, 0] ** q[0] * xi[:, 1] ** q[1] * xi[:, 2] ** q[2])
        D.append(torch.stack(cols, 1) @ coef)
    return torch.stack(D)


def _time_matrix(order):
    """R of U_k = U_1 - sum_m R_km dF_m: integrals from 0 to tau_k of the Lagrange
    basis in time on tau = 0 and the order - 1 Gauss points of [0, 1], projected as
    the continuous Galerkin form with test functions of the later levels."""
    import numpy as np
    x, _ = np.polynomial.legendre.leggauss(order - 1)
    tau = np.concatenate([[0.0], 0.5 * (x + 1.0)])
    gx, gw = np.polynomial.legendre.leggauss(2 * order)
    gx, gw = 0.5 * (gx + 1.0), 0.5 * gw
    m = len(tau)
    phi, dphi = np.empty((m, len(gx))), np.empty((m, len(gx)))
    for i in range(m):
        pol = np.poly1d(np.delete(tau, i), r=True) / np.prod(tau[i] - np.delete(tau, i))
        phi[i], dphi[i] = pol(gx), pol.deriv()(gx)
    K = np.einsum("kg,mg,g->km", phi[1:], dphi, gw)
    Mm = np.einsum("kg,mg,g->km", phi[1:], phi, gw)
    R = np.zeros((m, m))
    R[1:] = np.linalg.solve(K[:, 1:], Mm)
    return R


def _flux(u, s):
    """F(u).s of ideal MHD: u [8][...], s [3][...]."""
    rho, mom, e, b = u[0], u[1:4], u[4], u[5:8]
    v = mom / rho
    b2 = (b * b).sum(0)
    pt = (GAMMA - 1.0) * (e - 0.5 * (mom * v).sum(0) - 0.5 * b2) + 0.5 * b2
    vn, bn = (v * s).sum(0), (b * s).sum(0)
    return torch.cat([(rho * vn)[None], mom * vn + pt * s - b * bn,
                      ((e + pt) * vn - bn * (v * b).sum(0))[None], b * vn - v * bn])


def _exact_prism(case, seed):
    order = case["order"]
    X, U = _prism_inputs(order, case["zones"], seed, "cuda")
    D = _prism_basis(order, torch.from_numpy(geomhd.geo_prism_nodes(order)).cuda())
    R = _time_matrix(order)
    h = torch.einsum("aij,djz->adiz", D, X)
    S = torch.stack([torch.linalg.cross(h[1], h[2], dim=0), torch.linalg.cross(h[2], h[0], dim=0),
                     torch.linalg.cross(h[0], h[1], dim=0)])                       # [a][d][i][z]
    J = (S[2] * h[2]).sum(0)
    g = torch.einsum("aij,adjz->diz", D, S)

    def difference(W):
        u = W / J
        d = -_flux(u, g)
        for a in range(3):
            d += torch.einsum("ij,vjz->viz", D[a], _flux(u, S[a]))
        return PRISM_DT * d

    W = [J * U for _ in range(order)]
    for _ in range(order):
        dF = [difference(w) for w in W]
        W = [W[0]] + [W[0] - sum(float(R[k, q]) * dF[q] for q in range(order)) for k in range(1, order)]
    return torch.stack(W)


def exact(case, seed):
    """The prism predictor written out in 64 bits; a whole step has no short form
    of its own (its mesh tables alone are a program)."""
    return _exact_prism(case, seed) if case["kind"] == "prism" else None
