"""The calls a user of this library makes, as measurable cases.

Each case is one call (or the short sequence of calls that belongs together)
through the public binding, on the flows this repository is used for: lid-driven
cavities, the sphere at Mach 0.3, the viscous sphere, hexahedral grids, batches of
uneven meshes. listed() names them, draw() gives more of the same ranges, exact()
restates the Jacobian block's outputs in plain numpy.
"""
import math
from functools import lru_cache

import numpy as np
import torch

import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I

CAVITY = dict(mesh="cavity", Mach=0.15, Re=100.0, Pr=0.72, krylov=10, precision="fp64")
SPHERE = dict(mesh="sphere", Mach=0.3, Re=0.0, Pr=1.0, krylov=20, precision="fp64")


def listed():
    return [
        # the smallest solve in use: one implicit step of the 3,072-tetrahedron cavity that
        # converges to 1e-8 in about 1,950 such steps; launches and latency count
        dict(CAVITY, name="cavity_3k_step_hweno", kind="step", n=8, scheme="hweno"),
        # a small residual call (an outer program that drives its own time stepping), odd size
        dict(CAVITY, name="cavity_8k_residual_weno", kind="residual", n=11, scheme="weno"),
        # the paper's efficiency case: 48,000 tetrahedra clustered at the walls, Re 1000;
        # the whole steady loop with its residual test on the host, five steps of it
        dict(CAVITY, name="cavity_48k_solve_weno", kind="solve", n=20, h_min=0.025, Re=1000.0, scheme="weno", steps=5),
        # the compact residual with its gradient update on the same mesh
        dict(CAVITY, name="cavity_48k_residual_hweno", kind="residual", n=20, h_min=0.025, Re=1000.0, scheme="hweno"),
        # A itself, for programs with a Krylov method of their own: local time step, blocks,
        # product and preconditioner; patches of 9 x 9, 17 layers: nothing is a multiple of a block
        dict(SPHERE, name="sphere_50k_jacobian", kind="jacobian", n=9, layers=17, scheme="weno"),
        # an ordinary inviscid step, GMRES(20) x 3
        dict(SPHERE, name="sphere_124k_step_weno", kind="step", n=12, layers=24, scheme="weno"),
        # the viscous sphere, compact scheme, FP32 Krylov vectors (mixed precision)
        dict(SPHERE, name="sphere_295k_step_hweno_mixed", kind="step", n=16, layers=32, Mach=0.2535, Re=118.0, Pr=0.72,
             krylov=10, scheme="hweno", precision="mixed"),
        # hexahedra: the stand-in for the paper's 190,464-cell viscous-sphere grid, one step
        dict(SPHERE, name="hex_sphere_190k_step_weno", kind="step", mesh="hex_sphere", n=32, layers=31, Mach=0.2535,
             Re=118.0, Pr=0.72, krylov=10, scheme="weno"),
        # hexahedra with tilted planar faces, the compact residual, odd size
        dict(SPHERE, name="hex_box_36k_residual_hweno", kind="residual", mesh="hex_box", n=33, scheme="hweno"),
        # a batch of six meshes of 20k to 100k cells, cavities and viscous spheres mixed,
        # compact scheme, FP32 Krylov vectors: one step of all of them
        dict(name="batch_6_step_hweno_mixed", kind="batch", problems=6, n_min=20000, n_max=100000, krylov=10,
             scheme="hweno", precision="mixed"),
        # the largest residual call and the headline workload, one step: 2,359,296 tetrahedra
        dict(SPHERE, name="sphere_995k_residual_weno", kind="residual", n=24, layers=48, scheme="weno"),
        dict(SPHERE, name="sphere_2359k_step_weno", kind="step", n=32, layers=64, scheme="weno"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "residual", "residual", "jacobian", "solve"])
    mesh = rng.choice(["cavity", "sphere", "sphere", "hex_cavity", "hex_box", "hex_sphere"])
    if kind == "jacobian":
        mesh = rng.choice(["cavity", "sphere"])
    cells = math.exp(rng.uniform(math.log(500.0), math.log(400000.0 if kind in ("residual", "step") else 100000.0)))
    scheme = rng.choice(["weno", "hweno"])
    c = dict(kind=kind, mesh=mesh, scheme=scheme, Mach=round(rng.uniform(0.1, 0.5), 3), Re=0.0, Pr=1.0,
             krylov=rng.randint(8, 20), precision=rng.choice(["fp64", "fp64", "mixed"]) if kind == "step" else "fp64")
    if mesh in ("cavity", "hex_cavity") or rng.random() < 0.4:
        c.update(Re=round(math.exp(rng.uniform(math.log(50.0), math.log(1000.0))), 1), Pr=0.72)
    per = {"cavity": 6.0, "hex_cavity": 1.0, "hex_box": 1.0, "sphere": 36.0, "hex_sphere": 6.0}[mesh]
    if mesh in ("sphere", "hex_sphere"):
        c["n"] = max(3, round((cells / (2.0 * per)) ** (1.0 / 3.0)))
        c["layers"] = max(4, round(cells / (per * c["n"] ** 2)) + rng.randint(-1, 1))
    else:
        c["n"] = max(4, round((cells / per) ** (1.0 / 3.0)))
    if kind == "solve":
        c["steps"] = rng.randint(2, 6)
    return c


@lru_cache(maxsize=16)
def _mesh(mesh, n, layers, h_min, viscous):
    """The mesh a user brings (host arrays); kept for the other states of the same case."""
    wall = I.BC_NOSLIP_ADIA if viscous else I.BC_SLIP
    if mesh == "cavity":
        return I.cavity_mesh(n, h_min=h_min)
    if mesh == "sphere":
        return I.sphere_mesh(n, layers, stretch=I.sphere_stretch(layers), wall_tag=wall)
    if mesh == "hex_cavity":
        return I.hex_cavity_mesh(n)
    if mesh == "hex_box":
        return I.hex_tilted_box_mesh(n)
    return I.hex_sphere_mesh(n, layers, stretch=I.sphere_stretch(layers), wall_tag=wall)


def _mesh_of(case):
    return _mesh(case["mesh"], case["n"], case.get("layers", 0), case.get("h_min"), case["Re"] > 0.0)


@lru_cache(maxsize=4)
def _problems(count, n_min, n_max):
    return I.batch_problems(count, n_min, n_max)


def _conditions(case):
    if case["mesh"] in ("cavity", "hex_cavity"):
        return I.cavity_conditions(case["Mach"], case["Re"])
    return I.sphere_conditions(case["Mach"], case["Re"] if case["Re"] > 0.0 else None)


def _params(case, cond):
    return H.hgks_default_params(**{**cond, "scheme": H.HGKS_HWENO if case["scheme"] == "hweno" else H.HGKS_WENO,
                                    "precision": H.HGKS_MIXED if case.get("precision") == "mixed" else H.HGKS_FP64,
                                    "Pr": case["Pr"] if cond["viscous"] else 1.0, "krylov_dim": case["krylov"],
                                    "restarts": 3, "jacobi_sweeps": 2, "cfl": 10.0})


def _state(mesh, cond, seed, external):
    """A smooth disturbed flow about the initial one (an iterate of a solve): caller order."""
    u = cond["u_inf"]
    base = (cond["rho_inf"], u[0] + 0.05, u[1] + 0.03, u[2] - 0.02, cond["p_inf"])
    return I.smooth_state(mesh, seed=seed, amp=0.02, base=base, wavenumber=0.5 if external else 2.0)


def prepare(case, seed):
    s = {"case": case}
    compact = case["scheme"] == "hweno"
    if case["kind"] == "batch":
        probs = _problems(case["problems"], case["n_min"], case["n_max"])
        meshes = [H.hgks_mesh_create(p["mesh"], scheme_mask=2 if compact else 1) for p in probs]
        s["batch"] = H.hgks_batch_create(meshes, [_params(dict(case, Pr=0.72), p["cond"]) for p in probs])
        s["states"] = []
        for k, (p, h) in enumerate(zip(probs, meshes)):
            Q, G = _state(p["mesh"], p["cond"], seed + 1000 * k, p["kind"] == "sphere")
            Qd, Gd = h.to_internal(Q), h.to_internal(G)
            s["states"].append((Qd, Gd, torch.empty_like(Qd), torch.empty_like(Gd)))
        return s
    mesh, cond = _mesh_of(case), _conditions(case)
    s["mesh"] = H.hgks_mesh_create(mesh, scheme_mask=2 if compact else 1)
    s["params"] = _params(case, cond)
    Q, G = _state(mesh, cond, seed, "sphere" in case["mesh"])
    s["Q0"] = s["mesh"].to_internal(Q)
    s["G0"] = s["mesh"].to_internal(G) if compact else None
    n = s["Q0"].shape[1]
    if case["kind"] == "residual":
        s["R"], s["Gn"] = torch.empty_like(s["Q0"]), torch.empty_like(s["G0"]) if compact else None
    elif case["kind"] == "jacobian":
        g = torch.Generator().manual_seed(seed)
        s["x"], s["b"] = (torch.randn(5, n, generator=g, dtype=torch.float64).cuda() for _ in range(2))
        new = lambda rows: torch.empty(rows, n, dtype=torch.float64, device="cuda")  # noqa: E731
        s["dt"], s["diag"], s["off"], s["y"], s["z"] = new(1), new(25), new(25 * s["mesh"].faces_per_cell), new(5), new(5)
    else:
        s["Q"], s["G"] = torch.empty_like(s["Q0"]), torch.empty_like(s["G0"]) if compact else None
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "batch":
        compact = s["case"]["scheme"] == "hweno"
        for k, (Q0, G0, _, _) in enumerate(s["states"]):
            H.hgks_batch_set_state(s["batch"], k, Q0, G0 if compact else None)
        info = H.hgks_batch_gmres_step(s["batch"])
        for k, (_, _, Q, G) in enumerate(s["states"]):
            H.hgks_batch_get_state(s["batch"], k, Q, G if compact else None)
        return {"Q": [t[2] for t in s["states"]], "G": [t[3] for t in s["states"]] if compact else None,
                "res": [i.res_l1 for i in info], "nonphysical": [i.nonphysical for i in info]}
    m, p = s["mesh"], s["params"]
    if kind == "residual":
        H.hgks_residual(m, p, s["Q0"], s["G0"], s["R"], s["Gn"])
        return {"R": s["R"], "G": s["Gn"]}
    if kind == "jacobian":
        H.hgks_local_dt(m, p, s["Q0"], s["dt"])
        H.hgks_assemble(m, p, s["Q0"], s["dt"], s["diag"], s["off"])
        H.hgks_apply_jacobian(m, s["x"], s["y"])
        H.hgks_precondition(m, 2, s["b"], s["z"])
        return {"dt": s["dt"], "diag": s["diag"], "off": s["off"], "y": s["y"], "z": s["z"]}
    s["Q"].copy_(s["Q0"])                       # the step works in place: start from the same iterate
    if s["G"] is not None:
        s["G"].copy_(s["G0"])
    if kind == "step":
        i = H.hgks_gmres_step(m, p, s["Q"], s["G"])
        return {"Q": s["Q"], "G": s["G"], "res": i.res_l1, "lin": list(i.lin_res), "nonphysical": i.nonphysical}
    info, hist, _ = H.hgks_solve_steady(m, p, s["Q"], s["G"], drop_tol=1e-12, max_steps=s["case"]["steps"])
    return {"Q": s["Q"], "G": s["G"], "history": hist, "steps": info.steps}


def _size(case):
    """Cells, faces per cell and Gauss points per face."""
    n, L = case["n"], case.get("layers", 0)
    return {"cavity": (6 * n ** 3, 4, 3), "hex_cavity": (n ** 3, 6, 4), "hex_box": (n ** 3, 6, 4),
            "sphere": (36 * n * n * L, 4, 3), "hex_sphere": (6 * n * n * L, 6, 4)}[case["mesh"]]


def work(case):
    """Bytes: the state and the mesh's own data (fits, faces, neighbours) once, the outputs
    once. Flops: the formulas as the method states them, per cell, face and Gauss point; per
    Krylov vector three products with the off-diagonal blocks and modified Gram-Schmidt."""
    if case["kind"] == "batch":
        N, nf, ng = sum(p["n_cells"] for p in _problems(case["problems"], case["n_min"], case["n_max"])), 4, 3
    else:
        N, nf, ng = _size(case)
    compact = case["scheme"] == "hweno"
    fit = (9 * (nf + 3 * (1 + nf)) + nf * 21) if compact else (9 * 12 + 72)      # doubles of the least-squares maps
    mesh_b = 8.0 * (fit + 3 * nf * ng + 8 + 12 * nf / 2) + 8.0 * nf
    state = 20 if compact else 5
    product = 2.0 * 17 * nf
    if case["kind"] == "jacobian":
        return {"bytes": N * (8.0 * (5 + 12 * nf / 2 + 1 + 25 + 25 * nf + 4 * 5) + 8.0 * nf), "flops": N * (60.0 * nf + 3 * product)}
    residual_f = 10.0 * fit + nf * (210.0 * 5 + 250 * 5) + nf / 2 * ng * (1500.0 if compact else 1200.0)
    if case["kind"] == "residual":
        return {"bytes": N * (mesh_b + 16.0 * state), "flops": N * residual_f}
    k = case["krylov"]
    step_f = 3 * k * (3 * product + 20.0 * (k + 1) / 2)
    if case.get("precision") == "mixed":
        step_f = 0.0            # FP32, far below the FP64 part in time
    steps = case.get("steps", 1)
    return {"bytes": N * (mesh_b + 16.0 * state) * steps, "flops": N * (residual_f + step_f) * steps}


# ---- the Jacobian block in plain numpy -------------------------------------------------
# Only this block has a short restatement. The residual's (boundary-grown least-squares
# stencils, nonlinear weights, the gas-kinetic moments) is an independent solver of a
# thousand lines, and a step contains it: their float64 outputs have no value here.

def _spread(v):
    v = v.astype(np.uint64) & np.uint64(0x1FFFFF)
    for sh, mask in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                     (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        v = (v | (v << np.uint64(sh))) & np.uint64(mask)
    return v


def exact(case, seed):
    if case["kind"] != "jacobian" or _size(case)[0] > 200000:
        return None
    mesh, cond = _mesh_of(case), _conditions(case)
    N, g, cfl = len(mesh.tet4), cond["gamma"], 10.0
    X = mesh.xyz[mesh.tet4]
    cen = 0.25 * (X[:, 0] + X[:, 1] + X[:, 2] + X[:, 3])
    lo, ext = cen.min(0), (cen.max(0) - cen.min(0)).max()
    q = np.minimum(2097151.0, np.floor((cen - lo) / ext * 2097151.0))
    order = np.argsort(_spread(q[:, 0]) | _spread(q[:, 1]) << np.uint64(1) | _spread(q[:, 2]) << np.uint64(2), kind="stable")
    tet, X, cen = mesh.tet4[order], X[order], cen[order]          # cells along the space-filling curve
    Q = _state(mesh, cond, seed, "sphere" in case["mesh"])[0][order]
    r = torch.Generator().manual_seed(seed)
    x, b = (torch.randn(5, N, generator=r, dtype=torch.float64).numpy() for _ in range(2))
    vol = np.abs(np.einsum("ij,ij->i", X[:, 1] - X[:, 0], np.cross(X[:, 2] - X[:, 0], X[:, 3] - X[:, 0]))) / 6.0
    # local face p lies opposite vertex p; the neighbour is the other cell with the same vertices
    three = [[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]]
    keys = np.sort(np.stack([tet[:, f] for f in three], 1).reshape(-1, 3), axis=1)
    at = np.lexsort(keys.T[::-1])
    same = np.all(keys[at[1:]] == keys[at[:-1]], axis=1)
    nb = -np.ones(4 * N, dtype=np.int64)
    nb[at[:-1][same]], nb[at[1:][same]] = at[1:][same] // 4, at[:-1][same] // 4
    nb = nb.reshape(N, 4)
    nS = np.zeros((N, 4, 3))
    dist = np.zeros((N, 4))
    for p, f in enumerate(three):
        a = 0.5 * np.cross(X[:, f[1]] - X[:, f[0]], X[:, f[2]] - X[:, f[0]])
        a *= np.sign(np.einsum("ij,ij->i", a, X[:, f[0]] - X[:, p]))[:, None]
        nS[:, p] = a
        d = np.linalg.norm(cen[nb[:, p]] - cen, axis=1)
        n = a / np.linalg.norm(a, axis=1)[:, None]
        dist[:, p] = np.where(nb[:, p] >= 0, d, 2.0 * np.abs(np.einsum("ij,ij->i", n, X[:, f[0]] - cen)))
    S = np.linalg.norm(nS, axis=2)
    n = nS / S[:, :, None]
    rho, u = Q[:, 0], Q[:, 1:4] / Q[:, :1]
    pr = (g - 1) * (Q[:, 4] - 0.5 * rho * (u * u).sum(1))
    a = np.sqrt(g * pr / rho)
    nu = 2 * g * cond["mu"] / (case["Pr"] * rho * np.cbrt(vol)) if cond["viscous"] else np.zeros(N)
    dt = cfl * vol / (S * (np.abs(np.einsum("ipk,ik->ip", n, u)) + (a + nu)[:, None])).sum(1)
    j = np.where(nb >= 0, nb, np.arange(N)[:, None])
    Qf = 0.5 * (Q[:, None] + Q[j])
    uf = Qf[..., 1:4] / Qf[..., :1]
    pf = (g - 1) * (Qf[..., 4] - 0.5 * Qf[..., 0] * (uf * uf).sum(-1))
    lam = np.abs((uf * n).sum(-1)) + np.sqrt(g * pf / Qf[..., 0])
    if cond["viscous"]:
        lam = lam + 2 * cond["mu"] / (Qf[..., 0] * dist)
    d = vol / dt + (0.5 * lam * S).sum(1)
    E, phi = Q[:, 4] / rho, 0.5 * (g - 1) * (u * u).sum(1)
    un, Hj, off = np.einsum("ipk,ipk->ip", n, u[j]), (g * E - phi)[j], np.zeros((N, 4, 5, 5))
    off[..., 0, 1:4] = n
    off[..., 1:4, 0] = phi[j][..., None] * n - u[j] * un[..., None]
    off[..., 1:4, 1:4] = u[j][..., :, None] * n[..., None, :] - (g - 1) * n[..., :, None] * u[j][..., None, :]
    off[..., 1:4, 4] = (g - 1) * n
    off[..., 4, 0] = (phi[j] - Hj) * un
    off[..., 4, 1:4] = Hj[..., None] * n - (g - 1) * u[j] * un[..., None]
    off[..., 4, 4] = g * un
    for k in range(1, 4):
        off[..., k, k] += un
    off -= lam[..., None, None] * np.eye(5)
    off *= (0.5 * S * (nb >= 0))[..., None, None]

    def product(v):                                                # sum over the faces of the off-diagonal blocks
        return np.einsum("iprc,cip->ri", off, v[:, j])

    z = b / d
    for _ in range(2):
        z = (b - product(z)) / d
    diag = np.zeros((25, N))
    diag[::6] = d
    return {"dt": dt[None], "diag": diag, "off": off.reshape(N, 100).T.copy(), "y": d * x + product(x), "z": z}
