"""Both forms of the FP64 GMRES, one cooperative launch and separate launches, on the same
small meshes against the oracle: both cell kinds, two restart cycles, none to three Jacobi sweeps,
one to 64 Krylov vectors (a whole block of basis vectors followed by others; the upper half of a
warp from 33 on). The size limit is lowered inside the handle for the separate launches, which
otherwise belong to meshes above it. FP32 Krylov vectors and batches for the larger sizes.

Tolerances: the update's relative L2 error as every step is held to the oracle, 1e-9 (FP64: both
round differently, amplified by the conditioning of A, about 1e6 at CFL 10) and 1e-4 (FP32
vectors); a batch against the mesh alone 1e-9 and 2e-4 (both sides carry the error).
"""
import numpy as np
import pytest

import handle_shim
import oracle as O
import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MESHES = {
    "tet": lambda: (I.cavity_mesh(3), I.cavity_conditions(0.15, 100.0)),                                  # 162 cells
    "hex": lambda: (I.hex_cavity_mesh(5), I.cavity_conditions(0.15, 100.0)),                              # 125 cells
    "sphere": lambda: (I.sphere_mesh(4, 5, stretch=1.3), I.sphere_conditions(0.3)),                       # 2,880 cells
}
_cache = {}


@pytest.fixture(scope="module")
def shim(cuda, tmp_path_factory):
    return handle_shim.load(tmp_path_factory.mktemp("shim"))


def oracle_step(name, scheme, kw):
    key = (name, scheme, tuple(sorted(kw.items())))
    if key not in _cache:
        if name not in _cache:
            m, cond = MESHES[name]()
            u = cond["u_inf"]
            base = (cond["rho_inf"], u[0] + 0.05, u[1] + 0.03, u[2] - 0.02, cond["p_inf"])
            _cache[name] = (m, cond, O.OracleMesh(m), I.smooth_state(m, amp=0.03, base=base))
        m, cond, om, (Q, G) = _cache[name]
        p = O.make_params(scheme=scheme, Pr=0.72 if cond["viscous"] else 1.0, **cond, **kw)
        Qo, _, res, lin = om.gmres_step(p, Q, G if scheme else None)
        _cache[key] = (Qo - Q, res)
    return _cache[name] + _cache[key]


def step(shim, name, separate, tol, scheme=0, precision=0, **kw):
    import torch
    m, cond, _, (Q, G), ref, res = oracle_step(name, scheme, kw)
    hm = H.hgks_mesh_create(m, scheme_mask=1 << scheme)
    if separate:
        shim.hx_grid_cells(hm.handle, 0)
    p = H.hgks_default_params(scheme=scheme, Pr=0.72 if cond["viscous"] else 1.0, precision=precision, **cond, **kw)
    Qd, Gd = hm.to_internal(Q), hm.to_internal(G) if scheme else None
    dQ = torch.empty_like(Qd)
    H.hgks_launch_count(reset=True)
    info = H.hgks_gmres_step(hm, p, Qd, Gd, dQ)
    launches = H.hgks_launch_count()                     # residual, assembly, update: under a dozen
    assert launches > p.restarts * (4 + 3 * p.krylov_dim) if separate or precision else launches < 12, launches
    err = np.linalg.norm(hm.to_caller(dQ) - ref) / np.linalg.norm(ref)
    assert err < tol, err
    assert abs(info.res_l1 - res) <= 1e-11 * abs(res)


FORMS = pytest.mark.parametrize("separate", [False, True], ids=["one-launch", "separate"])


@FORMS
@pytest.mark.parametrize("name", ["tet", "hex"])
@pytest.mark.parametrize("k,sweeps", [(1, 2), (3, 0), (4, 1), (5, 3), (8, 2), (9, 1), (12, 3), (13, 0), (17, 2)])
def test_sizes_and_sweeps(shim, name, separate, k, sweeps):
    step(shim, name, separate, 1e-9, krylov_dim=k, restarts=2, jacobi_sweeps=sweeps)


@FORMS
@pytest.mark.parametrize("name,scheme,restarts", [("sphere", 0, 3), ("sphere", 1, 2), ("hex", 1, 3)])
def test_schemes_and_cycles(shim, name, separate, scheme, restarts):
    step(shim, name, separate, 1e-9, scheme=scheme, krylov_dim=10, restarts=restarts, jacobi_sweeps=2)


@FORMS
@pytest.mark.parametrize("name", ["sphere", "hex"])
@pytest.mark.parametrize("k", [32, 33, 40, 64])
def test_many_vectors(shim, name, separate, k):
    step(shim, name, separate, 1e-9, krylov_dim=k, restarts=1, jacobi_sweeps=1)


@pytest.mark.parametrize("name", ["sphere", "hex"])
@pytest.mark.parametrize("k", [33, 40, 64])
def test_many_vectors_fp32(shim, name, k):
    step(shim, name, False, 1e-4, precision=1, krylov_dim=k, restarts=1, jacobi_sweeps=1)


@pytest.mark.parametrize("precision,tol", [(0, 1e-9), (1, 2e-4)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("k", [33, 40, 64])
def test_many_vectors_in_a_batch(cuda, precision, tol, k):
    import torch
    m, cond = MESHES["sphere"]()
    Q, _ = I.smooth_state(m, amp=0.03, base=(1.0, 0.35, 0.03, -0.02, cond["p_inf"]))
    hm = H.hgks_mesh_create(m, scheme_mask=1)
    p = H.hgks_default_params(scheme=0, precision=precision, krylov_dim=k, restarts=1, **cond)
    Q0 = hm.to_internal(Q)
    Qs, Qb = Q0.clone(), torch.empty_like(Q0)
    H.hgks_gmres_step(hm, p, Qs)
    b = H.hgks_batch_create([hm, hm], [p, p])
    for s in range(2):
        H.hgks_batch_set_state(b, s, Q0)
    H.hgks_batch_gmres_step(b)
    for s in range(2):
        H.hgks_batch_get_state(b, s, Q=Qb)
        torch.cuda.synchronize()
        assert (torch.linalg.norm(Qb - Qs) / torch.linalg.norm(Qs - Q0)).item() <= tol


def test_a_captured_step_goes_with_its_basis(shim):
    """A call that needs more Krylov vectors moves the basis: the captured step, which holds its
    address, is dropped at once and captured anew by the next step."""
    m, cond = MESHES["tet"]()
    hm = H.hgks_mesh_create(m, scheme_mask=1)
    Q = hm.to_internal(I.smooth_state(m, amp=0.03, base=(1.0, 0.1, 0.05, -0.03, cond["p_inf"]))[0])
    dt = Q.new_empty(1, Q.shape[1])
    p = {k: H.hgks_default_params(Pr=0.72, krylov_dim=k, **cond) for k in (4, 12)}
    assert not shim.hx_captured(hm.handle)
    H.hgks_gmres_step(hm, p[4], Q.clone())
    assert shim.hx_captured(hm.handle)
    H.hgks_local_dt(hm, p[4], Q, dt)
    H.hgks_assemble(hm, p[4], Q, dt)
    assert shim.hx_captured(hm.handle)          # the basis is large enough: nothing moves
    H.hgks_assemble(hm, p[12], Q, dt)
    assert not shim.hx_captured(hm.handle)
    H.hgks_gmres_step(hm, p[4], Q.clone())
    assert shim.hx_captured(hm.handle)
