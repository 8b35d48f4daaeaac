"""The launch forms of the FP64 GMRES step against the oracle, at the sizes where one
gives way to the next: a cell shared by four lanes or two, one cell per thread, several
cells per thread, separate launches; Krylov sizes around a whole block of basis vectors
(8 in one launch, 4 in separate ones), none to three Jacobi sweeps, tetrahedra and
hexahedra, sizes that fill no warp.

Tolerance: the update's relative L2 error 1e-9, as every FP64 step is held to the oracle
(both round differently; GMRES amplifies that by the conditioning of A, about 1e6 at CFL 10).
"""
import numpy as np
import pytest

import oracle as O
import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def check(m, cond, **kw):
    import torch
    u = cond["u_inf"]
    base = (cond["rho_inf"], u[0] + 0.05, u[1] + 0.03, u[2] - 0.02, cond["p_inf"])
    Q, _ = I.smooth_state(m, amp=0.03, base=base)
    kw = dict(scheme=0, Pr=0.72 if cond["viscous"] else 1.0, **{**cond, **kw})
    hm = H.hgks_mesh_create(m, scheme_mask=1)
    Qd = hm.to_internal(Q)
    dQ = torch.empty_like(Qd)
    info = H.hgks_gmres_step(hm, H.hgks_default_params(**kw), Qd, None, dQ)
    Qo, _, res, lin = O.OracleMesh(m).gmres_step(O.make_params(**kw), Q)
    ref = Qo - Q
    err = np.linalg.norm(hm.to_caller(dQ) - ref) / np.linalg.norm(ref)
    assert err < 1e-9, err
    assert abs(info.res_l1 - res) <= 1e-11 * abs(res)


# (mesh, Krylov size, restarts, sweeps)
@pytest.mark.parametrize("n,k,restarts,sweeps", [(2, 3, 2, 2), (3, 9, 2, 2), (9, 8, 2, 1), (11, 17, 1, 3), (13, 1, 3, 2), (13, 10, 2, 0)])
def test_one_launch_tetrahedra(cuda, n, k, restarts, sweeps):
    check(I.cavity_mesh(n), I.cavity_conditions(0.15, 100.0), krylov_dim=k, restarts=restarts, jacobi_sweeps=sweeps)


@pytest.mark.parametrize("n,k", [(5, 9), (19, 7), (22, 8)])
def test_one_launch_hexahedra(cuda, n, k):
    check(I.hex_cavity_mesh(n), I.cavity_conditions(0.15, 100.0), krylov_dim=k, restarts=2)


def test_several_cells_per_thread(cuda):
    m = I.sphere_mesh(9, 21, stretch=I.sphere_stretch(21))           # 61,236 cells
    check(m, I.sphere_conditions(0.3), krylov_dim=9, restarts=2)


def test_separate_launches(cuda):
    m = I.sphere_mesh(20, 43, stretch=I.sphere_stretch(43))          # 619,200 cells
    check(m, I.sphere_conditions(0.3), krylov_dim=6, restarts=1)


@pytest.mark.parametrize("k", [1, 4, 5, 10])
def test_matrix_free_blocks(cuda, k):
    """Gram-Schmidt by blocks in separate launches with a first block of its own (matrix-free
    products): the step's tolerance against the oracle is that of the difference operator."""
    import torch
    m, cond = I.sphere_mesh(5, 7, stretch=1.3), I.sphere_conditions(0.3)
    Q, _ = I.smooth_state(m, amp=0.03, base=(1.0, 0.35, 0.03, -0.02, cond["p_inf"]))
    kw = dict(scheme=0, jv_mode=1, krylov_dim=k, restarts=2, **cond)
    hm = H.hgks_mesh_create(m, scheme_mask=1)
    Qd = hm.to_internal(Q)
    dQ = torch.empty_like(Qd)
    H.hgks_gmres_step(hm, H.hgks_default_params(**kw), Qd, None, dQ)
    Qo, _, _, _ = O.OracleMesh(m).gmres_step(O.make_params(**kw), Q)
    assert np.linalg.norm(hm.to_caller(dQ) - (Qo - Q)) / np.linalg.norm(Qo - Q) < 1e-4


def test_step_after_a_larger_krylov_size(cuda):
    """The basis moves when a later call needs more vectors; a step with the earlier
    parameters and buffers must not replay with the old addresses."""
    m, cond = I.sphere_mesh(4, 6, stretch=1.3), I.sphere_conditions(0.3)
    Q, _ = I.smooth_state(m, amp=0.03, base=(1.0, 0.35, 0.03, -0.02, cond["p_inf"]))
    hm = H.hgks_mesh_create(m, scheme_mask=1)
    Q0 = hm.to_internal(Q)
    Qd = Q0.clone()
    out = []
    for k in (4, 12, 4):
        Qd.copy_(Q0)
        H.hgks_gmres_step(hm, H.hgks_default_params(krylov_dim=k, **cond), Qd)
        out.append(Qd.clone())
    assert bool((out[0] == out[2]).all())
