"""Per-kernel timing names what ran: the one-launch GMRES of a small FP64 step under its own
name, not under that of the single Jacobi products it contains."""
import pytest

import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,jv_mode,one_launch", [(0, 0, True), (1, 0, False), (0, 1, False)],
                         ids=["fp64", "mixed", "matrix-free"])
def test_names_of_a_step(cuda, precision, jv_mode, one_launch):
    m, cond = I.cavity_mesh(4), I.cavity_conditions()
    hm = H.hgks_mesh_create(m, scheme_mask=1)
    Q = hm.to_internal(I.smooth_state(m, amp=0.05, base=(1.0, 0.1, 0.05, -0.03, cond["p_inf"]))[0])
    p = H.hgks_default_params(scheme=0, Pr=0.72, precision=precision, jv_mode=jv_mode, krylov_dim=4, restarts=2, **cond)
    H.hgks_profile_begin()
    H.hgks_gmres_step(hm, p, Q)
    prof = H.hgks_profile_end()
    parts = {"jacobi", "axpy_dot", "scale", "givens", "combine", "spmv"} & set(prof)
    if one_launch:
        assert prof["gmres"][1] == 1 and not parts, prof
    else:
        assert "gmres" not in prof and {"jacobi", "axpy_dot", "givens", "combine"} <= parts, prof
    assert {"recon", "flux", "gather", "assemble", "update"} <= set(prof)
