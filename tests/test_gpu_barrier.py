"""A one-launch GMRES whose grid barrier does not open: the wait ends by itself, the call
returns HGKS_ERR_CUDA, the caller's state is the step's start, and the next step is clean.

The barrier is kept shut by expecting one arrival more than the launch has blocks, with a
short limit of polls: every block gives up at the first barrier and returns.
"""
import pytest

import handle_shim
import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I

pytestmark = pytest.mark.gpu
POLLS = 1 << 22
ERR_CUDA = 3


@pytest.fixture(scope="module")
def shim(cuda, tmp_path_factory):
    return handle_shim.load(tmp_path_factory.mktemp("shim"))


def problem(scheme, hexa):
    cond = I.cavity_conditions()
    m = I.hex_cavity_mesh(6) if hexa else I.cavity_mesh(4)
    hm = H.hgks_mesh_create(m, scheme_mask=1 << scheme)
    Q, G = I.smooth_state(m, amp=0.05, base=(1.0, 0.1, 0.05, -0.03, cond["p_inf"]))
    p = H.hgks_default_params(scheme=scheme, Pr=0.72, krylov_dim=4, restarts=2, **cond)
    return hm, p, hm.to_internal(Q), hm.to_internal(G) if scheme else None


@pytest.mark.parametrize("scheme", [0, 1], ids=["weno", "hweno"])
def test_state_is_kept_when_a_barrier_gave_up(shim, scheme):
    """The record alone (as a barrier would leave it): the update is left out, the error reported once."""
    import torch
    hm, p, Q0, G0 = problem(scheme, False)
    Q, G = Q0.clone(), G0.clone() if scheme else None
    H.hgks_gmres_step(hm, p, Q, G)
    after = Q.clone()
    Q.copy_(Q0)
    if scheme:
        G.copy_(G0)
    assert shim.hx_set_stuck(hm.handle) == 0
    with pytest.raises(H.HGKSError) as e:
        H.hgks_gmres_step(hm, p, Q, G)
    assert e.value.status == ERR_CUDA and "barrier" in str(e.value)
    assert torch.equal(Q, Q0) and (not scheme or torch.equal(G, G0))
    H.hgks_gmres_step(hm, p, Q, G)
    assert torch.equal(Q, after)


@pytest.mark.parametrize("scheme,hexa", [(0, False), (1, True)], ids=["tet", "hex"])
def test_a_barrier_that_does_not_open(shim, scheme, hexa):
    import torch
    hm, p, Q0, G0 = problem(scheme, hexa)
    Q, G = Q0.clone(), G0.clone() if scheme else None
    shim.hx_barrier(hm.handle, 1, 1 << 12)
    with pytest.raises(H.HGKSError) as e:
        H.hgks_gmres_step(hm, p, Q, G)
    assert e.value.status == ERR_CUDA and "barrier" in str(e.value)
    assert torch.equal(Q, Q0) and (not scheme or torch.equal(G, G0))
    # a solve ends with the error after its first step, from the state it was given
    with pytest.raises(H.HGKSError) as e:
        H.hgks_solve_steady(hm, p, Q, G, drop_tol=1e-8, max_steps=3)
    assert e.value.status == ERR_CUDA
    assert torch.equal(Q, Q0) and (not scheme or torch.equal(G, G0))
    # the handle is usable: other parameters, so that the step is captured anew
    shim.hx_barrier(hm.handle, 0, POLLS)
    p.cfl = 7.0
    H.hgks_gmres_step(hm, p, Q, G)
    fresh, _, Qf, Gf = problem(scheme, hexa)
    H.hgks_gmres_step(fresh, p, Qf, Gf)
    assert torch.equal(Q, Qf) and (not scheme or torch.equal(G, Gf))
