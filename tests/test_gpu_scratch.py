"""Results do not depend on what device memory held before: the compact scheme has one
sub-polynomial per face, so on hexahedra six of the eight that the coefficient array has
room for are written. The rest keeps whatever the allocation held; here every byte is set so
that a double read from it is a NaN.

Tolerances: the residual parity tests' (2e-12 of the flux scale, 1e-11 of the gradient scale);
against a fresh handle the same kernels run on the same data, bit for bit.
"""
import numpy as np
import pytest

import handle_shim
import oracle as O
import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I
from test_gpu_hex import face_sums

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def shim(cuda, tmp_path_factory):
    return handle_shim.load(tmp_path_factory.mktemp("shim"))


MESHES = {
    "hexcav5": lambda: (I.hex_cavity_mesh(5, jitter=0.15), I.cavity_conditions()),
    "hextilt6": lambda: (I.hex_tilted_box_mesh(6), I.sphere_conditions(0.3)),
    "cavity4": lambda: (I.cavity_mesh(4), I.cavity_conditions()),
}


def state(m, cond):
    u = cond["u_inf"]
    return I.smooth_state(m, seed=I.BASE_SEED + 3, amp=0.05, base=(cond["rho_inf"], u[0] + 0.1, u[1] + 0.05, -0.03, cond["p_inf"]))


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("scheme", [0, 1], ids=["weno", "hweno"])
def test_residual_on_poisoned_coefficients(shim, name, scheme):
    import torch
    m, cond = MESHES[name]()
    Q, G = state(m, cond)
    kw = dict(scheme=scheme, Pr=0.72 if cond["viscous"] else 1.0, **cond)
    hm = H.hgks_mesh_create(m, scheme_mask=1 << scheme)
    assert shim.hx_fill_coef(hm.handle, 0xff) == 0
    Qd, Gd = hm.to_internal(Q), hm.to_internal(G) if scheme else None
    R, Gn = torch.empty_like(Qd), torch.empty_like(Gd) if scheme else None
    H.hgks_residual(hm, H.hgks_default_params(**kw), Qd, Gd, R, Gn)
    om = O.OracleMesh(m)
    out = om.residual(O.make_params(**kw), Q, G)
    Ro, Go = out if scheme else (out, None)
    scale, aov = face_sums(om, Q)
    assert (np.abs(hm.to_caller(R) - Ro) / scale).max() <= 2e-12
    if scheme:
        assert (np.abs(hm.to_caller(Gn) - Go) / (np.repeat(np.abs(Q), 3, axis=1) * aov[:, None])).max() <= 1e-11


def test_batch_residual_on_poisoned_coefficients(shim):
    import torch
    m, cond = MESHES["hexcav5"]()
    Q, G = state(m, cond)
    p = H.hgks_default_params(scheme=1, Pr=0.72, **cond)
    hm = H.hgks_mesh_create(m, scheme_mask=2)
    Qd, Gd = hm.to_internal(Q), hm.to_internal(G)
    out = []
    for byte in (0x00, 0xff):
        b = H.hgks_batch_create([hm], [p])
        H.hgks_batch_set_state(b, 0, Qd, Gd)
        assert shim.hx_fill_batch_coef(b.handle, byte) == 0
        H.hgks_batch_residual(b)
        R, Gn = torch.empty_like(Qd), torch.empty_like(Gd)
        H.hgks_batch_get_state(b, 0, R=R, G_new=Gn)
        torch.cuda.synchronize()
        out.append((R, Gn))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
