"""hgks_batch_autotune reports the block shapes that are launched: k_recon takes at most 128
threads a block on hexahedra, so 256 is neither timed nor reported there. Repeated, because the
choice among near equals is the clock's."""
import pytest

import paper_2304_09485_gb300 as H
from paper_2304_09485_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", [0, 1], ids=["weno", "hweno"])
def test_hexahedral_shapes(cuda, scheme):
    m, cond = I.hex_cavity_mesh(12), I.cavity_conditions()
    hm = H.hgks_mesh_create(m, scheme_mask=1 << scheme)
    Q, G = (hm.to_internal(a) for a in I.smooth_state(m, amp=0.05, base=(1.0, 0.1, 0.05, -0.03, cond["p_inf"])))
    b = H.hgks_batch_create([hm], [H.hgks_default_params(scheme=scheme, Pr=0.72, **cond)])
    H.hgks_batch_set_state(b, 0, Q, G if scheme else None)
    for _ in range(20):
        recon, flux = H.hgks_batch_autotune(b)
        assert recon in (64, 128) and flux in (64, 128, 256)
        info = H.hgks_batch_info(b)
        assert (info.blk_recon, info.blk_flux) == (recon, flux)
