"""The filter's work area where the device has no room for the usual one."""
import pytest
import torch

from paper_2410_14900_gb300 import _lib as L
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


def _geometry(V, H, W, n_mu, n_s):
    o = synth.sinusoid_orbit(V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=n_mu, n_s=n_s, pitch=1.0, ds=1.0, vol_x=16,
                vol_y=16, vol_z=16, voxel=(1.0, 1.0, 1.0), closed_orbit=1)
    return api.Geometry(desc, synth.projection_matrices(o, H, W, 1.0), o.vdl)


def test_a_smaller_work_area_where_the_usual_one_does_not_fit():
    size = (400, 200, 240, 120, 240)
    usual = _geometry(*size)
    cap = api.dc_geometry_get_tuning(usual)["chunk_capacity"]
    g = torch.rand((1, 400, 200, 240), device="cuda")
    ref = api.reconstruct(usual, g).double().cpu().numpy()
    Lh, smaller = L.load(), []
    for n in range(40):   # the n-th allocation of the set-up fails
        Lh.dc_debug_fail_alloc_after(n)
        try:
            geom = _geometry(*size)
        except L.DCError as e:
            assert e.code == L.DC_ERR_OOM
            continue
        finally:
            Lh.dc_debug_fail_alloc_after(-1)
        c = api.dc_geometry_get_tuning(geom)["chunk_capacity"]
        if c < cap:
            smaller.append(c)
            vol = api.reconstruct(geom, g).double().cpu().numpy()
            assert rel_l2(vol, ref) < 1e-6
            api.dc_sync_status(geom)
    assert len(smaller) == 1
