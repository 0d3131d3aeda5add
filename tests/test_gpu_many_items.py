"""Batches of more small items than one launch's grid holds: the boxes of an
item times the CTAs that share their views, times the items, beyond 65535."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


def _problem(V, H, W, vol, voxel, pitch):
    o = synth.sinusoid_orbit(V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=4, n_s=8, pitch=pitch, ds=pitch,
                vol_x=vol[2], vol_y=vol[1], vol_z=vol[0], voxel=(voxel,) * 3, closed_orbit=1)
    P = synth.projection_matrices(o, H, W, pitch)
    return api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)


# views shared by a cluster; 16-deep boxes of footprints too tall for 32-deep
# ones; the widths take the two ways of staging
@pytest.mark.parametrize("V,H,W,vol,voxel,B", [(64, 8, 8, (16, 16, 16), 1.0, 8200),
                                               (64, 8, 7, (16, 16, 16), 1.0, 8200),
                                               (2, 8, 8, (32, 4, 4), 5.0, 40000),
                                               (2, 8, 9, (32, 4, 4), 5.0, 40000)])
def test_more_items_than_a_grid_holds(V, H, W, vol, voxel, B):
    gg, og = _problem(V, H, W, vol, voxel, 2.0)
    rng = np.random.default_rng(W)
    few = rng.normal(size=(3, V, H, W)).astype(np.float32)
    idx = torch.arange(B, device="cuda") % 3
    gF = torch.as_tensor(few, device="cuda")[idx]
    got = api.dc_backproject(gg, gF)
    ref = orc.backproject(og, few)
    assert rel_l2(got[:3].double().cpu().numpy(), ref) < 1e-5
    assert torch.equal(got, got[:3][idx])  # an item's sums do not depend on its place
    gv = rng.normal(size=(3,) + vol).astype(np.float32)
    adj = api.dc_backproject_adjoint(gg, torch.as_tensor(gv, device="cuda")[idx])
    want = torch.as_tensor(orc.backproject_adjoint(og, gv), device="cuda")
    err = (adj.double() - want[idx]).flatten(1).norm(dim=1) / want[idx].flatten(1).norm(dim=1)
    assert float(err.max()) < 1e-5
