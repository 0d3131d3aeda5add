"""The backprojection's transpose for voxels finer than the pixels (0.75 pixels
per voxel and below: two CTAs per SM) against the FP64 oracle, 1e-5 relative
L2 as for every other scale."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


# on both sides of the line (pitch 1.5, 1.6 times the voxel); rows of whole
# quads and not; volumes within a box, one voxel beyond it, of whole boxes and
# of more boxes than three CTAs per SM hold at once (the two-CTA kernel)
@pytest.mark.parametrize("voxel", [0.05, 0.3, 0.70, 0.71])
@pytest.mark.parametrize("W", [40, 41])
@pytest.mark.parametrize("n,nz", [(9, 5), (33, 33), (32, 64), (145, 65)])
@pytest.mark.parametrize("relu", [False, True])
def test_fine_voxels(voxel, W, n, nz, relu):
    V, H, p = 34, 30, 1.5
    o = synth.sinusoid_orbit(V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=8, n_s=16, pitch=p, ds=p, vol_x=n, vol_y=n,
                vol_z=nz, voxel=(voxel,) * 3, vol_center=(2.0, -1.0, 3.0), closed_orbit=1)
    P = synth.projection_matrices(o, H, W, p)
    gg, og = api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)
    rng = np.random.default_rng(W * n)
    gv = rng.normal(size=(2, nz, n, n)).astype(np.float32)
    vol = rng.normal(size=gv.shape).astype(np.float32)
    got = api.dc_backproject_adjoint(gg, torch.as_tensor(gv, device="cuda"),
                                     torch.as_tensor(vol, device="cuda") if relu else None)
    ref = orc.backproject_adjoint(og, gv * (vol > 0) if relu else gv)
    assert rel_l2(got.double().cpu().numpy(), ref) < 1e-5
