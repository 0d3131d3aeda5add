"""DC_KAHAN over no more views than one plain sum takes: the same bits as
without it (one sum needs no compensation), for every storage form whose rows
TMA can address, on both sides of 32 views."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [1, 31, 32, 33])
@pytest.mark.parametrize("store", ["f32", "f32x2", "bf16", "f16"])
def test_one_sum_needs_no_compensation(V, store):
    H, W = 48, 64
    o = synth.sinusoid_orbit(V)
    # more 16-deep boxes than clusters would share
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=4, n_s=8, pitch=2.0, ds=2.0, vol_x=130,
                vol_y=100, vol_z=70, voxel=(0.8,) * 3, closed_orbit=1)
    P = synth.projection_matrices(o, H, W, 2.0)
    gg, og = api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)
    rng = np.random.default_rng(V)
    g = torch.as_tensor(rng.normal(size=(1, V, H, W)).astype(np.float32), device="cuda")
    scale, val = None, g
    if store == "f32x2":
        g = torch.stack([g, torch.nn.functional.pad(g, (0, 1))[..., 1:] - g], -1)
    elif store == "f16":
        scale = torch.full((1, V), 2.0 ** -8, device="cuda")
        g = (g / scale[..., None, None]).half()
        val = g.float() * scale[..., None, None]
    elif store == "bf16":
        g = g.bfloat16()
        val = g.float()
    ref = orc.backproject(og, val.double().cpu().numpy())
    for nz in (16, 32):
        api.dc_geometry_set_tuning(gg, 0, nz)
        plain = api.dc_backproject(gg, g, scale)
        comp = api.dc_backproject(gg, g, scale, kahan=True)
        assert rel_l2(comp.double().cpu().numpy(), ref) < 1e-5
        assert V > 32 or torch.equal(comp, plain)
