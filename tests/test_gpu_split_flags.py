"""DC_RELU and DC_ACCUM where the views of a box are shared by a cluster: the
flags act once, on the whole sum, for both ways of staging, against the FP64
oracle (1e-5 relative L2)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [64, 63])
@pytest.mark.parametrize("kahan", [False, True])
def test_flags_act_on_the_whole_sum(W, kahan):
    V, H = 70, 48
    o = synth.sinusoid_orbit(V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=4, n_s=8, pitch=2.0, ds=2.0, vol_x=33,
                vol_y=30, vol_z=35, voxel=(1.2,) * 3, closed_orbit=1)
    P = synth.projection_matrices(o, H, W, 2.0)
    gg, og = api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)
    assert api.dc_geometry_get_tuning(gg)["bp_nz"] == 16   # 27 boxes: shared
    rng = np.random.default_rng(W)
    g = rng.normal(size=(2, V, H, W)).astype(np.float32)
    old = rng.normal(size=(2, 35, 30, 33)).astype(np.float32) * 1e-4
    ref = orc.backproject(og, g)
    dev = torch.as_tensor(g, device="cuda")
    for accum in (False, True):
        for relu in (False, True):
            out = torch.as_tensor(old, device="cuda").clone()
            api.dc_backproject(gg, dev, out=out, accum=accum, kahan=kahan, relu=relu)
            want = ref + (old if accum else 0.0)
            want = np.maximum(want, 0.0) if relu else want
            assert rel_l2(out.double().cpu().numpy(), want) < 1e-5
