"""DC_KAHAN on rows that TMA cannot address compensates every view's term.

The first of 32 views gives each voxel a term T and the others 2^-26 of about
the same, under half a unit in T's last place: a plain FP32 sum stays at T, the
compensated one comes to within a unit of the exact sum, several units above
T.  With the views shared by a cluster each share is rounded once more before
the shares are added, half a unit."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

pytestmark = pytest.mark.gpu

V, H = 32, 60


@pytest.mark.parametrize("W,store", [(61, "f32"), (61, "f32x2"), (61, "bf16"), (61, "f16"),
                                     (62, "f32"), (62, "bf16"), (62, "f16")])
@pytest.mark.parametrize("nz,ulps", [(32, 1.0), (16, 1.5)])
def test_every_view_is_compensated(W, store, nz, ulps):
    o = synth.circle_orbit(V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=4, n_s=8, pitch=2.0, ds=2.0, vol_x=20,
                vol_y=20, vol_z=20, voxel=(1.5,) * 3, closed_orbit=1)
    P = synth.projection_matrices(o, H, W, 2.0)
    gg, og = api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)
    api.dc_geometry_set_tuning(gg, 0, nz)
    small = 2.0 ** -26

    def volume(rest):
        val = torch.full((1, V), rest, device="cuda")
        val[0, 0] = 1.0
        g = val[..., None, None].expand(1, V, H, W).contiguous()
        sc = None
        if store == "f32x2":
            right = torch.nn.functional.pad(g, (0, 1))[..., 1:]
            g = torch.stack([g, right - g], -1)
        elif store == "f16":
            sc, g = val.clamp(min=small), (g > 0).half()
        elif store == "bf16":
            g = g.bfloat16()
        return api.dc_backproject(gg, g, sc, kahan=True).cpu().numpy()

    first, both = volume(0.0), volume(small)
    tiny = np.full((1, V, H, W), small)
    tiny[0, 0] = 0.0
    want = orc.backproject(og, tiny)
    unit = np.spacing(first).astype(np.float64)
    assert (want > 3.5 * unit).all()
    assert (np.abs(both.astype(np.float64) - first - want) <= ulps * unit).all()
