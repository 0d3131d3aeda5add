"""The staged backprojection from g^F whose rows TMA cannot address (odd widths,
unaligned bases), and box depths, against the FP64 oracle and against the same
data in rows that TMA can address."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


def _problem(orbit, V, H, W, n, nz, voxel, pitch=1.5):
    o = {"circle": synth.circle_orbit, "sinusoid": synth.sinusoid_orbit}[orbit](V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=8, n_s=16, pitch=pitch, ds=pitch,
                vol_x=n, vol_y=n, vol_z=nz, voxel=(voxel,) * 3, vol_center=(2.0, -1.0, 3.0),
                closed_orbit=1)
    P = synth.projection_matrices(o, H, W, pitch)
    return api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)


def _store(g, store, offset):
    """g [B, V, H, W] in a storage form, its base `offset` elements into a buffer
    (16-bit: half a 4-byte unit), with NaN around it; (tensor, scale, FP32 values)."""
    B = g.shape[0]
    scale = None
    if store == "f32x2":
        right = torch.nn.functional.pad(g, (0, 1))[..., 1:]
        t = torch.stack([g, right - g], -1)
    elif store == "f16":
        scale = torch.full((B, g.shape[1]), 2.0 ** -8, device=g.device)
        t = (g / scale[..., None, None]).half()
    else:
        t = g.to({"f32": torch.float32, "bf16": torch.bfloat16}[store])
    per = 2 if store == "f32x2" else 1
    buf = torch.full((t.numel() + 64,), float("nan"), device=g.device, dtype=t.dtype)
    out = buf[per * offset:per * offset + t.numel()].view(t.shape)
    out.copy_(t)
    val = out[..., 0] if per == 2 else out.float() * (1 if scale is None else scale[..., None, None])
    return out, scale, val


# widths: odd; even but no 16-byte multiple in any form; aligned rows on an odd
# base; footprints that reach left and right of the detector and off it (the
# volume is larger than the field of view); volumes that end inside a box
@pytest.mark.parametrize("W,offset", [(53, 0), (54, 0), (53, 1), (56, 1), (56, 3), (2, 0)])
@pytest.mark.parametrize("store", ["f32", "f32x2", "bf16", "f16"])
@pytest.mark.parametrize("kahan", [False, True])
def test_rows_match_oracle(W, offset, store, kahan):
    orbit = "circle" if W == 53 else "sinusoid"
    gg, og = _problem(orbit, 35, 45, W, 21, 37, 1.7)
    rng = np.random.default_rng(W + offset)
    g = torch.as_tensor(rng.normal(size=(2, 35, 45, W)).astype(np.float32), device="cuda")
    gF, scale, val = _store(g, store, offset)
    ref = orc.backproject(og, val.double().cpu().numpy())
    for nz in (16, 32):
        api.dc_geometry_set_tuning(gg, 0, nz)
        vol = api.dc_backproject(gg, gF, scale, kahan=kahan)
        assert rel_l2(vol.double().cpu().numpy(), ref) < 1e-5
    api.dc_sync_status(gg)


@pytest.mark.parametrize("voxel,n,nz,depth", [(0.9, 224, 200, 32), (0.9, 40, 33, 16), (1.9, 160, 160, 16)])
def test_box_depth_of_the_geometry(voxel, n, nz, depth):
    """32 voxels per thread, or 16 where 32-deep boxes do not fit the staged
    tile or are fewer than the SMs."""
    gg, _ = _problem("circle", 8, 64, 64, n, nz, voxel, pitch=1.5)
    assert api.dc_geometry_get_tuning(gg)["bp_nz"] == depth


# rows of whole quads and not, detectors narrower than the projected volume,
# volumes smaller than a box, one voxel beyond it and of whole boxes
@pytest.mark.parametrize("W", [40, 41, 42])
@pytest.mark.parametrize("n,nz", [(7, 5), (17, 33), (32, 32), (21, 15)])
@pytest.mark.parametrize("relu", [False, True])
def test_adjoint_at_edges(W, n, nz, relu):
    gg, og = _problem("sinusoid", 34, 30, W, n, nz, 2.4)
    rng = np.random.default_rng(W * n)
    gv = rng.normal(size=(2, nz, n, n)).astype(np.float32)
    vol = rng.normal(size=gv.shape).astype(np.float32)
    got = api.dc_backproject_adjoint(gg, torch.as_tensor(gv, device="cuda"),
                                     torch.as_tensor(vol, device="cuda") if relu else None)
    ref = orc.backproject_adjoint(og, gv * (vol > 0) if relu else gv)
    assert rel_l2(got.double().cpu().numpy(), ref) < 1e-5
