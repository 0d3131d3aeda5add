"""The storage form of a g^F that only the next backprojection reads: which
calls take FP32 pairs, that both forms agree, and what happens where the pairs,
twice the memory, do not fit."""
import gc

import pytest
import torch

from paper_2410_14900_gb300 import api, synth
from paper_2410_14900_gb300.autograd import reconstruct

from cases import rel_l2

pytestmark = pytest.mark.gpu


def _geometry(V, H, W, n, voxel):
    o = synth.sinusoid_orbit(V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=8, n_s=64, pitch=1.0, ds=4.0, vol_x=n,
                vol_y=n, vol_z=n, voxel=(voxel,) * 3, vol_center=(1.0, 2.0, -1.0), closed_orbit=1)
    return api.Geometry(desc, synth.projection_matrices(o, H, W, 1.0), o.vdl)


# a volume of many boxes; one of few beside the same pixels; one pixel short of
# 4M; voxels of three pixels, whose footprints do not fit a tile; odd rows
@pytest.mark.parametrize("V,H,W,n,voxel,form", [
    (64, 256, 256, 160, 0.9, "f32x2"), (64, 256, 256, 48, 0.9, "f32"),
    (64, 256, 256, 16, 0.5, "f32"), (63, 256, 256, 160, 0.9, "f32"),
    (64, 256, 256, 160, 1.9, "f32"), (66, 256, 255, 160, 0.9, "f32")])
def test_form_and_agreement(V, H, W, n, voxel, form):
    geom = _geometry(V, H, W, n, voxel)
    assert api.transient_dtype(geom, 1) == form
    for other in ("bf16", "f16", "f32x2"):
        assert api.transient_dtype(geom, 1, other) == other
    g = torch.rand((1, V, H, W), device="cuda")
    gF, _ = api.dc_filter(geom, g, None, "f32")
    ref = api.dc_backproject(geom, gF, relu=True)
    vol = api.reconstruct(geom, g, relu=True)
    net = reconstruct(g, None, geom, True)
    assert torch.equal(vol, net)
    if form == "f32":
        assert torch.equal(vol, ref)
    assert rel_l2(vol.double().cpu().numpy(), ref.double().cpu().numpy()) < 1e-5


def test_a_centre_beside_the_source():
    """The middle view's source level with the volume's centre: no scale."""
    o = synth.circle_orbit(64)
    desc = dict(n_views=64, det_rows=256, det_cols=256, n_mu=8, n_s=64, pitch=1.0, ds=4.0, vol_x=32,
                vol_y=32, vol_z=32, voxel=(1.0,) * 3, closed_orbit=1)
    a = o.sources[32]
    desc["vol_center"] = (float(a[0]), float(a[1]), float(a[2]))
    geom = api.Geometry(desc, synth.projection_matrices(o, 256, 256, 1.0), o.vdl)
    assert geom.pixels_per_mm() > 1e6
    assert api.transient_dtype(geom, 1) == "f32"


def test_pairs_that_do_not_fit_give_way():
    V, H, W, n = 160, 256, 256, 160
    geom = _geometry(V, H, W, n, 0.9)
    assert api.transient_dtype(geom, 1) == "f32x2"
    g = torch.rand((1, V, H, W), device="cuda")
    gF, _ = api.dc_filter(geom, g, None, "f32")
    ref = api.dc_backproject(geom, gF)
    del gF
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # room for g^F in FP32 (42 MB) and the volume (16 MB), not for the pairs (84
    # MB); a pool of their own, where no block of earlier tests is free
    room = torch.cuda.memory_reserved() + (72 << 20)
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction(room / total)
    try:
        with torch.cuda.use_mem_pool(torch.cuda.MemPool()):
            vol = api.reconstruct(geom, g)
        same = torch.equal(vol, ref)
        del vol
        torch.cuda.empty_cache()
        with torch.cuda.use_mem_pool(torch.cuda.MemPool()):
            net = reconstruct(g, None, geom)
        assert same and torch.equal(net, ref)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
