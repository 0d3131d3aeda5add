"""Filter kernels that take four images at once: tile, band and group edges,
against the FP64 oracle (line sums 2e-6 relative L2, the transpose 1e-5, the
filter and its reverse mode 1e-4: the tolerances of the per-image kernels)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


def _problem(V, H, W, n_mu, n_s, B, ds=1.0, shift=None):
    """A sinusoid problem; `shift` moves each view's principal point (pixels)."""
    p = 1.3
    o = synth.sinusoid_orbit(V)
    P = synth.projection_matrices(o, H, W, p)
    if shift is not None:
        for i in range(V):
            P[i, 0] += shift * (i + 1) * P[i, 2]
            P[i, 1] -= 0.5 * shift * (i + 1) * P[i, 2]
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=n_mu, n_s=n_s, pitch=p, ds=ds * p,
                vol_x=12, vol_y=12, vol_z=12, voxel=(2.0, 2.0, 2.0), closed_orbit=1)
    return desc, P, o.vdl


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


def _host(t):
    torch.cuda.synchronize()
    return t.double().cpu().numpy()


# (views, rows, cols, angles, s-bins, batch): detectors at the edges of an
# 8-step band and of a TMA box (256 samples with the margins), line counts at
# the edges of a 32-line task, 1 to 4 images in the last group, more angles
# than one group holds, one angle
SHAPES = [(5, 8, 8, 7, 31, 1), (4, 9, 17, 12, 32, 1), (3, 16, 238, 9, 33, 1),
          (2, 239, 24, 16, 65, 3), (7, 41, 63, 33, 97, 1), (1, 40, 40, 1, 64, 1),
          (2, 33, 500, 6, 640, 1), (6, 64, 64, 45, 64, 2)]


@pytest.mark.parametrize("shape", SHAPES)
def test_four_image_kernels_at_edges(shape):
    V, H, W, n_mu, n_s, B = shape
    desc, P, vdl = _problem(V, H, W, n_mu, n_s, B)
    gg, og = api.Geometry(desc, P, vdl), orc.Geometry(desc, P, vdl)
    rng = np.random.default_rng(V * 1000 + W)
    img = rng.normal(size=(B, V, H, W)).astype(np.float32)
    sino = rng.normal(size=(B, V, n_mu, n_s)).astype(np.float32)
    R, T = _host(api.dc_radon2d(gg, _dev(img))), _host(api.dc_radon2d_adjoint(gg, _dev(sino)))
    for b in range(B):
        for i in range(V):
            cu, cv = og.principal_point(i)
            assert rel_l2(R[b, i], orc.radon(img[b, i], desc["pitch"], n_mu, n_s, desc["ds"],
                                             cu, cv)) < 2e-6
            assert rel_l2(T[b, i], orc.radon_T(sino[b, i], H, W, desc["pitch"], desc["ds"],
                                               cu, cv)) < 1e-5
    api.dc_sync_status(gg)


@pytest.mark.parametrize("shift", [None, 0.37, 1e-4])
@pytest.mark.parametrize("ds", [1.0, 0.6])
def test_principal_points_per_view(shift, ds):
    """Views that share a principal point and views that do not (which the
    per-image kernels take) give the oracle's filter and reverse mode, and no
    image of a group depends on its neighbours."""
    desc, P, vdl = _problem(6, 37, 50, 33, 70, 1, ds, shift)
    gg, og = api.Geometry(desc, P, vdl), orc.Geometry(desc, P, vdl)
    rng = np.random.default_rng(8)
    g = rng.uniform(0.0, 2.0, size=(1, 6, 37, 50)).astype(np.float32)
    G = rng.normal(size=g.shape).astype(np.float32)
    W = rng.uniform(0.2, 0.8, size=(6, 33, 70)).astype(np.float32)
    gF, _ = api.dc_filter(gg, _dev(g), _dev(W))
    assert rel_l2(_host(gF), orc.filter(og, g, W)) < 1e-4
    gr, gW = api.dc_filter_adjoint(gg, _dev(G), _dev(g), _dev(W))
    rr, rW = orc.filter_adjoint(og, g, G, W)
    assert rel_l2(_host(gr), rr) < 1e-4 and rel_l2(_host(gW), rW) < 1e-4
    other = g.copy()
    other[0, 1] = np.nan
    gF2, _ = api.dc_filter(gg, _dev(other), _dev(W))
    keep = [0, 2, 3, 4, 5]
    assert torch.equal(gF2[:, keep], gF[:, keep])
