"""The four-image 2-D backprojection with s-bins finer than the pixels, on
detectors whose height leaves the fewest pixels over in wide tiles (256 x 8):
the s-window that such a tile would stage does not fit an SM at ds = pitch / 2
and pitch / 3.  Against the FP64 oracle (transpose 1e-5 relative L2, the filter
and its reverse mode 1e-4: the tolerances of every other size)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import rel_l2

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


def _host(t):
    torch.cuda.synchronize()
    return t.double().cpu().numpy()


# 17 views: 8 rows per thread; 3 views: the 2-row tiles of small grids
@pytest.mark.parametrize("V,H,W", [(17, 200, 256), (17, 360, 512), (17, 40, 512), (17, 200, 512),
                                   (3, 200, 256), (3, 40, 512), (3, 7, 256), (17, 8, 256)])
@pytest.mark.parametrize("per_pitch", [1, 2, 3])
def test_wide_detectors_with_fine_bins(V, H, W, per_pitch):
    n_mu, n_s, p = 5, 600, 1.1
    o = synth.sinusoid_orbit(V)
    P = synth.projection_matrices(o, H, W, p)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=n_mu, n_s=n_s, pitch=p, ds=p / per_pitch,
                vol_x=12, vol_y=12, vol_z=12, voxel=(2.0, 2.0, 2.0), closed_orbit=1)
    gg, og = api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)
    rng = np.random.default_rng(H + W + per_pitch)
    sino = rng.normal(size=(1, V, n_mu, n_s)).astype(np.float32)
    T = _host(api.dc_radon2d_adjoint(gg, _dev(sino)))
    for i in (0, V - 1):
        cu, cv = og.principal_point(i)
        assert rel_l2(T[0, i], orc.radon_T(sino[0, i], H, W, p, desc["ds"], cu, cv)) < 1e-5
    g = rng.uniform(0.0, 2.0, size=(1, V, H, W)).astype(np.float32)
    G = rng.normal(size=g.shape).astype(np.float32)
    Wr = rng.uniform(0.2, 0.8, size=(V, n_mu, n_s)).astype(np.float32)
    gF, _ = api.dc_filter(gg, _dev(g), _dev(Wr))
    assert rel_l2(_host(gF), orc.filter(og, g, Wr)) < 1e-4
    gr, gW = api.dc_filter_adjoint(gg, _dev(G), _dev(g), _dev(Wr))
    rr, rW = orc.filter_adjoint(og, g, G, Wr)
    assert rel_l2(_host(gr), rr) < 1e-4 and rel_l2(_host(gW), rW) < 1e-4
    S = torch.empty((1, V, n_mu, n_s), device="cuda")
    api.dc_filter(gg, _dev(g), _dev(Wr), S_out=S)
    gr2, _ = api.dc_filter_adjoint(gg, _dev(G), None, _dev(Wr), S=S)
    assert rel_l2(_host(gr2), rr) < 1e-4
    api.dc_sync_status(gg)
