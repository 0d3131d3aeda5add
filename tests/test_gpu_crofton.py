"""The Eq. 9 weight generator on the GPU against the FP64 oracle, and a
reconstruction that uses it."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api, synth

from cases import arc_open, circle64, phantom_projections, ragged, random_nn, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["circle64", "ragged", "arc_open", "random_nn"])
@pytest.mark.parametrize("m,taper", [(2, 3), (1, 0), (0, 0)])
def test_crofton_weights_match_oracle(name, m, taper):
    case = {"circle64": circle64, "ragged": ragged, "arc_open": arc_open,
            "random_nn": random_nn}[name]()
    segs = {"arc_open": [(0, True), (20, False)], "random_nn": [(0, False)]}.get(name)
    gg = api.Geometry(case.desc, case.P, case.vdl)
    og = orc.Geometry(case.desc, case.P, case.vdl)
    W = api.dc_crofton_weights(gg, segs, m=m, taper=taper).double().cpu().numpy()
    ref = orc.crofton_weights(og, segs, m=m, taper=taper)
    K = np.stack([orc.redundancy_K(og, i) for i in range(case.desc["n_views"])])
    # compare the effective weight W*K: where K ~ 0 (plane tangent to the orbit
    # at the source) M is a ratio of vanishing terms and carries no weight
    err = rel_l2(W * np.abs(K), ref * np.abs(K))
    assert err < (1e-4 if m > 0 else 2e-3), err


def test_reconstruction_with_crofton_weights_matches_oracle():
    case = arc_open()
    segs = [(0, True), (20, False)]
    gg = api.Geometry(case.desc, case.P, case.vdl)
    og = orc.Geometry(case.desc, case.P, case.vdl)
    g = phantom_projections(case).astype(np.float32)
    W = api.dc_crofton_weights(gg, segs)
    vol = api.reconstruct(gg, torch.as_tensor(g, device="cuda"), W)
    ref = orc.reconstruct(og, g, orc.crofton_weights(og, segs))
    assert rel_l2(vol.double().cpu().numpy(), ref) < 1e-3


@pytest.mark.parametrize("V,n_mu,n_s", [(31, 17, 31), (32, 16, 32), (33, 5, 33), (63, 1, 65),
                                        (64, 33, 2), (3, 4, 40)])
@pytest.mark.parametrize("closed", [True, False])
def test_crofton_pair_groups_at_edges(V, n_mu, n_s, closed):
    """View counts at the edges of the 31-pair groups, s-bins and angles at
    the edges of a warp and of a CTA, on a tilted closed and an open orbit.

    A plane that contains another view to within FP32's rounding of its
    distance has no defined sign of f_j there, so the number of crossings that
    FP32 and FP64 see may differ by the pieces' end views: such planes (s = 0
    on this symmetric orbit) are not compared."""
    o = synth.tilted_sinusoid_orbit(V, tilt_max_deg=12.0, freq=2.0)
    desc = dict(n_views=V, det_rows=32, det_cols=32, n_mu=n_mu, n_s=n_s, pitch=4.0, ds=5.0,
                vol_x=8, vol_y=8, vol_z=8, voxel=(2.0, 2.0, 2.0), closed_orbit=int(closed))
    P = synth.projection_matrices(o, 32, 32, 4.0)
    segs = [(0, closed)] if V < 10 else [(0, closed), (V // 2, not closed)]
    gg, og = api.Geometry(desc, P, o.vdl), orc.Geometry(desc, P, o.vdl)
    W = api.dc_crofton_weights(gg, segs, m=2, taper=2).double().cpu().numpy()
    ref = orc.crofton_weights(og, segs, m=2, taper=2)
    K = np.abs(np.stack([orc.redundancy_K(og, i) for i in range(V)]))
    mu = np.arange(n_mu)[:, None] * np.pi / n_mu
    s = (np.arange(n_s) - 0.5 * (n_s - 1) + 0.5)[None, :] * 5.0
    for i in range(V):
        lx, ly, lz = og.frame(i)
        D = og.D(i)
        th = (D * np.cos(mu)[..., None] * lx + D * np.sin(mu)[..., None] * ly + s[..., None] * lz)
        th /= np.linalg.norm(th, axis=-1, keepdims=True)
        d = np.stack([og.source(j) - og.source(i) for j in range(V) if j != i])
        K[i][(np.abs(th @ d.T) < 4e-6 * np.linalg.norm(d, axis=1)).any(-1)] = 0.0
    assert (K > 0).any()
    assert rel_l2(W * K, ref * K) < 1e-4
