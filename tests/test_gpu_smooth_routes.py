"""The Gaussian layer's two kernels: few short lines take the one that holds
whole lines, more samples the tiled one.  Lines at the edges of the tiles (128
outputs, 64 lines) on both sides of the line between the two, against the FP64
oracle with the tolerance of every other size (1e-5 relative L2)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2410_14900_gb300 import api

from cases import rel_l2

pytestmark = pytest.mark.gpu


# views None: enough for the tiled kernel (more than 2^17 samples)
@pytest.mark.parametrize("n_mu,n_s,sigma,radius", [(127, 65, 20.0, 60), (128, 66, 7.0, 16),
                                                   (129, 130, 20.0, 60), (224, 64, 4.0, 1),
                                                   (225, 64, 4.0, 17), (1, 129, 5.0, 20),
                                                   (2, 3, 5.0, 40), (33, 40, 1.0, 0),
                                                   (150, 70, 90.0, 320)])
@pytest.mark.parametrize("views", [1, None])
@pytest.mark.parametrize("adjoint", [False, True])
def test_both_kernels(n_mu, n_s, sigma, radius, views, adjoint):
    V = views or (1 << 17) // (n_mu * n_s) + 1
    rng = np.random.default_rng(n_mu * 7 + n_s)
    W = rng.normal(size=(V, n_mu, n_s)).astype(np.float32)
    got = api.dc_gauss_smooth(torch.as_tensor(W, device="cuda"), sigma, radius, adjoint=adjoint)
    ref = orc.gauss_smooth(W, sigma, radius, adjoint=adjoint)
    got = got.double().cpu().numpy()
    assert rel_l2(got[..., :-1], ref[..., :-1]) < 1e-5
    np.testing.assert_array_equal(got[..., -1], W[..., -1])


def test_more_views_than_a_grid_holds():
    V = 65537
    W = torch.rand((V, 1, 2), device="cuda")
    # one sample a line, whose three taps sum to 1 but for their rounding
    assert torch.allclose(api.dc_gauss_smooth(W, 2.0, 1), W, rtol=1e-6, atol=0.0)


# A running sum of the taps rounds 2 radius times, one way for neighbouring sums,
# and scales every output by its error (4e-7 for the two axes at radius 60).  In 32
# parts it rounds some ten times: with the taps' own rounding (2 units of 6e-8)
# and the FMAs', which average out, 5 units are not reached.
@pytest.mark.parametrize("views", [4, 30])
@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("sigma,radius", [(5.0, 15), (20.0, 60)])
def test_taps_sum_to_one(views, adjoint, sigma, radius):
    rng = np.random.default_rng(radius)
    W = rng.uniform(0.2, 0.8, size=(views, 90, 64)).astype(np.float32)
    got = api.dc_gauss_smooth(torch.as_tensor(W, device="cuda"), sigma, radius, adjoint=adjoint)
    ref = orc.gauss_smooth(W, sigma, radius, adjoint=adjoint)
    assert rel_l2(got.double().cpu().numpy()[..., :-1], ref[..., :-1]) < 3e-7
