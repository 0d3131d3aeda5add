"""Eq. 9 weights with as many angles per CTA as the grid allows: 16 with a
remainder, fewer for few views, one (the edge test's oracle comparison)."""
import pytest

import test_gpu_crofton as edges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,n_mu,n_s", [(64, 161, 33), (32, 80, 40), (20, 62, 20), (2, 45, 31)])
def test_angles_per_cta(V, n_mu, n_s):
    edges.test_crofton_pair_groups_at_edges(V, n_mu, n_s, True)
