"""What each operand of the split density and adjoint is resolved against: every
point's X, Y and Z against their own largest values, every matrix's columns
against their own."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from workloads import Species, Workload

pytestmark = pytest.mark.gpu


def _on_an_axis(n_s, R=1e-4):
    """Outer atoms with n_s functions each, one of them R off the z axis, and all points
    that count within R of the middle atom: X and Y are 2e4 times smaller than Z there."""
    sp = [Species("X", 8.0, [0] * n_s, [0.2 + 0.5 * k / n_s for k in range(n_s)]), Species("Y", 8.0, [0], [1.0])]
    return Workload("on-an-axis", np.array([[0.0, 0.0, -2.0], [R, 0.0, 2.0], [0.0, 0.0, 0.0]]),
                    np.array([0, 0, 1], dtype=np.int32), sp, r_min=3 * R, n_rad=1, R=R, n_theta=9, n_phi=11, batch_max=99)


@pytest.mark.parametrize("n_s", [7, 15, 16, 60, 150])  # 15 to 301 functions
@pytest.mark.parametrize("slot", [2, 3, 4])
def test_small_components(n_s, slot):
    import torch
    t, g = q.setup(_on_an_axis(n_s))
    G = [None] * 5
    G[slot] = torch.tensor(np.random.default_rng(n_s).standard_normal(g.nnz), device="cuda")
    ref = q.q4c_density_full(t, g, G).cpu().numpy()
    for ks in (1, 2):
        q.q4c_grid_set_tiling(g, q.binding.TILE_BUCKETS, ks)
        y = q.q4c_density_full(t, g, G, "split").cpu().numpy()
        g.status()
        # the double-float basis holds each value within 2^-44; two values a product, two
        # products of the size of their difference; signs are random in result and error alike
        assert np.linalg.norm(y - ref) <= 8 * 2.0 ** -44 * np.linalg.norm(ref), ks
