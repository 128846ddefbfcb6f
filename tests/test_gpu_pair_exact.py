"""Level sums of the split products where every digit has one sign: the points of
a batch lie so close together that each function of the far atom, its gradient
along (1, 1, 1), is nearly constant over them, so that W0's three products add
3 n_p terms of one sign and nearly one size.  A level that passed 2^24 units
would lose its last bits.  Against the FP64 path, on both sides of the lines
between the two sizes of digit (113 and 341 points) and in both kernels."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from workloads import Species, Workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_theta,n_phi", [(7, 16), (6, 19), (17, 20), (11, 31)])  # 112, 114, 340, 341 points
@pytest.mark.parametrize("n_s", [100, 160])  # 200 and 320 functions
def test_sums_of_one_sign(n_theta, n_phi, n_s):
    import torch
    # phi_k = exp(-a_k r^2): 160 exponents give leading digits all over their range; the points
    # lie below the first knot of their own atom, whose functions are constant there
    sp = [Species("X", 8.0, [0] * n_s, [0.2 + 0.01 * k for k in range(n_s)])]
    wl = Workload("two-points", np.array([[0.0, 0.0, 0.0], [1.1, 1.1, 1.1]]), np.zeros(2, dtype=np.int32), sp,
                  r_min=2e-3, n_rad=1, R=1e-3, n_theta=n_theta, n_phi=n_phi, batch_max=n_theta * n_phi)
    t, g = q.setup(wl)
    assert g.info.max_nb == 2 * n_s and g.info.max_np == n_theta * n_phi
    v = torch.tensor(0.999 / g.export()["w"], device="cuda")  # D = w v = 0.999 at every point
    ref = q.q4c_integrate(t, g, v)
    got = q.q4c_integrate(t, g, v, "split")
    g.status()
    for k in range(2):  # V and W0 (the gradients are parallel: SO is rounding alone)
        # the double-float basis holds each value within 2^-44, and the terms have one sign: no cancellation
        assert float(torch.linalg.norm(got[k] - ref[k])) <= 4 * 2.0 ** -44 * float(torch.linalg.norm(ref[k])), k


def test_small_component_of_a_diagonal_tile():
    """Every point lies within 1e-4 of the axis of three atoms: X is 2e4 times smaller
    than Z, and SO_y = sum D (Z_i X_j - X_i Z_j) is as good as X only where X is sliced
    against its own largest values.  The outer atoms' 64 functions are one diagonal tile."""
    import torch
    R = 1e-4
    sp = [Species("X", 8.0, [0] * 32, [0.2 + 0.02 * k for k in range(32)]),
          Species("Y", 8.0, [0] * 200, [0.2 + 0.01 * k for k in range(200)])]
    wl = Workload("on-an-axis", np.array([[0.0, 0.0, -2.0], [0.0, 0.0, 2.0], [0.0, 0.0, 0.0]]),
                  np.array([0, 0, 1], dtype=np.int32), sp, r_min=2 * R, n_rad=1, R=R, n_theta=10, n_phi=18, batch_max=300)
    t, g = q.setup(wl)
    assert g.info.max_nb == 264
    ex = g.export()
    x, z = ex["xyz"][:, 0], ex["xyz"][:, 2]
    v = torch.tensor(np.where(np.abs(z) < 1.0, x / R, 0.0) / ex["w"], device="cuda")  # D = x / R about the middle atom
    ref = q.q4c_integrate(t, g, v)[3].cpu().numpy()
    got = q.q4c_integrate(t, g, v, "split")[3].cpu().numpy()
    g.status()
    # the block of the outer atoms: all its terms D (Z_i X_j - X_i Z_j) have one sign, values as above
    k = int(np.flatnonzero(ex["blk_col"][: ex["blk_ptr"][1]] == 1)[0])
    s = slice(int(ex["blk_off"][k]), int(ex["blk_off"][k + 1]))
    assert np.linalg.norm(ref[s]) > 0.0
    assert np.linalg.norm(got[s] - ref[s]) <= 4 * 2.0 ** -44 * np.linalg.norm(ref[s])
