"""The split density and adjoint at the edges of their tiles (32-function j-tiles,
16-function chunks, K segments of 112, shares of 256 functions, 128-point tiles)
against the FP64 path, for every subset of matrices that takes another route."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from gpu_helpers import rel_fro
from workloads import single_atom

pytestmark = pytest.mark.gpu
# the double-float basis holds each value within 2^-44 and the digits within
# 2^-48 of the largest of its point or column; random signs of up to 300 x 300
# terms cancel to about 1/300 of their sum of magnitudes: 2^-44 x 300 = 2e-11
TOL = 1e-10


@pytest.mark.parametrize("nb,batch_max", [(1, 7), (15, 200), (16, 128), (17, 129), (32, 200), (33, 200), (48, 60), (49, 200),
                                          (112, 129), (113, 200), (128, 129), (224, 1024), (256, 200), (257, 200),
                                          (300, 129)])
def test_density_and_adjoint_at_tile_edges(nb, batch_max):
    import torch
    l = (0,) * (nb % 3) + (1,) * (nb // 3)
    wl = single_atom(l, alphas=[0.2 + 0.11 * k for k in range(len(l))], n_rad=12, n_theta=6, n_phi=10, batch_max=batch_max)
    t, g = q.setup(wl)
    assert g.info.max_nb == nb
    rng = np.random.default_rng(nb)
    M = [torch.tensor(rng.standard_normal(g.nnz), device="cuda") for _ in range(5)]
    M[2:] = [3.0 ** k * m for k, m in enumerate(M[2:])]  # other column exponents per matrix
    for ks in (1, 2):
        q.q4c_grid_set_tiling(g, q.binding.TILE_BUCKETS, ks)
        n = q.q4c_density(t, g, M[0], "split").cpu().numpy()
        assert rel_fro(n, q.q4c_density(t, g, M[0]).cpu().numpy()) <= TOL
        for present in ((1, 1, 1, 1, 1), (0, 1, 0, 0, 0), (0, 0, 1, 0, 0), (0, 0, 0, 1, 1), (1, 0, 0, 0, 1), (0, 1, 1, 0, 1)):
            G = [m if p else None for m, p in zip(M, present)]
            y = q.q4c_integrate_backward(t, g, G, "split").cpu().numpy()
            ref = q.q4c_integrate_backward(t, g, G).cpu().numpy()
            full = q.q4c_integrate_backward(t, g, M).cpu().numpy()
            # a single atom's SO terms nearly vanish by symmetry: errors are of the terms' size
            assert np.linalg.norm(y - ref) <= TOL * max(np.linalg.norm(ref), np.linalg.norm(full)), (ks, present)
    g.status()
