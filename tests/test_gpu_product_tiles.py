"""The products of batches of at most 256 functions at the edges of their tiles:
one to four tiles of 64 functions, last tiles of 1 to 64, steps of 1 to 16 points
(an odd and an even number of them for the two slicer groups), both stage shapes,
against the FP64 path."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from workloads import column_operator, potential, single_atom

pytestmark = pytest.mark.gpu
# values good to 2^-44 and digits to 2^-47 of the column maxima, summed over up to
# 341 points of one sign or another: 2^-44 x sqrt(341) x the spread of an element
# against its columns' maxima (about 10 on one centre) = 1e-11
TOL = 1e-10


@pytest.mark.parametrize("nb,batch_max", [(1, 1), (4, 15), (15, 16), (16, 17), (17, 33), (48, 64), (63, 341), (64, 48),
                                          (65, 31), (80, 100), (128, 32), (129, 49), (192, 200), (193, 341), (255, 65)])
def test_products_and_columns(nb, batch_max):
    import torch
    l = (0,) * (nb % 3) + (1,) * (nb // 3)
    wl = single_atom(l, alphas=[0.2 + 0.05 * k for k in range(len(l))], n_rad=10, n_theta=5, n_phi=14,
                     batch_max=batch_max)
    t, g = q.setup(wl)
    assert g.info.max_nb == nb
    ex = g.export()
    # a potential without the atom's symmetry, so that no output vanishes
    v = potential(ex["xyz"], wl) * (1.0 + 0.3 * np.sin(ex["xyz"] @ np.array([1.0, 2.0, 3.0])))
    v = torch.tensor(v, device="cuda")
    eps, knots = column_operator(wl, 5)
    q.q4c_tables_set_columns(t, eps, knots)
    ref = q.q4c_integrate(t, g, v)
    F = q.q4c_integrate_columns(t, g, v)
    scale = float(torch.linalg.norm(ref[1]))  # W0: the size of the gradient products
    for ks in (1, 2):
        for bucket in range(q.binding.TILE_BUCKETS):
            q.q4c_grid_set_tiling(g, bucket, ks)
        got = q.q4c_integrate(t, g, v, "split")
        for k, (a, b) in enumerate(zip(got[:5], ref[:5])):
            assert float(torch.linalg.norm(a - b)) <= TOL * (float(torch.linalg.norm(b)) if k < 2 else scale), (ks, k)
        Fs = q.q4c_integrate_columns(t, g, v, "split")
        assert float(torch.linalg.norm(Fs - F)) <= TOL * float(torch.linalg.norm(F))
    g.status()
