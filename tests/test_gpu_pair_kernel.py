"""The products of large batches (two row tiles a step) at the edges of their
tiles: odd and even numbers of 64-function tiles, narrow last tiles, ragged and
largest point counts, against the FP64 path."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from workloads import column_operator, potential, single_atom

pytestmark = pytest.mark.gpu
# values good to 2^-44 and digits to 2^-47 of the column maxima, summed over up to
# 341 points of one sign or another: 2^-44 x sqrt(341) x the spread of an element
# against its columns' maxima (about 10 on one centre) = 1e-11
TOL = 1e-10


@pytest.mark.parametrize("nb,batch_max", [(256, 64), (257, 64), (271, 17), (272, 341), (320, 33), (321, 300), (384, 16), (447, 100)])
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
        q.q4c_grid_set_tiling(g, q.binding.TILE_BUCKETS - 1, ks)
        got = q.q4c_integrate(t, g, v, "split")
        for k, (a, b) in enumerate(zip(got[:5], ref[:5])):
            assert float(torch.linalg.norm(a - b)) <= TOL * (float(torch.linalg.norm(b)) if k < 2 else scale), (ks, k)
        Fs = q.q4c_integrate_columns(t, g, v, "split")
        assert float(torch.linalg.norm(Fs - F)) <= TOL * float(torch.linalg.norm(F))
    g.status()
