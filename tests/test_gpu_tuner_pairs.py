"""The tuner leaves the pair kernel (batches above 256 functions), which has one
shape, out of its timings: a bucket with nothing else is not timed and keeps its
shape; below the line it is timed as before."""
import pytest

import paper_2608_00773_gb300 as q
from gpu_helpers import LibCase, rel_fro
from workloads import single_atom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [256, 257])
@pytest.mark.parametrize("ks", [1, 2])
def test_bucket_of_large_batches(nb, ks):
    l = (0,) * (nb % 3) + (1,) * (nb // 3)
    lib = LibCase(single_atom(l, alphas=[0.2 + 0.05 * k for k in range(len(l))], n_rad=10, n_theta=5, n_phi=14,
                              batch_max=200))
    before = lib.integrate("split")
    q.q4c_grid_set_tiling(lib.grid, q.binding.TILE_BUCKETS - 1, ks)
    last, rowdot = q.q4c_autotune(lib.tables, lib.grid, lib.v)[-2:]
    lib.grid.status()
    assert last["batches"] == lib.grid.info.n_batches and rowdot["ms_one"] > 0 and rowdot["ms_two"] > 0
    if nb > 256:
        assert (last["ms_one"], last["ms_two"], last["k_steps"]) == (-1.0, -1.0, ks)
    else:
        assert last["ms_one"] > 0 and last["k_steps"] == (2 if last["ms_two"] < last["ms_one"] else 1)
    for a, b in zip(lib.integrate("split")[:2], before):
        assert rel_fro(a, b) <= 1e-13  # a shape changes no more than the order of FP64 additions
