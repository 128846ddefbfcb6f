"""Work waits that run out in every tensor kernel: the call returns, the grid
reports Q4C_ETIMEOUT once, and with the default limit the same calls give the
same results on the same context.  Each warp leaves its role as a whole (lanes
that disagreed about a time-out would leave the rest of their warp waiting)."""
import pytest

import paper_2608_00773_gb300 as q
from gpu_helpers import LibCase, rel_fro
from workloads import column_operator, single_atom

pytestmark = pytest.mark.gpu


# products of one and two K-steps a stage, the pair kernel (above 256 functions)
@pytest.mark.parametrize("nb,ks", [(100, 1), (100, 2), (300, 1), (300, 2)])
def test_every_tensor_kernel_gives_up_and_recovers(nb, ks):
    l = (0,) * (nb % 3) + (1,) * (nb // 3)
    lib = LibCase(single_atom(l, alphas=[0.2 + 0.05 * k for k in range(len(l))], n_rad=10, n_theta=5, n_phi=14,
                              batch_max=200))
    t, g, v = lib.tables, lib.grid, lib.v
    for bucket in range(q.binding.TILE_BUCKETS + 1):
        q.q4c_grid_set_tiling(g, bucket, ks)
    q.q4c_tables_set_columns(t, *column_operator(lib.wl, 5))
    G = lib.G(3)
    calls = [lambda: q.q4c_integrate(t, g, v, "split")[1], lambda: q.q4c_integrate_columns(t, g, v, "split"),
             lambda: q.q4c_density(t, g, G[0], "split"), lambda: q.q4c_integrate_backward(t, g, G, "split"),
             lambda: q.q4c_scf_pass(t, g, v, G, G, "split")[2]]
    ref = [c().cpu().numpy() for c in calls]
    g.status()
    try:
        q.q4c_set_wait_limit_ns(1)
        for c in calls:
            c()
            with pytest.raises(q.Q4CError) as e:
                g.status()
            assert e.value.status == 4
    finally:
        q.q4c_set_wait_limit_ns(0)
    for c, r in zip(calls, ref):
        # sums of up to 341 terms in another order of the FP64 atomics: 341 x 2^-53 < 1e-13
        assert rel_fro(c().cpu().numpy(), r) <= 1e-13
    g.status()
