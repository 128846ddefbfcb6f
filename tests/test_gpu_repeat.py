"""Equal calls of the split density and adjoint give equal bits, also where a
batch's functions are shared out over several work items (above 256), and the
potential may share its array with the density it is replaced by."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from gpu_helpers import LibCase, rel_fro
from workloads import single_atom

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,batch_max", [(256, 200), (257, 129), (513, 128), (800, 300)])  # 1, 2, 3, 4 shares
def test_equal_calls_repeat(nb, batch_max):
    import torch
    l = (0,) * (nb % 3) + (1,) * (nb // 3)
    lib = LibCase(single_atom(l, alphas=[0.2 + 0.01 * k for k in range(len(l))], n_rad=12, n_theta=6, n_phi=10,
                              batch_max=batch_max))
    t, g = lib.tables, lib.grid
    G = lib.G(9)
    calls = [lambda: [q.q4c_density(t, g, G[0], "split")], lambda: [q.q4c_integrate_backward(t, g, G, "split")],
             lambda: [q.q4c_density_full(t, g, G, "split")],
             lambda: q.q4c_scf_pass(t, g, lib.v, G, G, "split")[1:]]
    first = [c() for c in calls]
    for _ in range(8):
        for c, f in zip(calls, first):
            assert all(torch.equal(a, b) for a, b in zip(c(), f))
    # values good to 2^-44 of their own and digits to 2^-48 of their point's or column's largest, up
    # to 100 times an element on one centre: 1e-11
    assert rel_fro(first[0][0].cpu().numpy(), q.q4c_density(t, g, G[0]).cpu().numpy()) <= 1e-11
    assert rel_fro(first[1][0].cpu().numpy(), q.q4c_integrate_backward(t, g, G).cpu().numpy()) <= 1e-11
    # n over v: every batch's v is read before its n is written
    v = lib.v.clone()
    H, n, _ = q.q4c_scf_pass(t, g, v, G, None, "split", n_out=v)
    ref = q.q4c_integrate(t, g, lib.v, "split")
    g.status()
    assert torch.equal(n, first[3][0])
    for a, b in zip(H[:2], ref[:2]):
        assert float(torch.linalg.norm(a - b)) <= 1e-13 * float(torch.linalg.norm(b))
