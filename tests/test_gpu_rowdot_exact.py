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


@pytest.mark.parametrize("n_s", [7, 40, 150])
def test_small_matrix_beside_a_large_one(n_s):
    """W0 is 1e12 between a far atom and the first one, and the far atom's cutoff sphere
    divides the middle atom's points: outside it W0 adds nothing, and the SO matrices'
    columns are as good as alone only where W0's largest elements do not set their unit."""
    import torch
    wl = _on_an_axis(n_s)
    wl.xyz = np.vstack([wl.xyz, [[0.0, 0.0, wl.r_c]]])
    wl.species_of_atom = np.array([0, 0, 1, 1], dtype=np.int32)
    t, g = q.setup(wl)
    ex = g.export()
    rng = np.random.default_rng(n_s)
    M = [np.zeros(g.nnz)] + [rng.standard_normal(g.nnz) for _ in range(3)]
    for a, b in ((0, 3), (3, 0)):
        k = int(ex["blk_ptr"][a]) + int(np.flatnonzero(ex["blk_col"][ex["blk_ptr"][a]:ex["blk_ptr"][a + 1]] == b)[0])
        M[0][ex["blk_off"][k]:ex["blk_off"][k + 1]] = 1e12
    G = [None] + [torch.tensor(m, device="cuda") for m in M]
    z = ex["xyz"][:, 2]
    out = np.abs(z) < 1.0
    out &= z < 0.0  # about the middle atom, beyond the far one's sphere
    near = [0 in ex["batch_atoms"][a:b] and 3 in ex["batch_atoms"][a:b]
            for a, b in zip(ex["batch_atom_ptr"][:-1], ex["batch_atom_ptr"][1:])]
    assert np.repeat(near, np.diff(ex["batch_ptr"]))[out].sum() > 10  # in batches that hold W0's columns
    ref = q.q4c_density_full(t, g, G).cpu().numpy()[out]
    y = q.q4c_density_full(t, g, G, "split").cpu().numpy()[out]
    g.status()
    assert np.linalg.norm(y - ref) <= 8 * 2.0 ** -44 * np.linalg.norm(ref)  # as above
