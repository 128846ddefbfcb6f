"""Basis tiles of the split path where a warp's 32 points all lie outside a
centre's cutoff sphere, at the edges of a batch's 32-point groups, against the
FP64 path.  The tiles are memory of an earlier call (Phi alone, other places),
so a value not written would show."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from gpu_helpers import LibCase, rel_fro
from workloads import small_cluster

pytestmark = pytest.mark.gpu


def _outside(lib):
    """Pairs (centre of a batch, group of 32 of its points) without a point inside the cutoff, and all pairs."""
    ex, n_out, n_all = lib.ex, 0, 0
    for b in range(lib.grid.info.n_batches):
        x = ex["xyz"][ex["batch_ptr"][b]:ex["batch_ptr"][b + 1]]
        for A in ex["batch_atoms"][ex["batch_atom_ptr"][b]:ex["batch_atom_ptr"][b + 1]]:
            r = np.linalg.norm(x - lib.wl.xyz[A], axis=1)
            for p in range(0, len(x), 32):
                n_all += 1
                n_out += r[p:p + 32].min() >= lib.wl.r_c
    return n_out, n_all


@pytest.mark.parametrize("n_atoms,batch_max", [(6, 65), (8, 96), (8, 100), (11, 341)])
def test_groups_outside_the_cutoff(n_atoms, batch_max):
    import torch
    wl = small_cluster(n_atoms, seed=90 + n_atoms, n_rad=12, n_theta=5, n_phi=8, batch_max=batch_max)
    wl.r_on, wl.r_c = 2.5, 3.0
    lib = LibCase(wl)
    n_out, n_all = _outside(lib)
    assert 0 < n_out < n_all
    M = lib.random(n_atoms, "P")
    n64 = q.q4c_density(lib.tables, lib.grid, M, "fp64").cpu().numpy()
    n = q.q4c_density(lib.tables, lib.grid, M, "split").cpu().numpy()
    assert rel_fro(n, n64) <= 1e-9
    for a, r in zip(lib.integrate("split")[:5], lib.integrate("fp64")[:5]):
        assert rel_fro(a, r) <= 1e-9
    lib.grid.status()
