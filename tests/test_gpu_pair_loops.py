"""The FP64 pair loops and the k-phase fold at the edges of their tiles, against
plain FP64 sums of the same definitions."""
import numpy as np
import pytest

import paper_2608_00773_gb300 as q
from gpu_helpers import LibCase, rel_fro
from workloads import periodic_cell, small_cluster

pytestmark = pytest.mark.gpu
# every path sums the same FP64 products in another order: n_p n_b^2 terms of a
# batch, rounded at most (number of additions) x 2^-53 apart; 1e-12 is the
# repository's bound for the FP64 path
TOL = 1e-12


def _dense(lib):
    """(phi, grad) of every function at every point, the pattern as dense index matrix, v and w."""
    import torch
    wl, ex = lib.wl, lib.ex
    phi, grad = q.q4c_basis_eval(lib.tables, lib.grid, torch.tensor(ex["xyz"], device="cuda"))
    nf = wl.nf_of_atom
    f0 = np.concatenate([[0], np.cumsum(nf)])
    idx = np.full((f0[-1], f0[-1]), -1, np.int64)
    for A in range(wl.n_atoms):
        for k in range(ex["blk_ptr"][A], ex["blk_ptr"][A + 1]):
            B = ex["blk_col"][k]
            idx[f0[A]:f0[A + 1], f0[B]:f0[B + 1]] = ex["blk_off"][k] + np.arange(nf[A] * nf[B]).reshape(nf[A], nf[B])
    return phi.cpu().numpy(), grad.cpu().numpy(), idx


@pytest.mark.parametrize("n_atoms,batch_max", [(1, 1), (2, 7), (3, 8), (5, 9), (6, 33), (8, 65), (8, 300), (11, 1024)])
def test_fp64_pair_loops(n_atoms, batch_max):
    import torch
    wl = small_cluster(n_atoms, seed=40 + n_atoms, n_rad=9, n_theta=4, n_phi=7, batch_max=batch_max)
    lib = LibCase(wl)
    phi, grad, idx = _dense(lib)
    ok = idx >= 0
    w = lib.ex["w"]
    D = phi * (w * lib.v_host), grad * (w * lib.v_host)[None, :, None]
    g = [grad[:, :, k] for k in range(3)]
    d = [D[1][:, :, k] for k in range(3)]
    ref = [D[0] @ phi.T, sum(d[k] @ g[k].T for k in range(3))]
    ref += [d[a] @ g[b].T - d[b] @ g[a].T for a, b in ((1, 2), (2, 0), (0, 1))]
    for got, r in zip(lib.integrate("fp64")[:5], ref):
        out = np.zeros_like(got)
        out[idx[ok]] = r[ok]
        assert np.linalg.norm(got - out) <= TOL * max(np.linalg.norm(out), 1e-300)
    # the adjoint, the density and the gradient density of general (unsymmetric) matrices
    rng = np.random.default_rng(n_atoms)
    M = [rng.standard_normal(lib.grid.nnz) for _ in range(5)]
    G = [np.where(ok, m[np.maximum(idx, 0)], 0.0) for m in M]
    quad = lambda X, a, b: np.einsum("ip,ip->p", X.T @ a, b)  # noqa: E731  sum_ij X_ij a_i b_j
    n = quad(G[0], phi, phi)
    y = n + sum(quad(G[1], g[k], g[k]) for k in range(3))
    for k, (a, b) in enumerate(((1, 2), (2, 0), (0, 1))):
        y = y + quad(G[2 + k], g[a], g[b]) - quad(G[2 + k], g[b], g[a])
    T = [torch.tensor(m, device="cuda") for m in M]
    assert rel_fro(q.q4c_density(lib.tables, lib.grid, T[0]).cpu().numpy(), n) <= TOL
    assert rel_fro(q.q4c_density_full(lib.tables, lib.grid, T).cpu().numpy(), y) <= TOL
    assert rel_fro(q.q4c_integrate_backward(lib.tables, lib.grid, T).cpu().numpy(), w * y) <= TOL


@pytest.mark.parametrize("n_k,n_shell,cell", [(1, 2, (9.0, 10.0, 11.0)), (5, 2, (9.0, 10.0, 11.0)),
                                              (4, 3, (5.0, 5.0, 5.5)), (7, 3, (5.0, 5.0, 5.5))])
def test_kfold_remainders_and_long_runs(n_k, n_shell, cell):
    """One to four k-points a launch, runs of shifts below and above one phase table."""
    import torch
    wl = periodic_cell(cell=cell, n_atoms=2 if n_shell == 3 else 3, n_rad=4, n_theta=3, n_phi=4, n_shell=n_shell)
    t, g = q.setup(wl)
    ex = g.export()
    ptr, col, off = g.kpattern()
    rng = np.random.default_rng(n_k)
    H, ks = rng.standard_normal(g.nnz), rng.uniform(-0.5, 0.5, (n_k, 3))
    got = q.q4c_kfold(g, torch.tensor(H, device="cuda"), ks).cpu().numpy()
    row = np.repeat(np.arange(wl.n_atoms), np.diff(ex["blk_ptr"]))
    krow = np.repeat(np.arange(wl.n_atoms), np.diff(ptr))
    longest = 0
    for kb, (A, B) in enumerate(zip(krow, col)):
        qs = np.nonzero((row == A) & (ex["blk_col"] == B))[0]
        longest = max(longest, len(qs))
        for i, k in enumerate(ks):
            ref = sum(np.exp(2j * np.pi * (ex["blk_T"][x] @ k)) * H[ex["blk_off"][x]:ex["blk_off"][x + 1]] for x in qs)
            # a sum of len(qs) terms with phases good to a few 2^-53 times the reduced phase (|k.T| <= 9)
            assert np.abs(got[i, off[kb]:off[kb + 1]] - ref).max() <= 1e-14 * len(qs) * 10
    assert (longest > 32) == (n_shell == 3)  # 32 entries fill a table
