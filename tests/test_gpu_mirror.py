"""The mirror of the canonical half and the spinor blocks on both sides of the
line between one launch and two (2^20 elements of the pattern): copies of values,
so equal to the bit."""
import pytest

import paper_2608_00773_gb300 as q
from gpu_helpers import LibCase
from workloads import single_atom, small_cluster

pytestmark = pytest.mark.gpu


def _spinor(W0, x, y, z):
    import torch
    S = torch.empty((2 * W0.shape[0], 2 * W0.shape[1]), dtype=torch.complex128, device=W0.device)
    S[0::2, 0::2], S[0::2, 1::2] = torch.complex(W0, z), torch.complex(y, x)
    S[1::2, 0::2], S[1::2, 1::2] = torch.complex(-y, x), torch.complex(W0, -z)
    return S


@pytest.mark.parametrize("nb", [1, 5, 1024, 1025])
def test_one_block(nb):
    import torch
    lib = LibCase(single_atom((0,) * (nb % 3) + (1,) * (nb // 3), alphas=[0.2 + 0.01 * k for k in range(nb % 3 + nb // 3)],
                              n_rad=4, n_theta=3, n_phi=4, batch_max=64))
    assert lib.grid.nnz == nb * nb
    V, W0, x, y, z, SS = q.q4c_integrate(lib.tables, lib.grid, lib.v, "fp64", spinor=True)
    V, W0, x, y, z = (m.view(nb, nb) for m in (V, W0, x, y, z))
    assert torch.equal(V, V.T) and torch.equal(W0, W0.T)
    assert all(torch.equal(m, -m.T) for m in (x, y, z))
    assert torch.equal(SS.reshape(2 * nb, 2 * nb, 2), torch.view_as_real(_spinor(W0, x, y, z)))


def test_pairs_of_blocks():
    import torch
    lib = LibCase(small_cluster(5, seed=7, n_rad=6, n_theta=3, n_phi=4))
    outs = q.q4c_integrate(lib.tables, lib.grid, lib.v, "fp64", spinor=True)
    ptr, col, off = lib.pat
    nf = lib.wl.nf_of_atom
    blocks = {(A, int(col[k])): (int(off[k]), nf[A], nf[int(col[k])]) for A in range(len(nf))
              for k in range(ptr[A], ptr[A + 1])}
    for (A, B), (o, a, b) in blocks.items():
        m = [t[o:o + a * b].view(a, b) for t in outs[:5]]
        oT = blocks[(B, A)][0]
        mT = [t[oT:oT + a * b].view(b, a).T for t in outs[:5]]
        assert all(torch.equal(s, t if k < 2 else -t) for k, (s, t) in enumerate(zip(m, mT)))
        SS = outs[5].reshape(-1, 2)[4 * o:4 * (o + a * b)]  # (real, imaginary)
        assert torch.equal(SS.reshape(2 * a, 2 * b, 2), torch.view_as_real(_spinor(*m[1:])))
