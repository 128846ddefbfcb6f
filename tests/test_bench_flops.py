"""The FP64 path's roofline fraction counts the pair sums its kernels form."""
from types import SimpleNamespace

import bench


def test_fp64_pair_flops():
    batches = [(298, 57), (70, 24), (1, 1), (341, 205)]
    info = SimpleNamespace(flops_alg=sum(14.0 * n * b * b for n, b in batches), sum_np_nb=sum(n * b for n, b in batches))
    fma = 0
    for n, b in batches:
        pairs = sum(1 for i in range(b) for j in range(b) if i <= j)
        fma += n * pairs * (10 + 1 + 10)  # V, W0 (3), SO (2 each); density; adjoint
    assert bench.fp64_pair_flops(info) == 2.0 * fma
    assert bench.fp64_pair_flops(info) < sum(bench.step_flops(info).values())
