"""The float64-pipe share of bench.py's algorithmic counts: the split kernel's
contractions count where they run on that pipe (lines, 7-node triangles) and
not where they are digit products on the tensor cores."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("d,n_p,contractions", [(1, 5, True), (2, 7, True), (2, 12, False), (2, 18, False),
                                                (2, 27, False), (3, 12, False), (3, 25, False), (3, 78, False)])
def test_split_kernel_share(d, n_p, contractions):
    n_e = 100
    full = bench.algorithmic_flops("split_volume", n_e, n_p, d, 0)
    pointwise = n_e * n_p * (30 + 43 * d)
    assert bench.float64_pipe_flops("split_volume", n_e, n_p, d, 0) == (full if contractions else pointwise)
    assert pointwise < full


def test_other_kernels_in_full():
    for group in ("face", "hadamard_volume"):
        assert bench.float64_pipe_flops(group, 50, 18, 2, 300) == bench.algorithmic_flops(group, 50, 18, 2, 300)
    assert bench.float64_pipe_flops("root_solve", 50, 18, 2, 300) is None
