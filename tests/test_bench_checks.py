"""The comparison by which the benchmark checks its pipelined run against the whole batch."""
import torch

import bench


def test_results_that_differ_by_the_order_of_partial_sums_are_the_same_and_others_are_not():
    g = torch.Generator().manual_seed(1)
    a = torch.randn(1, 4, 300, 128, generator=g)
    assert bench.same_result(a, a.clone())
    assert bench.same_result(a * (1 + 3e-4 * torch.randn(a.shape, generator=g)), a)
    assert bench.same_result((a * (1 + 1e-4)).bfloat16(), a.bfloat16())
    one = a.clone()
    one[0, 1, 7, 5] += 0.05
    assert not bench.same_result(one, a)
    assert not bench.same_result(a * 1.005, a)
    assert not bench.same_result(a.roll(1, dims=2), a)
