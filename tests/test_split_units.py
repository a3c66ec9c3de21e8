"""Interval-scheme contractions (fast_split.cu) of many groups of uneven size: the launch
counts its finished column tiles in the caller's workspace, which holds a counter for each
tile whichever tile width the groups' sizes select.  Each group's result is that of a call
of its own."""
import numpy as np
import pytest
import torch


def uneven(small, large, groups, large_groups):
    return [small] * (groups - large_groups) + [large] * large_groups


def drawn(l_max, batch, seed):
    rng = np.random.default_rng(seed)
    return [int(rng.integers(0, (2 * l + 1) * batch + 1)) for l in range(l_max + 1)]


# 129 real lines: two tiles of 128 and one of 256
@pytest.mark.gpu
@pytest.mark.parametrize("N, dtype, counts", [
    (256, torch.float32, uneven(1, 129, 65, 26)),
    (256, torch.float32, uneven(2, 130, 65, 26)),
    (256, torch.complex64, uneven(1, 65, 65, 26)),
    (768, torch.float32, drawn(62, 5, 768 + 1000 * 62 + 5)),
    (768, torch.float32, uneven(64, 64, 65, 65)),
    (256, torch.float32, uneven(0, 257, 65, 65)),
])
def test_groups_of_uneven_size(lib, N, dtype, counts):
    plan = lib.Plan(N, 0.1 * N, len(counts) - 1, fp64=False, tf32x3=False, fast_split=True)
    g = torch.Generator().manual_seed(sum(counts))
    x = torch.randn(sum(counts), N, 2, generator=g)
    x = (torch.view_as_complex(x) if dtype.is_complex else x[..., 0]).contiguous().cuda()
    b = plan.forward_grouped(counts, x)
    y = plan.inverse_grouped(counts, b)
    c0 = 0
    for l, c in enumerate(counts):
        if c:
            assert torch.equal(plan.forward(l, x[c0:c0 + c]), b[c0:c0 + c]), l
            assert torch.equal(plan.inverse(l, b[c0:c0 + c]), y[c0:c0 + c]), l
        c0 += c
    plan.close()
