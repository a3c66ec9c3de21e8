"""FP64 calls on lines near the smallest normal number and below it (mm64.cuh): they go
through as larger ones do, up to the spacing 2^-1074 of what FP64 can hold there.

Bound: every operation rounds at 2^-1075 or at 2^-53 of its value; the inverse's
unnormalised FFT adds up N of its inputs' roundings, and its stages and the contraction
no more than as many again: 4 N 2^-1074 in all."""
import math

import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("N, fast", [(512, True), (768, False)])
@pytest.mark.parametrize("nchan", [1, 9])
def test_lines_below_the_normal_numbers(lib, N, fast, nchan):
    l = 3
    plan = lib.Plan(N, 0.1 * N, l, tf32x3=False, fast64=fast)
    g = torch.Generator().manual_seed(nchan)
    x = torch.view_as_complex(torch.randn(nchan, N, 2, generator=g, dtype=torch.float64)).cuda()
    x /= torch.linalg.vector_norm(x, dim=1, keepdim=True)
    b, y = plan.forward(l, x), plan.inverse(l, x)
    for k in range(-1030, -1010):
        small = x * math.ldexp(1.0, -1000) * math.ldexp(1.0, k + 1000)
        for got, want in ((plan.forward(l, small), b), (plan.inverse(l, small), y)):
            got = got * math.ldexp(1.0, 1000) * math.ldexp(1.0, -k - 1000)
            assert (got - want).abs().max().item() < 4 * N * math.ldexp(1.0, -1074 - k), k
    plan.close()
