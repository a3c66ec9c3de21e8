"""FP32 sine / cosine transforms scale by no common factor: their scale is folded into the
post-twiddle table in double precision (plan.cu), so each entry rounds for itself, where
one factor rounded to FP32 makes every output up to 6e-8 too large or too small.

l = 0: T_0 is the identity, and its products in split TF32 are exact.  The common factor
of a result y against the exact e is <y, e> / <e, e>.  What the FFT's own constants make of
it is the same in both directions, so the two directions' factors differ by the scales'
roundings and by those of the tables' N entries, 3e-8 each at random: below 2e-8."""
import math

import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("N", [768, 4864, 5376, 6400, 7424])
def test_no_common_factor(lib, N):
    plan = lib.Plan(N, 0.1 * N, 0, fp64=False)
    g = torch.Generator().manual_seed(N)
    x = torch.view_as_complex(torch.randn(64, N, 2, generator=g)).cuda()
    i = torch.arange(N, device="cuda")
    F = torch.sin(((i + 1)[:, None] * (2 * i + 1)[None, :] % (4 * N)).to(torch.float64) * (math.pi / (2 * N)))
    F *= math.sqrt(2.0 / N)
    F[N - 1] *= math.sqrt(0.5)
    F, x64 = F.to(torch.complex128), x.to(torch.complex128)
    factor = []
    for y, e in ((plan.forward(0, x), x64 @ F.T), (plan.inverse(0, x), x64 @ F)):
        y = y.to(torch.complex128)
        assert torch.linalg.vector_norm(y - e) / torch.linalg.vector_norm(e) < 1e-6
        factor.append(((y.conj() * e).sum().real / (e.abs() ** 2).sum()).item())
    assert abs(factor[0] - factor[1]) < 2e-8
    plan.close()
