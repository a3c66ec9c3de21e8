"""FP64 sine / cosine transforms on the longest grids (dct64.cu): a line lies on 8, 4 or
2 CTAs, or on one up to 4096 points, by the number of channels.  Every count of channels
is served, with the same bits, and the transform is the explicit matrix's.

Bound of |F x - y| / ||x|| (max over a channel): log2 N + sqrt(N) roundings at 2^-53
adding at random (the matrix product has the most), 1.2e-14 at N = 8192, times four."""
import math

import pytest
import torch


def channels(n, N, dtype):
    g = torch.Generator().manual_seed(n + N)
    x = torch.randn(n, N, 2, generator=g, dtype=torch.float64)
    return (torch.view_as_complex(x) if dtype.is_complex else x[..., 0]).contiguous().cuda()


@pytest.mark.gpu
@pytest.mark.parametrize("N", [4096, 8192])
@pytest.mark.parametrize("dtype", [torch.float64, torch.complex128])
def test_any_number_of_channels(lib, N, dtype):
    plan = lib.Plan(N, 0.1 * N, 0, tf32x3=False)   # l = 0: T_0 is the identity
    x = channels(160, N, dtype)
    b = plan.forward(0, x)
    i = torch.arange(N, device="cuda")
    F = torch.sin(((i + 1)[:, None] * (2 * i + 1)[None, :] % (4 * N)).to(torch.float64) * (math.pi / (2 * N)))
    F *= math.sqrt(2.0 / N)
    F[N - 1] *= math.sqrt(0.5)
    ref = x @ F.T.to(dtype)
    assert ((b - ref).abs().amax(1) / torch.linalg.vector_norm(x, dim=1)).max().item() < 5e-14
    y = plan.inverse(0, b)
    assert ((y - x).abs().amax(1) / torch.linalg.vector_norm(x, dim=1)).max().item() < 5e-14
    # 8 n, 4 n, 2 n CTAs up to 152, and the counts beyond each
    for n in (1, 19, 20, 38, 39, 76, 77, 152, 153):
        assert torch.equal(plan.forward(0, x[:n]), b[:n]), n
        assert torch.equal(plan.inverse(0, b[:n]), y[:n]), n
    if dtype.is_complex:
        k = plan.kinetic_grouped([160], x, 0.05)
        assert torch.equal(plan.kinetic_grouped([76], x[:76], 0.05), k[:76])
    plan.close()
