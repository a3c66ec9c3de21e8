"""The sine / cosine kernels take one line per CTA when a call has few channels
and several when it has many (dct_kernels.cuh, lines_per_cta): a channel's
result must not depend on which."""
import pytest
import torch


def channels(n, N, dtype):
    g = torch.Generator().manual_seed(n + N)
    x = torch.randn(n, N, 2, generator=g, dtype=torch.float64)
    return torch.view_as_complex(x).to(dtype).cuda()


# 152 SMs: one line per CTA up to 152 channels, two up to 304, and the most a CTA holds beyond
@pytest.mark.gpu
@pytest.mark.parametrize("N", [256, 768, 1024, 2048, 4352])
def test_result_independent_of_lines_per_cta(lib, N):
    # l = 0: T_0 is the identity, so the FP64 call is the sine transform alone
    # l = 0, 1 on the split plan: its contraction sums each channel in a fixed order
    plan = lib.Plan(N, 0.1 * N, 1, tf32x3=False, fast_split=True)
    for dtype, ls in ((torch.complex128, (0,)), (torch.complex64, (0, 1))):
        x = channels(17 * 152 + 1, N, dtype)
        for l in ls:
            b = plan.forward(l, x)
            y = plan.inverse(l, b)
            for n in (1, 152, 153, 305):
                assert torch.equal(plan.forward(l, x[:n]), b[:n]), (dtype, l, n)
                assert torch.equal(plan.inverse(l, b[:n].contiguous()), y[:n]), (dtype, l, n)
    plan.close()
