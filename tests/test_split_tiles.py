"""Interval-scheme contractions (fast_split.cu) take column tiles of 64, 128 or 256
lines by the groups' sizes, and 64-row or 256-row boxes by a tile's lines; dense
contractions (gemm_tf32x3.cu) tiles of 128 or 256 lines; the FP16-pair split of caller data (capi.cu) takes 16-byte or 4-byte loads by the
pointer.  A channel's sums are formed in the same order in each, so its result is
the same bits."""
import pytest
import torch


def channels(n, N, dtype):
    g = torch.Generator().manual_seed(n + N)
    x = torch.randn(n, N, 2, generator=g, dtype=torch.float64)
    return (torch.view_as_complex(x) if dtype.is_complex else x[..., 0]).to(dtype).cuda()


# 321 lines: one full tile of 256 and one of 65 (complex: 642 lines)
@pytest.mark.gpu
@pytest.mark.parametrize("N", [256, 1280, 2048])
@pytest.mark.parametrize("dtype,sizes", [(torch.float32, (1, 63, 64, 65, 128, 129, 192, 193, 256, 257)),
                                         (torch.complex64, (1, 32, 33, 64, 65, 96, 97, 128, 129))])
@pytest.mark.parametrize("fast", [True, False])
def test_result_independent_of_column_tiles(lib, N, dtype, sizes, fast):
    plan = lib.Plan(N, 0.1 * N, 3, tf32x3=not fast, fast_split=fast)
    x = channels(321, N, dtype)
    b = plan.forward(3, x)
    y = plan.inverse(3, b)
    assert torch.linalg.vector_norm(y - x) / torch.linalg.vector_norm(x) < 1e-5   # F T and back
    for n in sizes:
        assert torch.equal(plan.forward(3, x[:n]), b[:n]), n
        assert torch.equal(plan.inverse(3, b[:n]), y[:n]), n
        # the same channels as the last of three groups
        bc = plan.forward_grouped([2, 0, 5, n], torch.cat([x[:2], x[:5], x[:n]]))
        assert torch.equal(bc[7:], b[:n]), n
        assert torch.equal(plan.inverse_grouped([2, 0, 5, n], bc)[7:], y[:n]), n
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("N", [256, 768, 8192])
@pytest.mark.parametrize("dtype", [torch.float32, torch.complex64])
def test_split_of_unaligned_channels(lib, N, dtype):
    plan = lib.Plan(N, 0.1 * N, 2, tf32x3=False, fast_split=True)
    b = channels(9, N, dtype)
    b[3] = 0                        # no norm: scale 1
    b[5] *= 1e-15                   # a power-of-two scale far from 1
    ref = plan.inverse(2, b)
    assert not ref[3].any()
    nrm = torch.linalg.vector_norm
    back = plan.forward(2, ref[5:6])
    assert nrm((back - b[5]) * 1e15) / nrm(b[5] * 1e15) < 1e-5
    store = torch.empty(9 * N + 4, dtype=dtype, device="cuda")
    for off in (1, 2, 3):
        v = store[off:off + 9 * N].view(9, N)
        v.copy_(b)
        assert torch.equal(plan.inverse(2, v), ref), off
    plan.close()
