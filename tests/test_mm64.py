"""The FP64 contraction through exact FP16 digits (mm64.cu) against explicit
64-bit matrices: both forms (up to 4 real lines of a group, and more), edges of
the line tiles, of 16 in l and of the interval tree, and the scales of lines.

Bound of |b - T F x| / ||x|| (max over a channel): the FFT and the reference's
matrix products round at 2^-53 per operation with at most log2 N + sqrt(N)
operations adding at random, below 2e-14 for N <= 1024; the digits add less than
2^-58 sqrt(N)."""
import math

import pytest
import torch

TOL = 2e-14


def sine_cosine(N, l):
    """F_l as a matrix: orthonormal DST-II (even l, n = 1..N) or DCT-II (odd l, n = 0..N-1)."""
    i = torch.arange(N, device="cuda")
    n = torch.arange(N, device="cuda") + (1 if l % 2 == 0 else 0)
    # the angle n (2i + 1) pi / 2N, reduced in integers
    angle = (n[:, None] * (2 * i + 1)[None, :] % (4 * N)).to(torch.float64) * (math.pi / (2 * N))
    F = (torch.sin if l % 2 == 0 else torch.cos)(angle) * math.sqrt(2.0 / N)
    F[(n == 0) | (n == N) if l % 2 == 0 else n == 0] *= math.sqrt(0.5)
    return F


def lines(seed, nchan, N, dtype):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(nchan, N, 2, generator=g, dtype=torch.float64).cuda()
    x *= torch.exp(torch.randn(nchan, N, 1, generator=g, dtype=torch.float64).cuda() * 3)   # uneven magnitudes
    return torch.view_as_complex(x).contiguous() if dtype == torch.complex128 else x[..., 0].contiguous()


def rel(a, b, x):
    return ((a - b).abs().amax(-1) / torch.linalg.vector_norm(x, dim=-1)).max().item()


@pytest.mark.gpu
@pytest.mark.parametrize("N, fast", [(256, True), (512, True), (1024, True), (256, False), (768, False)])
def test_against_explicit_matrices(lib, N, fast):
    lmax = 64
    plan = lib.Plan(N, 0.1 * N, lmax, tf32x3=False, fast64=fast)
    for l in (0, 1, 2, 15, 16, 17, 32, 33, 63, 64):
        T, F = plan.get_T(l), sine_cosine(N, l)
        for dtype, counts in ((torch.float64, (1, 2, 3, 5, 16, 17)), (torch.complex128, (1, 2, 3, 9))):
            for n in counts:
                x = lines(l + n, n, N, dtype)
                A = (T @ F).to(dtype)
                assert rel(plan.forward(l, x), x @ A.T, x) < TOL, (l, dtype, n)
                assert rel(plan.inverse(l, x), x @ A, x) < TOL, (l, dtype, n)
    # groups of both forms in one call, and empty ones
    counts = [(0, 1, 2, 9)[l % 4] for l in range(lmax + 1)]
    x = lines(7, sum(counts), N, torch.complex128)
    b, y = plan.forward_grouped(counts, x), None
    y = plan.inverse_grouped(counts, x)
    c0 = 0
    for l, c in enumerate(counts):
        if c:
            A = (plan.get_T(l) @ sine_cosine(N, l)).to(torch.complex128)
            xs = x[c0:c0 + c]
            assert rel(b[c0:c0 + c], xs @ A.T, xs) < TOL, l
            assert rel(y[c0:c0 + c], xs @ A, xs) < TOL, l
        c0 += c
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nchan", [1, 9])
def test_scales_and_nonfinite_lines(lib, nchan):
    """Powers of two pass through exactly (each line has its own scale); zero lines
    give zeros; a line with a NaN gives NaN and leaves the others alone."""
    N, l = 512, 3
    plan = lib.Plan(N, 0.1 * N, l, tf32x3=False, fast64=True)
    x = lines(3, nchan, N, torch.complex128)
    x = torch.where(x.abs() > 1e-2, x, 0)
    b, y = plan.forward(l, x), plan.inverse(l, x)
    for k in (-800, -40, 40, 900):
        s = math.ldexp(1.0, k)
        assert torch.equal(plan.forward(l, x * s), b * s), k
        assert torch.equal(plan.inverse(l, x * s), y * s), k
    tiny = math.ldexp(1.0, -1000)   # below the common path's scales: 2^-1074 is the last bit there
    assert ((plan.inverse(l, x * tiny) / tiny - y).abs().max() / y.abs().max()).item() < 1e-12
    z = torch.zeros_like(x)
    assert torch.equal(plan.forward(l, z), z) and torch.equal(plan.inverse(l, z), z)
    many = lines(4, 3 * nchan, N, torch.complex128)
    ref, back = plan.forward(l, many), plan.inverse(l, many)
    for bad in (float("nan"), float("inf")):
        w = many.clone()
        w[nchan, 77] = bad
        for got, want in ((plan.forward(l, w), ref), (plan.inverse(l, w), back)):
            assert not torch.isfinite(got[nchan].real).any()
            keep = [c for c in range(3 * nchan) if c != nchan]
            assert torch.equal(got[keep], want[keep])
    plan.close()
