"""FP64 contractions keep the small entries of a line with large ones to 53 bits of their
own (mm64.cuh, to_double): l = 0, where T_0 is the identity and hands the line on as it is,
so what is left of the error is the sine transform's.

Bound of ||y - e|| / ||b||: the FFT's five stages of at most three roundings each and the
scale, at 2^-53 and random: sqrt(16) 2^-53 = 4.5e-16.  Rounding every entry at 2^-56 of the
largest adds sqrt(N / 3) 2^-56 = 7e-16 at N = 8192."""
import math

import numpy as np
import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("nchan", [1, 9])   # real lines: both forms
def test_one_large_entry(lib, nchan):
    N = 8192
    plan = lib.Plan(N, 0.1 * N, 0, tf32x3=False)
    g = torch.Generator().manual_seed(nchan)
    b = (torch.randn(nchan, N, generator=g, dtype=torch.float64) * 1e-5).cuda()
    at = torch.randint(N, (nchan,), generator=g)
    i = torch.arange(N, device="cuda")
    # y_i = sum_n b_n sqrt(2/N) sin((n + 1)(2i + 1) pi / 2N): the small part, then the large entry
    F = torch.sin(((i + 1)[:, None] * (2 * i + 1)[None, :] % (4 * N)).to(torch.float64) * (math.pi / (2 * N)))
    F *= math.sqrt(2.0 / N)
    F[N - 1] *= math.sqrt(0.5)
    b[torch.arange(nchan), at.cuda()] = 0.0
    e = b @ F
    for c in range(nchan):
        n = int(at[c])
        angle = (n + 1) * (2 * np.arange(N) + 1) % (4 * N) * (np.longdouble("3.14159265358979323846264338327950288") / (2 * N))
        big = np.sin(angle) * np.sqrt(np.longdouble(2.0) / N) * (np.sqrt(np.longdouble(0.5)) if n == N - 1 else 1)
        e[c] += torch.from_numpy(big.astype(np.float64)).cuda()
    b[torch.arange(nchan), at.cuda()] = 1.0
    y = plan.inverse(0, b)
    err = torch.linalg.vector_norm(y - e, dim=1) / torch.linalg.vector_norm(b, dim=1)
    assert err.max().item() < 4.5e-16
    plan.close()
