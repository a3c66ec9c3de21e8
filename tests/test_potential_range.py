"""Any finite potential is a phase (tdse.cu, tdse3d.cu), a hard wall at the largest FP64
number too: where steps share an angular pass, the two half steps' angles are one factor
tau on V, not a sum of two potentials.

A constant potential V multiplies the free propagation by exp(-i V tau) a step; the angle
V tau / 2 is rounded once and its sine and cosine are exact to rounding, so only the
products round: 1e-12 for five steps."""
import numpy as np
import pytest
import torch

TAU, STEPS = 0.05, 5


def phase(V):
    a = V * (0.5 * TAU)
    return complex(np.cos(a), -np.sin(a)) ** (2 * STEPS)


def state(nchan, N):
    g = torch.Generator().manual_seed(nchan)
    x = torch.view_as_complex(torch.randn(nchan, N, 2, generator=g, dtype=torch.float64)).cuda()
    return (x / torch.linalg.vector_norm(x)).contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("V", [3.0, -1.2e308, float(np.finfo(np.float64).max)])
@pytest.mark.parametrize("velocity", [False, True])
def test_constant_potential(lib, V, velocity):
    N, L = 512, 5
    plan = lib.Plan(N, 0.1 * N, L, tf32x3=False, fast64=True)
    E = torch.zeros(STEPS, dtype=torch.float64, device="cuda")
    for make, field, nchan in ((lambda: lib.Tdse(plan, L, TAU), E, L),
                               (lambda: lib.Tdse3d(plan, L, 1, TAU), torch.zeros(STEPS, 3, dtype=torch.float64, device="cuda"), 3 * L)):
        out = []
        for v in (0.0, V):
            t = make()
            t.set_potential(np.full(N, v))
            psi = state(nchan, N)
            (t.propagate_velocity if velocity else t.propagate)(psi, field, STEPS)
            out.append(psi)
            t.close()
        assert (out[1] - out[0] * phase(V)).abs().max().item() < 1e-12
    plan.close()
