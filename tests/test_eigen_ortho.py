"""The Gram-Schmidt step of the bound-state solver over a cluster of CTAs (eigen.cu),
columns in shared memory or in place, against the step written out with the plan's own
transforms: after n steps the states are orthonormal and equal the written-out ones.

Bound: a step is two FFTs, two contractions and ns projections, each rounding at 2^-53
of the norm; the projections amplify by the inverse of a state's part outside the lower
ones (above 1e-2 for random starts of at most 6 states here): 1e-12 for three steps."""
import numpy as np
import pytest
import torch


def written_out(plan, l, U, psi, tau, nsteps):
    u = torch.exp(-0.5 * tau * torch.from_numpy(U).cuda())
    k = torch.from_numpy(plan.get_k(l)).cuda()

    def mgs(x):
        x = list(x)
        norms = []
        for s in range(len(x)):
            for t in range(s):
                x[s] = x[s] - (x[s] @ x[t]) * x[t]
            norms.append(torch.linalg.vector_norm(x[s]))
            x[s] = x[s] / norms[-1]
        return torch.stack(x), torch.stack(norms)

    x, _ = mgs(psi)
    for _ in range(nsteps):
        b = plan.forward(l, (x * u).contiguous()) * torch.exp(-0.5 * tau * k * k)
        x, norms = mgs(plan.inverse(l, b.contiguous()) * u)
    return x, -torch.log(norms) / tau


# clusters of 2, 4 and 8 CTAs; 40 states of 2048 points and 64 of 8192 do not fit shared memory
@pytest.mark.gpu
@pytest.mark.parametrize("N, l, ns", [(256, 0, 1), (512, 3, 5), (768, 1, 4), (1024, 2, 6), (2048, 1, 5)])
def test_states(lib, N, l, ns):
    plan = lib.Plan(N, 0.1 * N, l, tf32x3=False)
    r = (np.arange(N) + 0.5) * 0.1
    U = -1.0 / r
    g = torch.Generator().manual_seed(N + ns)
    psi = torch.randn(ns, N, generator=g, dtype=torch.float64).cuda()
    ref, ref_lev = written_out(plan, l, U, psi, 0.05, 3)
    lev, _ = plan.radial_states(l, U, psi, 0.05, 3)
    assert (psi - ref).abs().max().item() < 1e-12
    assert np.abs(lev - ref_lev.cpu().numpy()).max() < 1e-10   # 1e-12 / tau and the norm's part
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("N, ns", [(256, 64), (2048, 64), (8192, 64)])
def test_many_states_orthonormal(lib, N, ns):
    plan = lib.Plan(N, 0.1 * N, 0, tf32x3=False)
    g = torch.Generator().manual_seed(N)
    psi = torch.randn(ns, N, generator=g, dtype=torch.float64).cuda()
    plan.radial_states(0, np.zeros(N), psi, 1e-4, 1)
    gram = psi @ psi.T
    assert (gram - torch.eye(ns, dtype=torch.float64, device="cuda")).abs().max().item() < 1e-12
    plan.close()
