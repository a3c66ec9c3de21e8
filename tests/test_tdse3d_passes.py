"""The angular passes of the all-m propagator (tdse3d.cu: exact digits per m, phi sums by
pairs of m and of angles, mirror pairs of nodes, adjacent half steps in one pass)
against the step written out with explicit matrices and the plan's kinetic step, at
the edges of the 16-row blocks and of M, and the gradient against central differences
of the written-out step.

Bound: a step is two unitary products of at most 800 channels, phases of a few
radians and two FFTs of 256 points, each operation rounding at 2^-53 and the P^m
orthogonal to 5e-15: below 3e-14 a step, 1e-13 for three steps.  Fourth-order
central differences of step 1e-3: rounding 1e-13 / 1e-3, truncation below that."""
import math

import pytest
import torch

N, DR, TAU = 256, 0.1, 0.05


def explicit(lib, plan, t3, L, M):
    eta = None
    P = []
    for m in range(M + 1):
        td = lib.Tdse(plan, L, TAU, m=m)
        eta, _, p = td.angular()
        P.append(torch.from_numpy(p).cuda())
        td.close()
    eta = torch.from_numpy(eta).cuda()
    NM = 2 * M + 1
    phi = 2 * math.pi * torch.arange(NM, dtype=torch.float64, device="cuda") / NM
    Y = torch.stack([(P[abs(m)][l - abs(m)][:, None] * torch.exp(1j * m * phi)).reshape(-1) / math.sqrt(NM)
                     for l, m in t3.channels], 1)
    st = torch.sqrt(torch.clamp(1 - eta * eta, min=0))
    n = torch.stack([(st[:, None] * torch.cos(phi)).reshape(-1), (st[:, None] * torch.sin(phi)).reshape(-1),
                     (eta[:, None] * torch.ones_like(phi)).reshape(-1)])
    counts = [0] * (plan.l_max + 1)
    for l, _ in t3.channels:
        counts[l] += 1
    r = (torch.arange(N, dtype=torch.float64, device="cuda") + 0.5) * DR
    V = -1.0 / torch.sqrt(r * r + 0.5)

    def run(psi, F, nsteps, hold):
        for s in range(nsteps):
            ph = torch.exp(-0.5j * TAU * (V + (F[s // hold] @ n)[:, None] * r))
            psi = Y.conj().T @ (ph * (Y @ psi))
            psi = plan.kinetic_grouped(counts, psi.contiguous(), TAU)
            psi = Y.conj().T @ (ph * (Y @ psi))
        return psi

    return run, V, r


def state(nchan, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.view_as_complex(torch.randn(nchan, N, 2, generator=g, dtype=torch.float64)).cuda()
    return (x / torch.linalg.vector_norm(x)).contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("L, M", [(1, 0), (1, 2), (2, 1), (5, 3), (16, 1), (17, 2), (31, 0), (32, 8), (32, 12)])
def test_steps(lib, L, M):
    plan = lib.Plan(N, N * DR, L + M, tf32x3=False, fast64=True)
    t3 = lib.Tdse3d(plan, L, M, TAU)
    run, V, _ = explicit(lib, plan, t3, L, M)
    t3.set_potential(V.cpu().numpy())
    F = torch.tensor([[0.3, -0.2, 0.5], [-0.4, 0.6, 0.1]], dtype=torch.float64, device="cuda")
    for nsteps, hold in ((1, 1), (3, 2)):
        psi = state(t3.nchan, L + M + nsteps)
        got = t3.propagate(psi.clone(), F, nsteps, hold)
        assert torch.linalg.vector_norm(got - run(psi, F, nsteps, hold)).item() < 1e-13
    free = t3.propagate(psi.clone(), None, 2)
    assert torch.linalg.vector_norm(free - run(psi, torch.zeros(2, 3, dtype=torch.float64, device="cuda"), 2, 1)).item() < 1e-13
    t3.close()
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("L, M, nsteps, hold, K", [(3, 0, 1, 1, 1), (4, 1, 5, 2, 2), (7, 2, 4, 1, 9)])
def test_gradient(lib, L, M, nsteps, hold, K):
    plan = lib.Plan(N, N * DR, L + M, tf32x3=False, fast64=True)
    t3 = lib.Tdse3d(plan, L, M, TAU)
    run, V, r = explicit(lib, plan, t3, L, M)
    t3.set_potential(V.cpu().numpy())
    ns = -(-nsteps // hold)
    F = torch.linspace(-0.6, 0.7, 3 * ns, dtype=torch.float64, device="cuda").reshape(ns, 3)
    psi = state(t3.nchan, L + M)
    O, g = t3.gradient(psi, F, nsteps, hold, 9.0, K)

    def obs(f):
        return (run(psi, f, nsteps, hold)[:, r > 9.0].abs() ** 2).sum().item()

    assert abs(O.item() - obs(F)) < 1e-12
    h = 1e-3
    for k in range(ns):
        for c in range(3):
            d = torch.zeros_like(F)
            d[k, c] = h
            fd = (8 * (obs(F + d) - obs(F - d)) - (obs(F + 2 * d) - obs(F - 2 * d))) / (12 * h)
            assert abs(g[k, c].item() - fd) < 1e-9 * max(1.0, abs(fd)), (k, c, g[k, c].item(), fd)
    t3.close()
    plan.close()
