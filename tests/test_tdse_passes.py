"""The angular passes of the fixed-m propagator (tdse.cu: exact digits, mirror pairs
of nodes, adjacent half steps in one pass) against the step written out with the
propagator's own P and the plan's kinetic step, for channel counts at the edges of
the 16-row blocks, and the gradient against that of the written-out step.

Bound: a step is two orthogonal L x L products, phases of at most a few radians and
two FFTs of 256 points, each operation rounding at 2^-53: below 1e-14 a step of the
state's norm, 1e-13 for the steps below.  The gradient is compared with fourth-order
central differences of step 1e-3: rounding 1e-13 / 1e-3, truncation below that."""
import pytest
import torch

N, DR, TAU = 256, 0.1, 0.05


def written_out(plan, td, L, m, psi, E, nsteps, hold, sign=1.0):
    _, _, P = td.angular()
    eta = torch.from_numpy(td.angular()[0]).cuda()
    P = torch.from_numpy(P).cuda().to(torch.complex128)
    r = (torch.arange(N, dtype=torch.float64, device="cuda") + 0.5) * DR
    V = -1.0 / torch.sqrt(r * r + 0.5)
    counts = [0] * (plan.l_max + 1)
    for l in range(m, m + L):
        counts[l] = 1

    def half(x, e):
        return P @ (torch.exp(-0.5j * sign * TAU * (V + e * r * eta[:, None])) * (P.T @ x))

    order = range(nsteps) if sign > 0 else range(nsteps - 1, -1, -1)
    for s in order:
        psi = half(plan.kinetic_grouped(counts, half(psi, E[s // hold]), sign * TAU), E[s // hold])
    return psi


def state(L, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.view_as_complex(torch.randn(L, N, 2, generator=g, dtype=torch.float64)).cuda()
    return (x / torch.linalg.vector_norm(x)).contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("L, m", [(1, 0), (2, 0), (7, 1), (15, 0), (16, 2), (17, 0), (33, 0), (63, 1), (64, 0)])
def test_steps(lib, L, m):
    plan = lib.Plan(N, N * DR, 64, tf32x3=False, fast64=True)
    td = lib.Tdse(plan, L, TAU, m=m)
    E = torch.tensor([0.3, -0.2, 0.7], dtype=torch.float64, device="cuda")
    for nsteps, hold in ((1, 1), (2, 1), (5, 2)):
        psi = state(L, 3 * L + nsteps)
        got = td.propagate(psi.clone(), E, nsteps, hold)
        assert torch.linalg.vector_norm(got - written_out(plan, td, L, m, psi, E.cpu(), nsteps, hold)).item() < 1e-13
        back = td.propagate(got.clone(), E, nsteps, hold, backward=True)
        assert torch.linalg.vector_norm(back - psi).item() < 1e-13
    # no steps: the state stays
    psi = state(L, 1)
    assert torch.equal(td.propagate(psi.clone(), E, 0, 1), psi)
    td.close()
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("L, nsteps, hold, K", [(3, 1, 1, 1), (9, 6, 1, 2), (16, 7, 2, 3), (17, 5, 5, 20), (33, 6, 3, 1)])
def test_gradient(lib, L, nsteps, hold, K):
    plan = lib.Plan(N, N * DR, 40, tf32x3=False, fast64=True)
    td = lib.Tdse(plan, L, TAU)
    ns = -(-nsteps // hold)
    E = torch.linspace(0.5, -0.8, ns, dtype=torch.float64)
    psi = state(L, L + K)
    O, g = td.gradient(psi, E.cuda(), nsteps, hold, 9.0, K)
    r = (torch.arange(N, dtype=torch.float64, device="cuda") + 0.5) * DR

    def obs(e):
        return (written_out(plan, td, L, 0, psi, e, nsteps, hold)[:, r > 9.0].abs() ** 2).sum().item()

    assert abs(O.item() - obs(E)) < 1e-12
    h = 1e-3
    for k in range(ns):   # fourth-order central differences: error h^4 f^(5) / 30, rounding 1e-14 / h
        d = torch.zeros(ns, dtype=torch.float64)
        d[k] = h
        fd = (8 * (obs(E + d) - obs(E - d)) - (obs(E + 2 * d) - obs(E - 2 * d))) / (12 * h)
        assert abs(g[k].item() - fd) < 1e-9 * max(1.0, abs(fd)), (k, g[k].item(), fd)
    td.close()
    plan.close()
