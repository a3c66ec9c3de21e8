"""What the performance of this library is measured on: the calls that programs make of it.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (plan,
propagator, inputs), ``run`` is one pass through the public entry points, ``work`` what that pass
cannot do without, ``exact`` the same outputs in 64 bits by plain torch.  Kinds of cases:

  transform   one grouped call (or a forward + inverse pair) on channels of all l
  tdse        split-operator steps of a state of fixed m (both gauges)
  gradient    an observable of the propagated state and its gradient over the field samples
  tdse3d      split-operator steps with all m and a field of any direction
  states      bound states of one l by imaginary time
  batch       the kinetic step of transforms on several grids, replayed as a CUDA graph

Plans by ``scheme``: "split" the FP16-pair interval scheme (FP32 / complex64 calls), "default" a plan
without options (dense split-TF32 factors and dense FP64 ones), "fast64" the O(N l log N) FP64 scheme,
"fp64" dense FP64 factors (the only FP64 form of grids whose N / 64 is no power of two).
"""
import math

import numpy as np
import torch

from paper_1509_07115_gb300 import dsbt

DR = 0.1          # radial step of every case
TAU = 0.05        # time step
NTERMS = 8        # Gaussians of an input function
DTYPES = {"c64": torch.complex64, "f32": torch.float32, "c128": torch.complex128, "f64": torch.float64}
BYTES = {"c64": 8, "f32": 4, "c128": 16, "f64": 8}


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one molecule-sized basis on a short grid, where launches and host time count
        dict(name="forward_c64_n256", kind="transform", op="forward", scheme="split", dtype="c64", N=256, l_max=4,
             batch=1, ragged=False),
        # a propagator's kinetic step on one wavefunction with all m (1024 channels)
        dict(name="kinetic_c64_n2048", kind="transform", op="kinetic", scheme="split", dtype="c64", N=2048, l_max=31,
             batch=1, ragged=False),
        # the same for eight wavefunctions at the benchmark's size (32768 channels, 1 GiB each way)
        dict(name="kinetic_c64_n4096_x8", kind="transform", op="kinetic", scheme="split", dtype="c64", N=4096,
             l_max=63, batch=8, ragged=False),
        # real coefficients back to the radial grid, a grid of 25 * 256 points, uneven channel counts
        dict(name="inverse_f32_n6400_ragged", kind="transform", op="inverse", scheme="split", dtype="f32", N=6400,
             l_max=24, batch=4, ragged=True),
        # a plan made without options, complex64: the dense split-TF32 factors
        dict(name="forward_c64_default_plan", kind="transform", op="forward", scheme="default", dtype="c64", N=1024,
             l_max=16, batch=2, ragged=False),
        # double precision analysis and synthesis of one wavefunction (1024 channels)
        dict(name="round_trip_c128_n2048", kind="transform", op="round_trip", scheme="fast64", dtype="c128", N=2048,
             l_max=31, batch=1, ragged=False),
        # double precision kinetic step on a grid that only the dense FP64 factors serve (5 * 256 points)
        dict(name="kinetic_c128_n1280", kind="transform", op="kinetic", scheme="fp64", dtype="c128", N=1280,
             l_max=20, batch=1, ragged=False),
        # strong-field propagation of an m = 0 state, l < 64, soft Coulomb potential, length gauge
        dict(name="tdse_n2048_l64", kind="tdse", scheme="fast64", N=2048, L=64, m=0, gauge="length", nsteps=40,
             hold=2),
        # one iteration of pulse shaping: ionisation beyond a radius and its gradient over the field samples
        dict(name="tdse_gradient_n1024_l32", kind="gradient", scheme="fast64", N=1024, L=32, m=0, nsteps=24, hold=2,
             every=6),
        # all m, a field that turns: 544 channels
        dict(name="tdse3d_n2048_544", kind="tdse3d", scheme="fast64", N=2048, L=32, M=8, gauge="length", nsteps=4,
             hold=2),
        # hydrogen's lowest s states by imaginary time (the radial grid of the published tables, dr = 0.1)
        dict(name="states_n1024", kind="states", scheme="fp64", N=1024, l=0, nstates=4, nsteps=100),
        # twelve transforms of different grids and l_max as one captured kinetic step
        dict(name="batch_12_grids", kind="batch", transforms=12, n_top=8192, l_top=64, pick=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["transform"] * 6 + ["tdse", "tdse", "gradient", "tdse3d", "states", "batch"])
    if kind == "transform":
        scheme = rng.choice(["split", "split", "split", "default", "fast64", "fp64"])
        dtype = rng.choice(["c64", "c64", "f32"]) if scheme == "split" else \
            rng.choice(["c64", "c128"]) if scheme == "default" else rng.choice(["c128", "c128", "f64"])
        op = rng.choice(["forward", "inverse", "round_trip"] + (["kinetic"] * 3 if dtype[0] == "c" else []))
        if scheme == "split":
            N, l_max = 256 * _log_int(rng, 1, 32), _log_int(rng, 2, 64)
        elif scheme == "fast64":
            N, l_max = 1 << rng.randint(8, 12), _log_int(rng, 2, 40)
        else:
            N, l_max = 256 * _log_int(rng, 1, 8), _log_int(rng, 2, 24)
        # real elements of one array: the span of the listed sizes in this precision
        most = (1 << 26) if scheme == "split" else (1 << 22)
        batch = max(1, min(16, most // (2 * (l_max + 1) ** 2 * N)))
        return dict(kind=kind, op=op, scheme=scheme, dtype=dtype, N=N, l_max=l_max, batch=rng.randint(1, batch),
                    ragged=rng.random() < 0.5)
    if kind == "tdse":
        fast = rng.random() < 0.75
        N = 1 << rng.randint(9, 11) if fast else 256 * rng.choice([3, 5, 6, 7])
        return dict(kind=kind, scheme="fast64" if fast else "fp64", N=N, L=_log_int(rng, 8, 60), m=rng.choice([0, 0, 1, 2]),
                    gauge=rng.choice(["length", "velocity"]), nsteps=rng.randint(5, 40), hold=rng.randint(1, 4))
    if kind == "gradient":
        return dict(kind=kind, scheme="fast64", N=1 << rng.randint(8, 10), L=_log_int(rng, 6, 40), m=0,
                    nsteps=rng.randint(6, 24), hold=rng.randint(1, 3), every=rng.randint(2, 8))
    if kind == "tdse3d":
        return dict(kind=kind, scheme="fast64", N=1 << rng.randint(8, 11), L=rng.randint(4, 28), M=rng.randint(1, 7),
                    gauge=rng.choice(["length", "velocity"]), nsteps=rng.randint(2, 5), hold=rng.randint(1, 2))
    if kind == "states":
        return dict(kind=kind, scheme="fp64", N=256 * rng.randint(1, 6), l=rng.randint(0, 3), nstates=rng.randint(1, 6),
                    nsteps=rng.randint(40, 160))
    return dict(kind=kind, transforms=rng.randint(3, 10), n_top=256 * rng.randint(6, 16), l_top=rng.randint(12, 48),
                pick=rng.randint(1, 1 << 20))


# ------------------------------------------------------------------ inputs

def counts_of(case):
    """Channels per l: all m times the batch, or (ragged) any number up to that, some l empty."""
    full = [(2 * l + 1) * case["batch"] for l in range(case["l_max"] + 1)]
    if not case["ragged"]:
        return full
    rng = np.random.default_rng(case["N"] + 1000 * case["l_max"] + case["batch"])
    got = [int(rng.integers(0, c + 1)) for c in full]
    got[-1] = max(1, got[-1])
    return got


def functions(gen, x, ls, a_lo, a_hi):
    """Unit-norm complex128 functions sum_j c_j x^(l+1) exp(-a_j x^2), c_j ~ CN(0, 1), a_j ~ LogU[a_lo, a_hi], one
    per entry of ls, on the points x (each Gaussian normalised before the sum): radial wavefunctions, and the
    momentum-space ones, which have the same form."""
    n = len(ls)
    c = torch.randn(n, NTERMS, 2, generator=gen, dtype=torch.float64)
    a = torch.exp(torch.empty(n, NTERMS, dtype=torch.float64).uniform_(math.log(a_lo), math.log(a_hi), generator=gen))
    c, a = torch.view_as_complex(c).cuda(), a.cuda()
    ls = torch.as_tensor(ls, dtype=torch.float64, device="cuda")
    out = torch.empty(n, x.numel(), dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 23) // x.numel())
    for s in range(0, n, step):
        e = min(n, s + step)
        g = (ls[s:e, None, None] + 1) * torch.log(x) - a[s:e, :, None] * (x * x)
        g = torch.exp(g - g.amax(dim=2, keepdim=True))
        g = g / torch.linalg.vector_norm(g, dim=2, keepdim=True)
        z = torch.complex((c.real[s:e, :, None] * g).sum(1), (c.imag[s:e, :, None] * g).sum(1))
        out[s:e] = z / torch.linalg.vector_norm(z, dim=1, keepdim=True)
    return out


def grid(N):
    return (torch.arange(N, dtype=torch.float64, device="cuda") + 0.5) * DR


def momenta(N):
    return (torch.arange(N, dtype=torch.float64, device="cuda") + 1) * (math.pi / (N * DR))


def channels(case, seed):
    """(counts, input array) of a transform case."""
    counts = counts_of(case)
    gen = torch.Generator().manual_seed(seed)
    ls = np.repeat(np.arange(len(counts)), counts)
    if case["op"] == "inverse":   # coefficients: k^(l+1) exp(-k^2 / 4a)
        x = functions(gen, momenta(case["N"]), ls, 0.05, 5.0)
    else:
        x = functions(gen, grid(case["N"]), ls, 0.05, 5.0)
    if case["dtype"] in ("f32", "f64"):
        x = x.real.contiguous()
    return counts, x.to(DTYPES[case["dtype"]])


def wave(gen, N, ls):
    """A normalised state over channels ls, the higher ones weaker, some ten atomic units wide."""
    psi = functions(gen, grid(N), ls, 0.01, 0.5)
    psi *= torch.as_tensor([0.6 ** i for i in range(len(ls))], dtype=torch.float64, device="cuda")[:, None]
    return (psi / torch.linalg.vector_norm(psi)).contiguous()


def pulse(gen, n, amplitude, width=None):
    """Field samples under a sin^2 envelope (width: components per sample)."""
    env = torch.sin(math.pi * (torch.arange(n, dtype=torch.float64) + 0.5) / n) ** 2
    u = torch.empty((n,) if width is None else (n, width), dtype=torch.float64).uniform_(-1, 1, generator=gen)
    return (amplitude * u * (env if width is None else env[:, None])).cuda()


def samples_of(case):
    return -(-case["nsteps"] // case["hold"])


def channels3d(L, M):
    return [(l, m) for l in range(M + L) for m in range(-M, M + 1) if abs(m) <= l <= abs(m) + L - 1]


def soft_coulomb(N):
    r = grid(N)
    return -1.0 / torch.sqrt(r * r + 0.5)


def bound_inputs(case, seed):
    gen = torch.Generator().manual_seed(seed)
    N = case["N"]
    r = grid(N)
    guess = functions(gen, r, [case["l"]] * case["nstates"], 0.005, 0.5).real.contiguous()
    return (-1.0 / r).cpu().numpy(), guess


def batch_list(case):
    rng = np.random.default_rng(case["pick"])
    n = case["transforms"]
    Ns = 256 * rng.integers(2, case["n_top"] // 256 + 1, size=n)
    ls = rng.integers(8, case["l_top"] + 1, size=n)
    return [(int(N), int(l), [2 * k + 1 for k in range(int(l) + 1)]) for N, l in zip(Ns, ls)]


def batch_input(case, seed):
    gen = torch.Generator().manual_seed(seed)
    parts = [functions(gen, grid(N), np.repeat(np.arange(l + 1), c), 0.05, 5.0).to(torch.complex64).reshape(-1)
             for N, l, c in batch_list(case)]
    return torch.cat(parts)


# ------------------------------------------------------------------ what a program holds, and one pass

def plan_for(scheme, N, l_max):
    if scheme == "default":
        return dsbt.Plan(N, N * DR, l_max)
    if scheme == "split":
        return dsbt.Plan(N, N * DR, l_max, fp64=False, tf32x3=False, fast_split=True)
    return dsbt.Plan(N, N * DR, l_max, tf32x3=False, fast64=scheme == "fast64")


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "transform":
        s["plan"] = plan_for(case["scheme"], case["N"], case["l_max"])
        s["counts"], s["x"] = channels(case, seed)
        s["y"] = torch.empty_like(s["x"])
        if case["op"] == "round_trip":
            s["b"] = torch.empty_like(s["x"])
        s["plan"].workspace(sum(s["counts"]), s["x"].dtype)
    elif kind in ("tdse", "gradient"):
        gen = torch.Generator().manual_seed(seed)
        m, L = case["m"], case["L"]
        s["plan"] = plan_for(case["scheme"], case["N"], m + L - 1)
        s["tdse"] = dsbt.Tdse(s["plan"], L, TAU, m=m)
        s["psi"] = wave(gen, case["N"], range(m, m + L))
        s["E"] = pulse(gen, samples_of(case), 0.05)
        if kind == "tdse" and case["gauge"] == "velocity":
            s["A"] = pulse(gen, samples_of(case), 0.25)
        if kind == "gradient":
            s["E"].requires_grad_(True)
    elif kind == "tdse3d":
        gen = torch.Generator().manual_seed(seed)
        L, M = case["L"], case["M"]
        s["plan"] = plan_for(case["scheme"], case["N"], M + L - 1)
        s["tdse"] = dsbt.Tdse3d(s["plan"], L, M, TAU)
        s["tdse"].set_potential(soft_coulomb(case["N"]).cpu().numpy())
        s["psi"] = wave(gen, case["N"], [l for l, _ in channels3d(L, M)])
        s["F"] = pulse(gen, samples_of(case), 0.05, 3)
        if case["gauge"] == "velocity":
            s["A"] = pulse(gen, samples_of(case), 0.25, 3)
    elif kind == "states":
        s["plan"] = plan_for(case["scheme"], case["N"], case["l"])
        s["U"], s["guess"] = bound_inputs(case, seed)
    else:
        s["batch"] = dsbt.Batch(batch_list(case), DR, scheme="interval")
        s["x"] = batch_input(case, seed)
        s["y"] = torch.empty_like(s["x"])
        torch.cuda.synchronize()   # the capture runs the step once on a stream of its own
        s["graph"] = s["batch"].capture_kinetic(s["x"], TAU, s["y"])
    return s


R_CUT = 10.0


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "transform":
        plan, op = s["plan"], case["op"]
        if op == "forward":
            return plan.forward_grouped(s["counts"], s["x"], out=s["y"])
        if op == "inverse":
            return plan.inverse_grouped(s["counts"], s["x"], out=s["y"])
        if op == "kinetic":
            return plan.kinetic_grouped(s["counts"], s["x"], TAU, out=s["y"])
        b = plan.forward_grouped(s["counts"], s["x"], out=s["b"])
        return b, plan.inverse_grouped(s["counts"], b, out=s["y"])
    if kind == "tdse":   # the state goes on from pass to pass, as in a propagation
        if case["gauge"] == "velocity":
            return s["tdse"].propagate_velocity(s["psi"], s["A"], case["nsteps"], case["hold"])
        return s["tdse"].propagate(s["psi"], s["E"], case["nsteps"], case["hold"])
    if kind == "gradient":
        O = dsbt.TdseObservable.apply(s["E"], s["tdse"], s["psi"], case["nsteps"], case["hold"], R_CUT, case["every"])
        return O.detach(), torch.autograd.grad(O, s["E"])[0]
    if kind == "tdse3d":
        if case["gauge"] == "velocity":
            return s["tdse"].propagate_velocity(s["psi"], s["A"], case["nsteps"], case["hold"], F=s["F"])
        return s["tdse"].propagate(s["psi"], s["F"], case["nsteps"], case["hold"])
    if kind == "states":
        psi = s["guess"].clone()
        levels, energies = s["plan"].radial_states(case["l"], s["U"], psi, TAU, case["nsteps"])
        return levels, energies, psi
    s["batch"].launch_graph(s["graph"])
    return s["y"]


# ------------------------------------------------------------------ what a pass cannot do without

def line_flops(N, l):
    """T_l on one real line by the O(N l) form of the transform: 2 l N multiply-adds."""
    return 4.0 * l * N


def fft_flops(N):
    """The sine / cosine transform of one complex channel."""
    return 5.0 * N * math.log2(N)


def kinetic_flops(N, l, lines):
    """F, T, T^T and F^T on `lines` real lines."""
    return 2 * lines * (line_flops(N, l) + fft_flops(N) / 2)


def work(case):
    kind = case["kind"]
    if kind == "transform":
        counts, N = counts_of(case), case["N"]
        per = 2 if case["dtype"][0] == "c" else 1
        passes = 2 if case["op"] in ("kinetic", "round_trip") else 1
        arrays = 4 if case["op"] == "round_trip" else 2
        return {"bytes": arrays * sum(counts) * N * BYTES[case["dtype"]],
                "flops": sum(kinetic_flops(N, l, per * c) for l, c in enumerate(counts)) * passes / 2}
    if kind in ("tdse", "gradient"):
        N, L, m = case["N"], case["L"], case["m"]
        angular = 8.0 * L * L * N   # to the angular grid and back, one complex state
        step = angular + sum(kinetic_flops(N, m + i, 2) for i in range(L))
        if kind == "gradient":   # forward, the segments again, the adjoint steps with their products
            return {"bytes": L * N * 16.0, "flops": case["nsteps"] * (3 * step + angular)}
        if case["gauge"] == "velocity":
            step += angular
        return {"bytes": 2 * L * N * 16.0, "flops": case["nsteps"] * step}
    if kind == "tdse3d":
        N, L, NM = case["N"], case["L"], 2 * case["M"] + 1
        angular = 8.0 * NM * L * L * N + 2 * L * N * 5 * NM * math.log2(max(2, NM))
        ls = [l for l, _ in channels3d(L, case["M"])]
        step = angular * (2 if case["gauge"] == "velocity" else 1) + sum(kinetic_flops(N, l, 2) for l in ls)
        return {"bytes": 2 * len(ls) * N * 16.0, "flops": case["nsteps"] * step}
    if kind == "states":
        N, ns = case["N"], case["nstates"]
        step = kinetic_flops(N, case["l"], ns) + 2.0 * N * ns * (ns + 1)
        return {"bytes": 2 * ns * N * 8.0, "flops": case["nsteps"] * step}
    trs = batch_list(case)
    return {"bytes": sum(2 * N * sum(c) * 8.0 for N, _, c in trs),
            "flops": sum(kinetic_flops(N, l, 2 * n) for N, _, c in trs for l, n in enumerate(c))}


# ------------------------------------------------------------------ the same in 64 bits, by plain torch

def parity(l):
    return 1 if l % 2 == 0 else 0


def factors(N, ls):
    """T_l of every l in ls, [len(ls)][N][N]: rows from the difference equation of the discrete Legendre polynomials
    in x, l(l+1) Q = B (Q(x+1) - Q) - D (Q - Q(x-1)), normalised; the rows n < ceil((l+1)/2) are the polynomials of
    degree 2n - p_l on the whole grid."""
    ls = torch.as_tensor(list(ls), dtype=torch.float64, device="cuda")[:, None]
    p = 1.0 - torch.remainder(ls, 2)
    T = torch.zeros(ls.shape[0], N, N, dtype=torch.float64, device="cuda")
    n = torch.arange(N, dtype=torch.float64, device="cuda")[None, :] + p
    M, top = 2 * n - 1, ls * (ls + 1)
    q, d = torch.ones_like(n), torch.zeros_like(n)
    for x in range(N - 1):
        k = x + 1
        q, d, M = q[:, 1:], d[:, 1:], M[:, 1:]   # rows below the k-th still march
        d = (top * q + x * (x - M - 1) * d) / ((x + 1) * (x - M))
        q = q + d
        torch.diagonal(T, -k, 1, 2).copy_(d)
    torch.diagonal(T, 0, 1, 2).fill_(1.0)
    # completion rows
    rows = int(ls.max().item()) // 2 + 1
    n = torch.arange(rows, dtype=torch.float64, device="cuda")[None, :] + p
    e, M = 2 * n - p, 2 * (N + p - 1)
    q, d = torch.ones_like(n), torch.zeros_like(n)
    C = torch.zeros(ls.shape[0], rows, N, dtype=torch.float64, device="cuda")
    for x in range(N):
        C[:, :, N - 1 - x] = q
        d = (e * (e + 1) * q + x * (x - M - 1) * d) / ((x + 1) * (x - M))
        q = q + d
    extra = n < torch.floor((ls + 2) / 2)
    T[:, :rows] = torch.where(extra[:, :, None], C, T[:, :rows])
    T[:, :, 0] *= torch.sqrt((1 + p) / 2)   # weight of m = 0 (odd l)
    T /= torch.linalg.vector_norm(T, dim=2, keepdim=True)
    return T


def cosine(x):
    """Orthonormal DCT-II along the last axis (complex)."""
    N = x.shape[-1]
    k = torch.arange(N, dtype=torch.float64, device="cuda")
    X = torch.fft.fft(torch.cat([x, x.flip(-1)], -1))[..., :N] * torch.exp(-0.5j * math.pi * k / N) * math.sqrt(0.5 / N)
    X[..., 0] *= math.sqrt(0.5)
    return X


def cosine_back(X):
    """Its transpose."""
    N = X.shape[-1]
    k = torch.arange(N, dtype=torch.float64, device="cuda")
    X = X * math.sqrt(0.5 / N)
    X[..., 0] *= math.sqrt(0.5)
    w = torch.exp(0.5j * math.pi * k / N)
    return torch.fft.ifft(X * w, 2 * N)[..., :N] * (2 * N) + torch.fft.fft(X * w.conj(), 2 * N)[..., :N]


def alternate(N):
    return 1.0 - 2.0 * torch.remainder(torch.arange(N, dtype=torch.float64, device="cuda"), 2)


def fourier(l, x):
    return cosine(x) if l % 2 else cosine(x * alternate(x.shape[-1])).flip(-1)


def fourier_back(l, b):
    return cosine_back(b) if l % 2 else cosine_back(b.flip(-1)) * alternate(b.shape[-1])


def times(A, z):
    """Real A [..][m][n] on complex z [..][c][n] along the last axis."""
    return torch.complex(z.real @ A.transpose(-1, -2), z.imag @ A.transpose(-1, -2))


def forward64(l, T, x):
    return times(T, fourier(l, x))


def inverse64(l, T, b):
    return fourier_back(l, times(T.transpose(-1, -2), b))


def momentum(l, N):
    """k of coefficient s = n - p_l: n dk, the completion rows N dk."""
    n = torch.arange(N, dtype=torch.float64, device="cuda") + parity(l)
    return torch.where(n < (l + 2) // 2, float(N), n) * (math.pi / (N * DR))


def kinetic64(l, T, x, tau):
    k = momentum(l, x.shape[-1])
    return inverse64(l, T, forward64(l, T, x) * torch.exp(-0.5j * tau * k * k))


def transform64(case, counts, x):
    N, real = case["N"], not x.is_complex()
    x = x.to(torch.complex128)
    T = factors(N, range(len(counts)))
    b, y = torch.empty_like(x), torch.empty_like(x)
    c0 = 0
    for l, c in enumerate(counts):
        at = slice(c0, c0 + c)
        c0 += c
        if not c:
            continue
        if case["op"] == "forward":
            y[at] = forward64(l, T[l], x[at])
        elif case["op"] == "inverse":
            y[at] = inverse64(l, T[l], x[at])
        elif case["op"] == "kinetic":
            y[at] = kinetic64(l, T[l], x[at], TAU)
        else:
            b[at] = forward64(l, T[l], x[at])
            y[at] = inverse64(l, T[l], b[at])
    if real:
        b, y = b.real.contiguous(), y.real.contiguous()
    return (b, y) if case["op"] == "round_trip" else y


def angular64(L, m):
    """(eta, P[i][j]) of the L-point Gauss-Legendre rule: normalised associated Legendre functions l = m .. m+L-1
    times the root of the weight, orthonormalised on the rule in order of l."""
    eta, w = np.polynomial.legendre.leggauss(L)
    eta, w = eta[::-1].copy(), w[::-1].copy()
    rows = [np.sqrt(w) * math.sqrt(0.5)]
    for k in range(1, m + 1):
        rows[0] = rows[0] * np.sqrt((2 * k + 1) / (2 * k)) * np.sqrt(1 - eta ** 2)
    if L > 1:
        rows.append(math.sqrt(2 * m + 3) * eta * rows[0])
    for l in range(m + 2, m + L):
        a = math.sqrt((4 * l * l - 1) / (l * l - m * m))
        b = math.sqrt(((l - 1) ** 2 - m * m) / (4 * (l - 1) ** 2 - 1))
        rows.append(a * (eta * rows[-1] - b * rows[-2]))
    Q, R = np.linalg.qr(np.array(rows).T)
    return torch.as_tensor(eta, device="cuda"), torch.as_tensor((Q * np.sign(np.diag(R))).T.copy(), device="cuda")


def to_slots(l, b):
    """Coefficients by momentum n = 1 .. N (odd l: coefficient 0 takes n = N) with the factor (-i)^l s_l."""
    return 1j * torch.roll(b, -1, -1) if l % 2 else b


def from_slots(l, c):
    return torch.roll(-1j * c, 1, -1) if l % 2 else c


def tdse64(case, psi, E, A, tau):
    """All steps of a fixed-m propagation."""
    N, L, m = case["N"], case["L"], case["m"]
    ls = list(range(m, m + L))
    T = factors(N, ls)
    eta, P = angular64(L, m)
    r, V, kt = grid(N), soft_coulomb(N), momenta(N)
    k2 = torch.stack([momentum(l, N) ** 2 for l in ls])

    def half(x, e):
        g = times(P.T, x.T).T
        g = g * torch.exp(-0.5j * tau * (V + e * r * eta[:, None]))
        return times(P, g.T).T

    def each(f, x):
        return torch.stack([f(l, x[i]) for i, l in enumerate(ls)])

    for s in range(case["nsteps"]):
        e = 0.0 if E is None else E[s // case["hold"]]
        x = half(psi, e)
        x = times(T, each(fourier, x)[:, None])[:, 0]
        if A is None:
            x = x * torch.exp(-0.5j * tau * k2)
        else:
            x = each(to_slots, x * torch.exp(-0.25j * tau * k2))
            g = times(P.T, x.T).T * torch.exp(1j * tau * A[s // case["hold"]] * kt * eta[:, None])
            x = each(from_slots, times(P, g.T).T) * torch.exp(-0.25j * tau * k2)
        x = each(fourier_back, times(T.transpose(1, 2), x[:, None])[:, 0])
        psi = half(x, e)
    return psi


def tdse3d64(case, psi, F, A, tau):
    N, L, M = case["N"], case["L"], case["M"]
    NM = 2 * M + 1
    chans = channels3d(L, M)
    T = factors(N, range(M + L))
    P = [angular64(L, m)[1] for m in range(M + 1)]
    eta = angular64(L, 0)[0]
    phi = 2 * math.pi * torch.arange(NM, dtype=torch.float64, device="cuda") / NM
    Y = torch.stack([(P[abs(m)][l - abs(m)][:, None] * torch.exp(1j * m * phi)).reshape(-1) / math.sqrt(NM)
                     for l, m in chans], 1)
    st = torch.sqrt(torch.clamp(1 - eta * eta, min=0))
    n = torch.stack([(st[:, None] * torch.cos(phi)).reshape(-1), (st[:, None] * torch.sin(phi)).reshape(-1),
                     (eta[:, None] * torch.ones_like(phi)).reshape(-1)])
    r, V, kt = grid(N), soft_coulomb(N), momenta(N)
    groups = [(l, [c for c, (k, _) in enumerate(chans) if k == l]) for l in range(M + L)]

    def half(x, f):
        g = Y @ x
        g *= torch.exp(-0.5j * tau * (V + (f @ n)[:, None] * r))
        return Y.conj().T @ g

    for s in range(case["nsteps"]):
        f = F[s // case["hold"]]
        x = half(psi, f)
        if A is None:
            for l, at in groups:
                x[at] = kinetic64(l, T[l], x[at], tau)
        else:
            for l, at in groups:
                x[at] = to_slots(l, forward64(l, T[l], x[at]) * torch.exp(-0.25j * tau * momentum(l, N) ** 2))
            g = Y @ x
            g *= torch.exp(1j * tau * (A[s // case["hold"]] @ n)[:, None] * kt)
            x = Y.conj().T @ g
            for l, at in groups:
                x[at] = inverse64(l, T[l], from_slots(l, x[at]) * torch.exp(-0.25j * tau * momentum(l, N) ** 2))
        psi = half(x, f)
    return psi


def states64(case, U, guess):
    N, l, ns = case["N"], case["l"], case["nstates"]
    T = factors(N, [l])[0]
    U = torch.as_tensor(U, device="cuda")
    u, k = torch.exp(-0.5 * TAU * U), momentum(l, N)

    def orthonormal(x):
        norms = []
        x = list(x)
        for s in range(ns):
            for t in range(s):
                x[s] = x[s] - (x[s] @ x[t]) * x[t]
            norms.append(torch.linalg.vector_norm(x[s]))
            x[s] = x[s] / norms[-1]
        return torch.stack(x), torch.stack(norms)

    x, _ = orthonormal(guess)
    for _ in range(case["nsteps"]):
        b = forward64(l, T, (x * u).to(torch.complex128)) * torch.exp(-0.5 * TAU * k * k)
        x, norms = orthonormal(inverse64(l, T, b).real * u)
    b = forward64(l, T, x.to(torch.complex128)).real
    energies = (0.5 * k * k * b * b).sum(1) + (U * x * x).sum(1)
    return (-torch.log(norms) / TAU).cpu().numpy(), energies.cpu().numpy(), x


def exact(case, seed):
    kind = case["kind"]
    if kind == "transform":
        counts, x = channels(case, seed)
        return transform64(case, counts, x)
    gen = torch.Generator().manual_seed(seed)
    if kind in ("tdse", "gradient"):
        psi = wave(gen, case["N"], range(case["m"], case["m"] + case["L"]))
        E = pulse(gen, samples_of(case), 0.05)
        if kind == "tdse":
            A = pulse(gen, samples_of(case), 0.25) if case["gauge"] == "velocity" else None
            return tdse64(case, psi, E if A is None else None, A, TAU)
        E.requires_grad_(True)
        O = (tdse64(case, psi, E, None, TAU)[:, grid(case["N"]) > R_CUT].abs() ** 2).sum()
        return O.detach(), torch.autograd.grad(O, E)[0]
    if kind == "tdse3d":
        psi = wave(gen, case["N"], [l for l, _ in channels3d(case["L"], case["M"])])
        F = pulse(gen, samples_of(case), 0.05, 3)
        A = pulse(gen, samples_of(case), 0.25, 3) if case["gauge"] == "velocity" else None
        return tdse3d64(case, psi, F, A, TAU)
    if kind == "states":
        return states64(case, *bound_inputs(case, seed))
    x = batch_input(case, seed)
    out, at = [], 0
    for N, l_max, counts in batch_list(case):
        T = factors(N, range(l_max + 1))
        for l, c in enumerate(counts):
            z = x[at:at + c * N].reshape(c, N).to(torch.complex128)
            out.append(kinetic64(l, T[l], z, TAU).reshape(-1))
            at += c * N
        del T
    return torch.cat(out)
