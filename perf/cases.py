"""Measured cases of the reconstruction library: what a program built on it calls.

A case is one call (or one autograd forward and backward) through the Python
binding, on inputs and a context that the program already holds. Meshes cover
the library's range (16^3 to 512^3, N = 2^a 3^b); inputs are seeded random
fields with the statistics of the method's own: BBKS linear modes at 10% of
the fiducial power (where a reconstruction starts) or at full power (the
clustered truth), log-normal overdensities and halo masses, particles in
clumps and in between.

``exact`` restates each call in float64 torch. Gradients of this method are
discontinuous where a hidden unit of the network switches or a particle enters
another cell, so a rounding-sized change of the input moves some of their
values by far more than the rounding. The inputs keep that small: the networks
of the gradient cases have biases that hold every ReLU decision away from zero,
and the gradients that enter the PM adjoint are smooth over a few cells, as the
residual's and the features' smoothing makes them. (The plain-TF32 and bfloat16
networks round their operands so coarsely that a rounding-sized change moves
single masses by 4e-3; they are not here.)
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1805_02247_gb300 import pmrecon, synth

MESHES = [16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 162, 192, 216, 256, 288, 324, 384, 432, 486, 512]
OMEGA_M, SIGMA8, GAMMA, A0 = 0.3175, 0.8, 0.21, 0.1
R_M, SIGMA_N2, M_SCALE = 3.0, 0.25, 1e12
NN_FWD, NN_BWD = 2 * (81 * 50 + 50 * 30 + 30), 2 * (30 + 30 * 50 + 50 * 81)


def listed():
    return [
        # the default synthetic problem: the smallest whole evaluation, where launches and latency count
        {"name": "eval_32", "kind": "eval", "N": 32, "L": 100.0, "nsteps": 3, "power": 0.1, "head": 0, "lpt": 1,
         "N_sm": 2.0, "M0": 1e12},
        # the headline benchmark's evaluation: 256^3, 10 steps, the starting point of a reconstruction
        {"name": "eval_256", "kind": "eval", "N": 256, "L": 400.0, "nsteps": 10, "power": 0.1, "head": 0, "lpt": 1,
         "N_sm": 4.0, "M0": 1e12},
        # one L-BFGS iteration of the paper's two-network model with 2LPT, at the mesh of the annealed
        # reconstruction, as the server runs it (own stream, evaluations replayed as a CUDA graph); f_eff counts the
        # smoothed residual's independent points
        {"name": "step_128", "kind": "step", "N": 128, "L": 400.0, "nsteps": 5, "power": 0.1, "head": 1, "lpt": 2,
         "N_sm": 4.0, "M0": 1e12, "f_eff": 0.01},
        # the PM model as a differentiable layer of somebody's own loss, full power (clustered particles)
        {"name": "pm_grad_192", "kind": "pm_grad", "N": 192, "L": 400.0, "nsteps": 5, "power": 1.0, "lpt": 1},
        # the same layer on a small mesh, as a serving job's model calls see it
        {"name": "pm_grad_64", "kind": "pm_grad", "N": 64, "L": 200.0, "nsteps": 5, "power": 0.1, "lpt": 2},
        # halo masses of an evolved density, no gradient
        {"name": "nn_map_256", "kind": "nn_map", "N": 256, "L": 400.0, "head": 0, "path": 0},
        # the network layer's input gradient, two-network head, a mesh whose z lines end in a ragged tile
        {"name": "nn_adjoint_192", "kind": "nn_adjoint", "N": 192, "L": 400.0, "head": 1, "path": 0},
        # one PM force at the largest mesh a context takes
        {"name": "force_512", "kind": "force", "N": 512, "L": 400.0},
        # Gaussian smoothing on a mesh that is not a power of two times 64
        {"name": "smooth_216", "kind": "smooth", "N": 216, "L": 400.0, "R": 4.0},
        # mass-weighted paint of a catalogue in no order: clumped and unwrapped positions, fewer than one per cell
        {"name": "paint_128", "kind": "paint", "N": 128, "L": 400.0, "np": 1500001, "mass": True, "lattice": False},
        # number density of a simulation's particles, listed in the order of their lattice points
        {"name": "paint_256", "kind": "paint", "N": 256, "L": 400.0, "np": 16777216, "mass": False, "lattice": True},
        # the optimiser's two-loop direction with a full memory
        {"name": "direction_192", "kind": "direction", "N": 192, "L": 400.0, "k": 10},
    ]


def draw(rng):
    def mesh(lo, hi):
        n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min((m for m in MESHES if lo <= m <= hi), key=lambda m: abs(math.log(m / n)))

    kind = rng.choice(["eval", "eval", "step", "pm_grad", "nn_map", "nn_adjoint", "force", "smooth", "paint",
                       "direction"])
    hi = {"eval": 256, "step": 144, "pm_grad": 256, "nn_map": 256, "nn_adjoint": 192, "force": 512, "smooth": 512,
          "paint": 256, "direction": 192}[kind]
    N = mesh(16, hi)
    # 200 to 400 Mpc/h boxes, cells no smaller than the benchmark's
    c = {"kind": kind, "N": N, "L": round(rng.uniform(max(200.0, min(400.0, 1.5625 * N)), 400.0), 1)}
    if kind == "eval":
        c.update(nsteps=rng.randint(5, 10), power=0.1, head=rng.choice([0, 0, 1]) if N < 256 else 0,
                 lpt=rng.choice([1, 2]) if N < 256 else 1, N_sm=rng.choice([3.0, 4.0, 6.0]), M0=1e12)
    elif kind == "step":
        c.update(nsteps=rng.randint(3, 8), power=0.1, head=rng.choice([0, 1]), lpt=rng.choice([1, 2]),
                 N_sm=rng.choice([3.0, 4.0]), M0=1e12, f_eff=0.01)
        if N == 144:
            c["nsteps"] = min(c["nsteps"], 4)
    elif kind == "pm_grad":
        c.update(nsteps=rng.randint(1, 8), power=rng.choice([0.1, 0.3, 1.0]), lpt=rng.choice([1, 2]))
    elif kind == "nn_map":
        c.update(head=rng.choice([0, 1]), path=rng.choice([0, 0, 0, 2]))
    elif kind == "nn_adjoint":
        c.update(head=rng.choice([0, 1]), path=rng.choice([0, 0, 2]))
    elif kind == "smooth":
        c.update(R=round(rng.uniform(1.0, 20.0), 2))
    elif kind == "paint":
        lattice = rng.choice([False, True])
        n = N**3 if lattice else min(N**3, int(N**3 * math.exp(rng.uniform(math.log(0.02), 0.0))) | 1)
        c.update(np=n, mass=rng.choice([False, True]), lattice=lattice)
    elif kind == "direction":
        c.update(k=rng.randint(1, 10))
    return c


# ------------------------------------------------------------------ the method in plain torch (any dtype)

def _freqs(N, dtype):
    dev = torch.device("cuda")
    n = torch.fft.fftfreq(N, d=1.0 / N, device=dev, dtype=dtype)
    nz = torch.arange(N // 2 + 1, device=dev, dtype=dtype)
    return n[:, None, None], n[None, :, None], nz[None, None, :]


def _k2(N, dtype):
    return sum((2 * math.pi / N * f) ** 2 for f in _freqs(N, dtype))


def _half_weights(N, dtype):
    w = torch.full((N // 2 + 1,), 2.0, device="cuda", dtype=dtype)
    w[0] = w[N // 2] = 1.0
    return w


def _irfft(s):
    N = s.shape[0]
    return torch.fft.irfftn(s, s=(N, N, N))


def _smooth(f, R_cells):
    if R_cells == 0:
        return f
    N = f.shape[0]
    return _irfft(torch.exp(-0.5 * R_cells**2 * _k2(N, f.dtype)) * torch.fft.rfftn(f))


def _odd(N, j, dtype):
    """k_j / k^2, zero at k = 0 and on component j's Nyquist plane (times i: a gradient of the inverse Laplacian)."""
    f = _freqs(N, dtype)
    k2 = _k2(N, dtype)
    k2[0, 0, 0] = 1.0
    m = (2 * math.pi / N) * f[j] / k2
    m[0, 0, 0] = 0.0
    return torch.where(f[j].abs() == N // 2, torch.zeros_like(m), m)


def _grad_invlap(sk, scale):
    N = sk.shape[0]
    return torch.stack([_irfft(1j * (scale * _odd(N, j, sk.real.dtype)) * sk) for j in range(3)])


def _bbks(k):
    q = np.maximum(k, 1e-30) / GAMMA
    return (np.log1p(2.34 * q) / (2.34 * q)
            * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25)


def _power(N, L):
    """P(k) N^6 / L^3 on the half array, float64, 0 at k = 0."""
    k = np.exp(np.linspace(math.log(1e-6), math.log(1e3), 400001))
    x = k * 8.0
    w = np.where(x < 1e-3, 1 - x * x / 10, 3 * (np.sin(x) - x * np.cos(x)) / x**3)
    sig2 = np.trapezoid(k**4 * _bbks(k) ** 2 * w**2, np.log(k)) / (2 * math.pi**2)
    n2 = np.arange(3 * (N // 2) ** 2 + 1, dtype=np.float64)
    kk = 2 * math.pi * np.sqrt(n2) / L
    tab = SIGMA8**2 / sig2 * kk * _bbks(kk) ** 2 * float(N) ** 6 / L**3
    tab[0] = 0.0
    f = _freqs(N, torch.float64)
    idx = sum(x * x for x in f).round().long()
    return torch.from_numpy(tab).cuda()[idx]


def _growth(a):
    """D, G_p, G_f of flat LCDM: D = E int_0^a (a E)^-3 da / norm, by Gauss-Legendre in t = sqrt(a)."""
    t, w = np.polynomial.legendre.leggauss(96)

    def integral(b):
        u = 0.5 * math.sqrt(b) * (t + 1)
        return 0.5 * math.sqrt(b) * np.sum(w * 2 * u**4 * (OMEGA_M + (1 - OMEGA_M) * u**6) ** -1.5)

    E = math.sqrt(OMEGA_M / a**3 + 1 - OMEGA_M)
    norm = integral(1.0)
    D = E * integral(a) / norm
    dD = (-1.5 * OMEGA_M / a**4 / E * integral(a) + E / (a * E) ** 3) / norm
    return D, a**3 * E * dD, 1.5 * OMEGA_M * D


def _corners(x, N):
    """x [3][np] grid units: flat cell indices and weights of the 8 CIC corners."""
    i = torch.floor(x.detach())
    d = x - i
    i = i.long() % N
    for o in range(8):
        b = [(o >> 2) & 1, (o >> 1) & 1, o & 1]
        c = [(i[a] + b[a]) % N for a in range(3)]
        w = [d[a] if b[a] else 1 - d[a] for a in range(3)]
        yield (c[0] * N + c[1]) * N + c[2], w[0] * w[1] * w[2]


def _paint(x, N, mass=None):
    rho = torch.zeros(N**3, device=x.device, dtype=x.dtype)
    for idx, w in _corners(x, N):
        rho = rho.index_add(0, idx, w if mass is None else w * mass)
    return rho.view(N, N, N)


def _readout3(F, x, N):
    f = F.reshape(3, -1)
    return sum(w * f[:, idx] for idx, w in _corners(x, N))


def _lattice(N):
    g = torch.arange(N, device="cuda", dtype=torch.float64)
    return torch.stack(torch.meshgrid(g, g, g, indexing="ij")).reshape(3, -1)


def _pm64(s, case):
    """Final overdensity of the modes s (complex128), differentiable."""
    N = case["N"]
    q = _lattice(N)
    D, Gp, _ = _growth(A0)
    psi = _grad_invlap(s, 1.0).reshape(3, -1)
    disp, p = D * psi, Gp * psi
    if case["lpt"] == 2:
        f = _freqs(N, torch.float64)
        k2 = _k2(N, torch.float64)
        k2[0, 0, 0] = 1.0

        def hess(i, j):
            m = (2 * math.pi / N) ** 2 * f[i] * f[j] / k2
            if i != j:
                m = torch.where((f[i].abs() == N // 2) | (f[j].abs() == N // 2), torch.zeros_like(m), m)
            m[0, 0, 0] = 0.0
            return _irfft(m * s)

        xx, yy, zz = hess(0, 0), hess(1, 1), hess(2, 2)
        src = xx * yy + xx * zz + yy * zz - hess(0, 1) ** 2 - hess(0, 2) ** 2 - hess(1, 2) ** 2
        psi2 = _grad_invlap(torch.fft.rfftn(src), -1.0).reshape(3, -1)
        disp, p = disp - 3 / 7 * D * D * psi2, p - 6 / 7 * D * Gp * psi2
    n = case["nsteps"]
    a = [A0 + (1 - A0) * i / n for i in range(n + 1)]
    for i in range(n):
        ah, ap = 0.5 * (a[i] + a[i + 1]), A0 if i == 0 else 0.5 * (a[i - 1] + a[i])
        kick = (_growth(ah)[1] - _growth(ap)[1]) / _growth(a[i])[2]
        drift = (_growth(a[i + 1])[0] - _growth(a[i])[0]) / _growth(ah)[1]

        def move(disp, p, kick=kick, drift=drift):
            x = q + disp
            F = _grad_invlap(torch.fft.rfftn(_paint(x, N) - 1.0), 1.5 * OMEGA_M)
            p = p + kick * _readout3(F, x, N)
            return disp + drift * p, p

        disp, p = checkpoint(move, disp, p, use_reentrant=False)
    return checkpoint(lambda d: _paint(q + d, N) - 1.0, disp, use_reentrant=False)


def _unpack(w):
    cut = [4050, 50, 1500, 30, 30, 1, 60, 20, 200, 10, 10, 1]
    shapes = [(50, 81), (50,), (30, 50), (30,), (30,), (), (20, 3), (20,), (10, 20), (10,), (10,), ()]
    out, o = [], 0
    for n, sh in zip(cut, shapes):
        if o < w.numel():
            out.append(w[o:o + n].view(sh))
        o += n
    return out


def _R_feat(case):
    """Feature scales in Mpc/h: the default ones, and for a whole evaluation 2, 3 and 4 cells."""
    if case["kind"] in ("eval", "step"):
        return [n * case["L"] / case["N"] for n in (2.0, 3.0, 4.0)]
    return [1.0, 2.0, 4.0]


def _features(delta, case):
    cell = case["L"] / case["N"]
    return torch.stack([_smooth(delta, R / cell) for R in _R_feat(case)])


def _mass_map(delta, w, case, a=3.0):
    """M(delta) of the network, by x-slabs (each recomputed in the backward)."""
    N = case["N"]
    f = _features(delta, case)
    W = _unpack(w.to(delta.dtype))

    def slab(f, x0, x1):
        xs = torch.arange(x0 - 1, x1 + 1, device=f.device) % N
        g = f[:, xs]
        a1 = 0
        for ox in range(3):
            gx = g[:, ox:ox + x1 - x0]
            for oy in range(3):
                for oz in range(3):
                    v = torch.roll(gx, (1 - oy, 1 - oz), (2, 3)).reshape(3, -1)
                    a1 = a1 + W[0].view(50, 3, 27)[:, :, ox * 9 + oy * 3 + oz] @ v
        z1 = torch.relu(a1 + W[1][:, None])
        z2 = torch.relu(W[2] @ z1 + W[3][:, None])
        y = W[4] @ z2 + W[5]
        if case["head"] == 0:
            m = torch.nn.functional.softplus(y, threshold=60.0)
        else:
            c = f[:, x0:x1].reshape(3, -1)
            h = torch.nn.functional.elu(W[6] @ c + W[7][:, None])
            h = torch.nn.functional.elu(W[8] @ h + W[9][:, None])
            m = torch.sigmoid(a * y) * (W[10] @ h + W[11])
        return M_SCALE * m

    step = max(1, (1 << 20) // (N * N))
    return torch.cat([checkpoint(slab, f, x, min(N, x + step), use_reentrant=False)
                      for x in range(0, N, step)]).view(N, N, N)


def _loss64(s, data, w, case):
    cell = case["L"] / case["N"]
    P = _power(case["N"], case["L"])
    P[0, 0, 0] = math.inf
    prior = 0.5 * (_half_weights(case["N"], torch.float64) * (s.real**2 + s.imag**2) / P).sum()
    MR = _smooth(_mass_map(_pm64(s, case), w, case), R_M / cell)
    DR = _smooth(data, R_M / cell)
    r = _smooth(torch.log((MR + case["M0"]) / (DR + case["M0"])), case["N_sm"])
    res = case.get("f_eff", 1.0) * (r * r).sum() / (4 * SIGMA_N2)
    return prior, res


def _loss_and_grad64(s, data, w, case):
    s = s.detach().requires_grad_(True)
    prior, res = _loss64(s, data, w, case)
    (g,) = torch.autograd.grad(prior + res, s)
    g[0, 0, 0] = 0.0
    return [float(prior + res), float(prior), float(res)], g


# ------------------------------------------------------------------ inputs

def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(seed * 16 + salt)


def _normal(shape, seed, salt):
    return torch.randn(shape, generator=_gen(seed, salt), device="cuda", dtype=torch.float32)


def _modes(case, seed, salt, power):
    """Linear modes s(k): white noise coloured by the power spectrum (float32 half array)."""
    N = case["N"]
    amp = torch.sqrt(power * _power(N, case["L"]) / N**3)
    return (amp * torch.fft.rfftn(_normal((N, N, N), seed, salt).double())).to(torch.complex64)


def _lognormal(case, seed, salt, power):
    """A log-normal field of mean ~1 with the linear modes' correlations, its log at unit variance at most."""
    N = case["N"]
    g = _irfft(_modes(case, seed, salt, power))
    g = g / torch.clamp(g.std(), min=1.0)
    return torch.exp(g - 0.5 * g.var())


def _margin_weights(w, f):
    """The weights with biases that keep every hidden unit on (even units) or off (odd) over the fields f, at least
    half its range of pre-activations away from zero, and the output scaled to mean 0.5 and unit spread."""
    N = f.shape[-1]
    w = w.clone()
    W1, b1, W2, b2, w3, b3 = _unpack(w)[:6]
    at = torch.randint(0, N, (3, 1 << 16), generator=_gen(1, 0), device="cuda")
    rows = [f[c][tuple((at[a] + o[a]) % N for a in range(3))] for c in range(3)
            for o in [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)]]
    v = torch.stack(rows)
    for W, b in ((W1, b1), (W2, b2)):
        pre = (W.double() @ v.double()).float()
        lo, hi = pre.min(1).values, pre.max(1).values
        on = torch.arange(b.numel(), device="cuda") % 2 == 0
        b.copy_(torch.where(on, -lo + 0.5 * (hi - lo), -hi - 0.5 * (hi - lo)))
        v = torch.relu(pre + b[:, None])
    y = w3.double() @ v.double()
    w3.div_(y.std())
    b3.copy_(0.5 - y.mean() / y.std())
    return w


def _weights(case, seed, field=None):
    w = torch.from_numpy(synth.two_net_weights(seed) if case.get("head") == 1 else synth.xavier_weights(seed)).cuda()
    if case.get("head") == 1:
        w[5951:5961] *= 0.2  # the mass network's output weights: masses stay positive on dense voxels too
    return w if field is None else _margin_weights(w, _features(field, case))


def _inputs(case, seed):
    N, kind = case["N"], case["kind"]
    if kind in ("eval", "step"):
        s = _modes(case, seed, 0, case["power"])
        scale = M_SCALE * (3.3 if case["head"] == 1 else 1.0)  # the mean mass of either network as set up below
        data = scale * _lognormal(case, seed, 1, 1.0) * torch.exp(0.3 * _normal((N, N, N), seed, 2))
        return {"s": s, "data": data, "w": _weights(case, seed, _lognormal(case, seed, 0, case["power"]) - 1.0)}
    if kind == "pm_grad":
        # a loss gradient as smooth as a residual's that was smoothed over some cells
        return {"s": _modes(case, seed, 0, case["power"]), "g": _smooth(_normal((N, N, N), seed, 1), 8.0)}
    if kind in ("nn_map", "nn_adjoint"):
        delta = _lognormal(case, seed, 0, 1.0) - 1.0
        if kind == "nn_map":
            return {"delta": delta, "w": _weights(case, seed)}
        return {"delta": delta, "w": _weights(case, seed, delta), "g": 1e-12 * _normal((N, N, N), seed, 1)}
    if kind in ("force", "smooth"):
        return {"delta": _lognormal(case, seed, 0, 1.0) - 1.0}
    if kind == "paint":
        n = case["np"]
        if case["lattice"]:  # lattice points moved by a Zel'dovich displacement of 10% power at a = 1, box wrapped
            psi = _grad_invlap(_modes(case, seed, 0, 0.1), 1.0).reshape(3, -1)
            x = torch.remainder(_lattice(N).float() + psi, float(N)).contiguous()
        else:
            g = _gen(seed, 0)
            x = torch.rand((3, n), generator=g, device="cuda") * (3 * N) - N  # unwrapped positions
            centre = torch.rand((3, max(1, n // 50)), generator=g, device="cuda") * N
            pick = torch.rand(n, generator=g, device="cuda") ** 1.5 * centre.shape[1]
            pick = pick.long().clamp(max=centre.shape[1] - 1)
            clump = centre[:, pick] + 0.8 * torch.randn((3, n), generator=g, device="cuda")
            x = torch.where(torch.rand(n, generator=g, device="cuda") < 0.5, clump, x).contiguous()
        return {"x": x, "mass": torch.exp(0.5 * _normal((n,), seed, 1)) if case["mass"] else None}
    n = 2 * N * N * (N // 2 + 1)
    S = _normal((case["k"], n), seed, 0).double()
    # curvature pairs of a positive diagonal with spread 0.5 to 2
    Y = S * torch.exp(math.log(2.0) * (2 * torch.rand(n, generator=_gen(seed, 1), device="cuda").double() - 1))
    return {"g": _normal((n,), seed, 2).double(), "S": S, "Y": Y}


def prepare(case, seed):
    st = _inputs(case, seed)
    kind = case["kind"]
    cfg = pmrecon.default_config(N=case["N"], L=case["L"], nsteps=case.get("nsteps", 1), head=case.get("head", 0),
                                 nn_path=case.get("path", 0), lpt_order=case.get("lpt", 1), R_feat=_R_feat(case),
                                 f_eff=case.get("f_eff", 1.0),
                                 lbfgs_m=10 if kind in ("eval", "step", "direction") else 1)
    stream = torch.cuda.Stream() if kind == "step" else torch.cuda.current_stream()
    w = st["w"] if "w" in st else torch.from_numpy(synth.xavier_weights(1)).cuda()
    torch.cuda.synchronize()  # inputs made on the current stream, used on the context's
    st.update(case=case, kind=kind, stream=stream, ctx=pmrecon.Context(cfg, w, stream))
    if kind == "step":
        st["ctx"].use_graphs(True)
        st["now"] = torch.empty_like(st["s"])
    return st


def run(st):
    ctx, case, kind = st["ctx"], st["case"], st["kind"]
    R_sm = case.get("N_sm", 0.0) * case["L"] / case["N"]  # residual smoothing, Mpc/h
    if kind == "eval":
        parts, g = ctx.loss_and_grad(st["s"], st["data"], R_sm, case["M0"])
        return {"loss": list(parts), "grad": g}
    if kind == "step":  # a stage's first iteration, always from the same modes
        with torch.cuda.stream(st["stream"]):
            st["now"].copy_(st["s"])
            ctx.lbfgs_reset()
            parts, _ = ctx.recon_step(st["now"], st["data"], R_sm, case["M0"])
        return {"loss": list(parts), "s": st["now"]}
    if kind == "pm_grad":
        s = st["s"].detach().requires_grad_(True)
        delta = pmrecon.PMForward.apply(s, ctx)
        (g,) = torch.autograd.grad(delta, s, st["g"])
        return {"delta": delta.detach(), "grad": g}
    if kind == "nn_map":
        return ctx.nn_halo_map(st["delta"])
    if kind == "nn_adjoint":
        return ctx.nn_halo_map_adjoint(st["delta"], st["g"])
    if kind == "force":
        return ctx.force(st["delta"])
    if kind == "smooth":
        return ctx.smooth(st["delta"], case["R"])
    if kind == "paint":
        return ctx.paint(st["x"], st["mass"])
    return ctx.lbfgs_direction(st["g"], st["S"], st["Y"])


def work(case):
    N, kind = case["N"], case["kind"]
    N3, NH = N**3, N * N * (N // 2 + 1)
    fft = 2.5 * N3 * math.log2(N3)  # one real 3D transform
    ics = 3 * fft if case.get("lpt", 1) == 1 else 13 * fft
    # per step: density (1 transform), three force components, paint and readout of every particle
    pm = ics + case.get("nsteps", 0) * (4 * fft + 200 * N3) + 60 * N3
    if kind in ("eval", "step"):
        smooth = 2 * fft
        one = 3 * pm + (NN_FWD + NN_BWD) * N3 + 14 * smooth
        n = 1 if kind == "eval" else 2  # the first iteration evaluates the start and at least one trial
        return {"bytes": n * (16 * NH + 4 * N3), "flops": n * one}
    if kind == "pm_grad":
        return {"bytes": 16 * NH + 8 * N3, "flops": 3 * pm}
    if kind == "nn_map":
        return {"bytes": 8 * N3, "flops": 4 * fft + NN_FWD * N3}
    if kind == "nn_adjoint":
        return {"bytes": 12 * N3, "flops": 8 * fft + (NN_FWD + NN_BWD) * N3}
    if kind == "force":
        return {"bytes": 16 * N3, "flops": 4 * fft}
    if kind == "smooth":
        return {"bytes": 8 * N3, "flops": 2 * fft}
    if kind == "paint":
        return {"bytes": 4 * N3 + (16 if case["mass"] else 12) * case["np"], "flops": 40 * case["np"]}
    n = 2 * NH
    return {"bytes": 8 * n * (2 * case["k"] + 2), "flops": 8 * case["k"] * n}


# ------------------------------------------------------------------ the same calls in float64

def exact(case, seed):
    v = _inputs(case, seed)
    N, kind = case["N"], case["kind"]
    if kind == "eval":
        parts, g = _loss_and_grad64(v["s"].to(torch.complex128), v["data"].double(), v["w"], case)
        return {"loss": parts, "grad": g}
    if kind == "step":
        s = v["s"].to(torch.complex128)
        data = v["data"].double()
        parts, g = _loss_and_grad64(s, data, v["w"], case)
        # first direction -D g with the prior's inverse Hessian D = P / w, Armijo backtracking from 1
        d = -_power(N, case["L"]) / _half_weights(N, torch.float64) * g
        gd = float((g.real * d.real + g.imag * d.imag).sum())
        t = 1.0
        for _ in range(20):
            with torch.no_grad():
                prior, res = (float(x) for x in _loss64(s + t * d, data, v["w"], case))
            if prior + res <= parts[0] + 1e-4 * t * gd:
                return {"loss": [prior + res, prior, res], "s": s + t * d}
            t *= 0.5
        return None
    if kind == "pm_grad":
        s = v["s"].to(torch.complex128).requires_grad_(True)
        delta = _pm64(s, case)
        (g,) = torch.autograd.grad(delta, s, v["g"].double())
        return {"delta": delta.detach(), "grad": g}
    if kind == "nn_map":
        with torch.no_grad():
            return _mass_map(v["delta"].double(), v["w"], case)
    if kind == "nn_adjoint":
        delta = v["delta"].double().requires_grad_(True)
        (g,) = torch.autograd.grad(_mass_map(delta, v["w"], case), delta, v["g"].double())
        return g
    if kind == "force":
        return _grad_invlap(torch.fft.rfftn(v["delta"].double()), 1.5 * OMEGA_M)
    if kind == "smooth":
        return _smooth(v["delta"].double(), case["R"] / (case["L"] / N))
    if kind == "paint":
        w = torch.fmod(v["x"], float(N))  # the library's float32 wrap rule: a cell index is a whole number
        w = torch.where(w < 0, w + float(N), w)
        w = torch.where(w >= N, torch.zeros_like(w), w).double()
        return _paint(w, N, None if v["mass"] is None else v["mass"].double())
    q = v["g"].clone()
    S, Y = v["S"], v["Y"]
    rho = [1.0 / torch.dot(S[t], Y[t]) for t in range(case["k"])]
    alpha = [None] * case["k"]
    for t in reversed(range(case["k"])):
        alpha[t] = rho[t] * torch.dot(S[t], q)
        q -= alpha[t] * Y[t]
    q *= torch.dot(S[-1], Y[-1]) / torch.dot(Y[-1], Y[-1])
    for t in range(case["k"]):
        q += (alpha[t] - rho[t] * torch.dot(Y[t], q)) * S[t]
    return -q
