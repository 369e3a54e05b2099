"""The workloads whose speed is measured, as a user's program runs them.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (the
plan, the density on the GPU or in pinned host memory), ``run`` makes one pass through the
package's public entry points, ``exact`` evaluates the same discrete problem in 64 bits with
plain torch and numpy.

Kinds of case:

* ``cube``     one density on a cube, ``Plan.solve`` (time loops: one plan, many solves)
* ``box``      one density on a box with its own point count per axis, ``Plan.solve``
* ``batch``    independent densities of uneven size, ``solve_batched``
* ``host``     one density in pinned host memory, ``Plan.solve_host``
* ``checked``  several densities of one size with the a-posteriori indicator, the call that
               the grid selector's refinement makes
* ``train``    one full-batch gradient of the grid selector's network
"""
import ctypes
import math

import numpy as np
import torch

from paper_1612_01799_gb300 import Plan, _lib, selector, solve_batched

TOL = {"f32": 1e-6, "f64": 1e-12}     # plan tolerances of the benchmark workloads
BATCH_SIZES = (64, 96, 128, 160, 192)  # grid sizes of the batched benchmark
FEATURES, HIDDEN = 64, 64              # the selector network's widths


def _smooth(lo, hi):
    """Even counts with no prime factor above 5: every size a plan can have."""
    out = []
    for n in range(lo, hi + 1, 2):
        m = n
        for f in (2, 3, 5):
            while m % f == 0:
                m //= f
        if m == 1:
            out.append(n)
    return out


def _pick(rng, lo, hi):
    """One of the sizes in [lo, hi], spread over the logarithm."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_smooth(lo, hi), key=lambda n: abs(math.log(n / x)))


def listed():
    return [
        # The smallest solves: a simulation step or a coarse grid, bound by launches.
        {"name": "cube_f32_n32", "kind": "cube", "n": 32, "dtype": "f32"},
        # The FP64 unit workload (one Gaussian-like density, N = 32).
        {"name": "cube_f64_n32", "kind": "cube", "n": 32, "dtype": "f64"},
        # The headline workload: N = 256 (padded 512^3), FP32 and FP64.
        {"name": "cube_f32_n256", "kind": "cube", "n": 256, "dtype": "f32"},
        {"name": "cube_f64_n256", "kind": "cube", "n": 256, "dtype": "f64"},
        # The large single solve: N = 512 (padded 1024^3).
        {"name": "cube_f32_n512", "kind": "cube", "n": 512, "dtype": "f32"},
        # Sizes that follow from a physical spacing and are no power of two: N = 400 (padded
        # 800^3), and the 162^3 grid of the paper's tables in FP64.
        {"name": "cube_f32_n400", "kind": "cube", "n": 400, "dtype": "f32"},
        {"name": "cube_f64_n162", "kind": "cube", "n": 162, "dtype": "f64"},
        # An elongated domain sampled with one spacing: a different count on every axis.
        {"name": "box_f32_64_128_192", "kind": "box", "nx": 64, "ny": 128, "nz": 192, "dtype": "f32"},
        # Many independent densities of uneven size in one call.
        {"name": "batch_f32_16", "kind": "batch", "count": 16, "sizes": 5, "dtype": "f32"},
        # End to end on host buffers: the copies are part of the call.
        {"name": "host_f32_n256", "kind": "host", "n": 256, "dtype": "f32"},
        # The selector's refinement: densities that chose the same size, solved and checked.
        {"name": "checked_f32_n96_b12", "kind": "checked", "n": 96, "count": 12, "dtype": "f32"},
        # Training the selector: loss and gradient over the whole training set.
        {"name": "train_b384", "kind": "train", "count": 384, "k": 12, "dtype": "f32"},
    ]


def draw(rng):
    kind = rng.choice(["cube", "cube", "cube", "box", "box", "batch", "host", "checked", "train"])
    if kind == "cube":
        dtype = rng.choice(["f32", "f32", "f64"])
        return {"kind": kind, "n": _pick(rng, 16, 400 if dtype == "f32" else 200), "dtype": dtype}
    if kind == "box":
        dtype = rng.choice(["f32", "f32", "f64"])
        hi = 256 if dtype == "f32" else 128
        return {"kind": kind, "nx": _pick(rng, 16, hi), "ny": _pick(rng, 16, hi), "nz": _pick(rng, 16, hi),
                "dtype": dtype}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 24), "sizes": rng.randint(1, 5), "dtype": "f32"}
    if kind == "host":
        dtype = rng.choice(["f32", "f32", "f64"])
        return {"kind": kind, "n": _pick(rng, 32, 256 if dtype == "f32" else 160), "dtype": dtype}
    if kind == "checked":
        n = rng.choice([n for n in selector.CANDIDATES if n <= 192])
        return {"kind": kind, "n": n, "count": rng.randint(1, max(1, min(16, (256 // n) ** 3))), "dtype": "f32"}
    return {"kind": kind, "count": int(math.exp(rng.uniform(math.log(32), math.log(512)))), "k": rng.randint(4, 16),
            "dtype": "f32"}


# ---- the inputs -------------------------------------------------------------------------------

def _counts(case):
    """Points per axis of every density of the case."""
    if case["kind"] == "box":
        return [(case["nx"], case["ny"], case["nz"])]
    if case["kind"] == "batch":
        # As many of the benchmark's sizes as the case says, dealt out in turn.
        return [(BATCH_SIZES[i % case["sizes"]],) * 3 for i in range(case["count"])]
    return [(case["n"],) * 3] * (case["count"] if case["kind"] == "checked" else 1)


def _lengths(n):
    """Half-lengths of the domain: one spacing on every axis, 10 for the longest."""
    return tuple(10.0 * q / max(n) for q in n)


def _density(rng, n, fine):
    """Sum of 1 to 6 anisotropic normalised Gaussians (centres within 0.3, widths 0.05 to 0.15
    of the half-length on each axis, charges in [-1, 1] with a net charge), FP64 on the GPU,
    [z][y][x].  fine: widths of 0.8 to 1.6 grid spacings instead, a density that the grid
    barely resolves, whose spectrum has a tail above the round-off."""
    L = _lengths(n)
    g = int(rng.integers(1, 7))
    while True:
        q = rng.uniform(-1.0, 1.0, size=g)
        if abs(q.sum()) >= 0.1:
            break
    f = []
    for a in range(3):
        x = -L[a] + (np.arange(n[a]) + 0.5) * (2.0 * L[a] / n[a])
        c = rng.uniform(-0.3, 0.3, size=(g, 1)) * L[a]
        s = rng.uniform(1.6 / n[a], 3.2 / n[a], size=(g, 1)) if fine else rng.uniform(0.05, 0.15, size=(g, 1))
        s = s * L[a]
        f.append(torch.from_numpy(np.exp(-0.5 * ((x - c) / s) ** 2) / (math.sqrt(2.0 * math.pi) * s)).cuda())
    f[2] = f[2] * torch.from_numpy(q).cuda()[:, None]
    yx = (f[1][:, :, None] * f[0][:, None, :]).reshape(g, -1)
    return (f[2].T @ yx).reshape(n[2], n[1], n[0])


def _densities(case, seed):
    rng = np.random.default_rng([seed, 1])
    dt = torch.float32 if case["dtype"] == "f32" else torch.float64
    return [_density(rng, n, case["kind"] == "checked").to(dt) for n in _counts(case)]


def _training_set(case, seed):
    """Standardised features, target log10 errors and network parameters (FP32, numpy)."""
    rng = np.random.default_rng([seed, 2])
    B, K = case["count"], case["k"]
    x = rng.standard_normal((B, FEATURES)).astype(np.float32)
    t = rng.uniform(-9.0, 0.0, size=(B, K)).astype(np.float32)
    parts = []
    for fan_in, fan_out in ((FEATURES, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN, K)):
        lim = math.sqrt(6.0 / (fan_in + fan_out))
        parts += [rng.uniform(-lim, lim, size=fan_out * fan_in), rng.uniform(-0.1, 0.1, size=fan_out)]
    return x, t, np.concatenate(parts).astype(np.float32)


def _plan(n, dtype, max_batch=1):
    if len(set(n)) == 1:
        p = Plan(n[0], 10.0, TOL[dtype], dtype, max_batch=max_batch)
    else:
        p = Plan(n, _lengths(n), TOL[dtype], dtype)
    if dtype == "f64":
        p.arith = "df"    # what FP64 plans pick here; fixed so that every run measures the same
    return p


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t, params = _training_set(case, seed)
        net = selector.Network(case["k"])
        net.params.copy_(torch.from_numpy(params))
        return {"kind": kind, "net": net, "x": torch.from_numpy(x).cuda(), "t": torch.from_numpy(t).cuda()}
    rho = _densities(case, seed)
    if kind == "host":
        host = rho[0].cpu().pin_memory()
        return {"kind": kind, "plan": _plan(_counts(case)[0], case["dtype"]), "rho": host,
                "out": torch.empty_like(host).pin_memory()}
    state = {"kind": kind, "rho": rho, "out": [torch.empty_like(r) for r in rho]}
    if kind == "batch":
        sizes = [n[0] for n in _counts(case)]
        plans = {n: _plan((n, n, n), case["dtype"], sizes.count(n)) for n in sorted(set(sizes))}
        state["plans"] = [plans[n] for n in sizes]
    elif kind == "checked":
        count = case["count"]
        state["plan"] = _plan(_counts(case)[0], case["dtype"], count)
        state["rho_p"] = (ctypes.c_void_p * count)(*[r.data_ptr() for r in rho])
        state["out_p"] = (ctypes.c_void_p * count)(*[u.data_ptr() for u in state["out"]])
    else:
        state["plan"] = _plan(_counts(case)[0], case["dtype"])
    return state


def run(state):
    kind = state["kind"]
    if kind in ("cube", "box"):
        return state["plan"].solve(state["rho"][0], out=state["out"][0])
    if kind == "batch":
        return solve_batched(state["plans"], state["rho"], state["out"])
    if kind == "host":
        return state["plan"].solve_host(state["rho"], out=state["out"])
    if kind == "checked":
        count = len(state["rho"])
        eta = (ctypes.c_double * count)()
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        _lib.check(_lib.load().poisson_solve_checked_batched(state["plan"].handle, count, state["rho_p"],
                                                             state["out_p"], eta, stream),
                   "poisson_solve_checked_batched")
        return {"u": state["out"], "eta": np.array(eta[:])}
    loss = state["net"].gradient(state["x"], state["t"])
    return {"loss": loss, "grad": state["net"].grad}


def work(case):
    """Bytes: the inputs once and the outputs once.  Operations: the zero-padded transforms
    (5 L log2 L per complex transform of length L = 2 n, half that for the real x axis, the
    zero half of the padding left out) both ways and the symbol product."""
    if case["kind"] == "train":
        B, K = case["count"], case["k"]
        npar = 3 * (HIDDEN * HIDDEN + HIDDEN) + K * HIDDEN + K
        return {"bytes": 4 * (B * (FEATURES + K) + 2 * npar), "flops": 6 * B * (3 * HIDDEN * HIDDEN + K * HIDDEN)}
    s = 4 if case["dtype"] == "f32" else 8
    nbytes = flops = 0
    for nx, ny, nz in _counts(case):
        def fft(n):
            return 5.0 * 2 * n * math.log2(2 * n)
        nbytes += 2 * s * nx * ny * nz
        flops += 2 * (ny * nz * 0.5 * fft(nx) + nz * (nx + 1) * fft(ny) + 2 * ny * (nx + 1) * fft(nz))
        flops += 2 * (nx + 1) * 2 * ny * 2 * nz
    return {"bytes": nbytes, "flops": int(flops)}


def tolerance(case):
    """About four times the error against 64 bits that the passes show: 1.0e-7 to 2.0e-7 in
    FP32, 6.2e-15 to 7.8e-15 in double-float, 2.4e-7 for the gradient."""
    if case["kind"] == "train":
        return {"rel": 1e-6}
    return {"rel": 8e-7 if case["dtype"] == "f32" else 3e-14}


# ---- the same discrete problem in 64 bits -----------------------------------------------------

def _gauss_sum(eps, delta, r_max):
    """1/(4 pi r) = (1/(2 pi^{3/2})) int exp(-r^2 e^{2s} + s) ds by the trapezoid rule with the
    largest step 2/m whose relative error on [delta, r_max] is at most eps."""
    t_lo = eps * math.sqrt(math.pi) / (8.0 * r_max)
    lo, hi = -10.0, 30.0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if math.erfc(mid) > 0.25 * eps else (lo, mid)
    t_hi = 0.5 * (lo + hi) / delta
    r = np.exp(np.linspace(math.log(delta), math.log(r_max), 4096))
    r[0], r[-1] = delta, r_max
    for m in range(2, 4000):
        h = 2.0 / m
        s = h * np.arange(math.floor(math.log(t_lo) / h), math.ceil(math.log(t_hi) / h) + 1)
        tau, w = np.exp(s), h * np.exp(s) / (2.0 * math.pi ** 1.5)
        u = np.exp(-(r[:, None] * tau) ** 2) @ w
        if np.abs(4.0 * math.pi * r * u - 1.0).max() <= eps:
            return tau, w
    raise ValueError("no step meets eps")


def _moment(p, tau, d):
    """int_0^d r^p exp(-tau^2 r^2) dr, p = 2 or 4."""
    x = tau * d
    if x < 0.5:
        return sum((-tau * tau) ** n * d ** (2 * n + p + 1) / (math.factorial(n) * (2 * n + p + 1)) for n in range(30))
    e, er = math.exp(-x * x), math.erf(x)
    if p == 2:
        return math.sqrt(math.pi) * er / (4.0 * tau ** 3) - d * e / (2.0 * tau ** 2)
    return 3.0 * math.sqrt(math.pi) * er / (8.0 * tau ** 5) - e * (d ** 3 / (2.0 * tau ** 2) + 3.0 * d / (4.0 * tau ** 4))


def _axis_factor(tau, n):
    """A_j(k) = 2 int_0^2 exp(-tau_j^2 t^2) cos(pi k t / 2) dt, k = 0..n."""
    kap = 0.5 * math.pi * np.arange(n + 1)
    gx, gw = np.polynomial.legendre.leggauss(16)
    P = max(16, (n + 1) // 2)
    t = ((2.0 * np.arange(P)[:, None] + 1.0 + gx) / P).ravel()
    w = np.tile(gw / P, P)
    A = np.empty((len(tau), n + 1))
    wide = tau >= 3.0
    tw = tau[wide][:, None]
    A[wide] = math.sqrt(math.pi) / tw * np.exp(-kap ** 2 / (4.0 * tw ** 2))
    A[~wide] = 2.0 * (w * np.exp(-(tau[~wide][:, None] * t) ** 2)) @ np.cos(np.outer(t, kap))
    return A


def _solve64(rho, tol):
    """The zero-padded convolution of one density in FP64 (CPU tensor) and its tail indicator."""
    nz, ny, nx = rho.shape
    n = (nx, ny, nz)
    L = _lengths(n)
    lam = max(L)
    l = [q / lam for q in L]
    delta = max(min(2.0 * L[a] / (50.0 * n[a]) for a in range(3)), 1e-3)
    tau, w = _gauss_sum(min(max(0.1 * tol, 1e-14), 1e-7), delta, 2.0 * math.sqrt(sum(q * q for q in l)))
    c0 = 0.5 * delta ** 2 - 4.0 * math.pi * sum(a * _moment(2, b, delta) for a, b in zip(w, tau))
    c2 = (0.25 * delta ** 4 - 4.0 * math.pi * sum(a * _moment(4, b, delta) for a, b in zip(w, tau))) / 6.0
    A = [torch.from_numpy(l[a] * _axis_factor(tau * l[a], n[a])).cuda() for a in range(3)]
    kap2 = [torch.from_numpy((0.5 * math.pi * np.arange(n[a] + 1) / l[a]) ** 2).cuda() for a in range(3)]
    F = torch.fft.rfftn(rho.double(), s=(2 * nz, 2 * ny, 2 * nx))
    mirror = torch.cat([torch.arange(ny + 1), torch.arange(ny - 1, 0, -1)]).cuda()
    weight = torch.full((nx + 1,), 2.0, dtype=torch.float64, device="cuda")
    weight[0] = weight[nx] = 1.0
    shell_yx = ((torch.arange(ny + 1) >= ny - ny // 8)[:, None] | (torch.arange(nx + 1) >= nx - nx // 8)).cuda()[mirror]
    wA, total, shell = torch.from_numpy(w).cuda()[:, None] * A[2], 0.0, 0.0
    for kz in range(nz + 1):
        g = (A[1] * wA[:, kz, None]).T @ A[0]
        g = (g + c0 - c2 * (kap2[2][kz] + kap2[1][:, None] + kap2[0]))[mirror]
        for z in {kz, (2 * nz - kz) % (2 * nz)}:
            e = (F[z].real ** 2 + F[z].imag ** 2) * weight
            total += float(e.sum())
            shell += float(e.sum() if kz >= nz - nz // 8 else e[shell_yx].sum())
            F[z] *= g
    u = torch.fft.irfftn(F, s=(2 * nz, 2 * ny, 2 * nx))[:nz, :ny, :nx] * lam ** 2
    return u.cpu(), math.sqrt(shell / total)


def exact(case, seed):
    if case["kind"] == "train":
        x, t, params = (torch.from_numpy(a).double() for a in _training_set(case, seed))
        params.requires_grad_(True)
        h, off = x, 0
        for layer in range(4):
            out = HIDDEN if layer < 3 else case["k"]
            W = params[off:off + out * h.shape[1]].view(out, -1)
            b = params[off + W.numel():off + W.numel() + out]
            off += W.numel() + out
            h = h @ W.T + b
            if layer < 3:
                h = torch.relu(h)
        loss = ((h - t) ** 2).mean()
        loss.backward()
        return {"loss": loss.detach().reshape(1), "grad": params.grad}
    res = [_solve64(r, TOL[case["dtype"]]) for r in _densities(case, seed)]
    if case["kind"] in ("cube", "box", "host"):
        return res[0][0]
    if case["kind"] == "batch":
        return [u for u, _ in res]
    return {"u": [u for u, _ in res], "eta": np.array([e for _, e in res])}
