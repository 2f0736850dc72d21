"""What a user of this library has it compute, over the sizes, precisions and options it is used with.

A case is a dict of plain values.  Keys (the ones an operation does not use are left out):
  op         "spectrum" (sigw_generate[_batch] + sigw_spectrum), "scan" (sigw_target_scan), "jackknife"
             (sigw_generate + sigw_spectrum_jackknife), "fft" (sigw_fft3d / sigw_fft3d_noalloc) or "serve" (a server
             that gets a burst of mixed requests)
  N          lattice side;  precision 32 or 64;  batch  realisations of one call
  map        "gauss", "local", "usr", "nonlocal", or "mixed" (one parameter point per realisation)
  shells     how many target shells, spread over 1..N/2 (0: every shell, the library's own default)
  n_alpha    separable terms;  sigma  width of the log-normal peak;  nstar  its place in units of the fundamental
  targets    target frequencies of a scan;  M  sub-volumes per side of the jackknife
  direction  -1 / +1, noalloc  whether the entry point without a plan is used
  requests   burst size of the server;  nmax  its largest lattice

The spectra of a 32-bit plan are single-precision numbers (the library hands them out in double arrays, whatever the
plan's precision); ``run`` returns them in the type of the plan.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2605_27231_gb300 import sigw

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # the smallest call: the plan-free transform of a latency-critical caller
        {"name": "fft32_noalloc", "op": "fft", "N": 32, "precision": 32, "direction": -1, "noalloc": True},
        # the library's transform on the headline lattice, spectrum to field
        {"name": "fft256_inverse", "op": "fft", "N": 256, "precision": 32, "direction": 1, "noalloc": False},
        # the paper's own workload: 20 target frequencies, one box each, Gaussian, the smaller of its two lattices
        {"name": "scan64", "op": "scan", "N": 64, "precision": 32, "map": "gauss", "targets": 20, "n_alpha": 50,
         "sigma": 0.5},
        # the same on its larger lattice with a local non-Gaussian field
        {"name": "scan128_local", "op": "scan", "N": 128, "precision": 32, "map": "local", "targets": 20, "n_alpha": 50,
         "sigma": 0.5},
        # the double-precision reference run on the smallest science lattice, all shells
        {"name": "gauss32_f64", "op": "spectrum", "N": 32, "precision": 64, "map": "gauss", "batch": 1, "shells": 0,
         "n_alpha": 50, "sigma": 0.5, "nstar": 8.0},
        # a parameter scan: eight points of mixed maps in one batch, all shells
        {"name": "batch64_mixed", "op": "spectrum", "N": 64, "precision": 32, "map": "mixed", "batch": 8, "shells": 0,
         "n_alpha": 50, "sigma": 0.5, "nstar": 8.0},
        # one local non-Gaussian spectrum, all shells
        {"name": "local128", "op": "spectrum", "N": 128, "precision": 32, "map": "local", "batch": 1, "shells": 0,
         "n_alpha": 50, "sigma": 0.5, "nstar": 16.0},
        # the headline workload, four seeds at once, on some of its shells
        {"name": "usr256", "op": "spectrum", "N": 256, "precision": 32, "map": "usr", "batch": 4, "shells": 6,
         "n_alpha": 50, "sigma": 0.3, "nstar": 32.0},
        # the largest lattice, one shell (40 terms, so that several plans fit the memory side by side)
        {"name": "broad512", "op": "spectrum", "N": 512, "precision": 32, "map": "local", "batch": 1, "shells": 1,
         "n_alpha": 40, "sigma": 1.0, "nstar": 64.0},
        # error bars: the jackknife over 4^3 sub-volumes, every shell it offers, on the non-local map (whose field takes
        # further transform round trips)
        {"name": "jackknife64_nonlocal", "op": "jackknife", "N": 64, "precision": 32, "map": "nonlocal", "batch": 1,
         "shells": 0, "n_alpha": 50, "sigma": 0.5, "nstar": 16.0, "M": 4},
        # the server: a burst of requests of two lattice sizes and mixed parameters
        {"name": "serve_burst", "op": "serve", "N": 64, "nmax": 128, "precision": 32, "map": "mixed", "requests": 8,
         "n_alpha": 50},
    ]


COST_MOST = 0.26  # seconds a drawn case is meant to take at most, by _cost


def _cost(c, shells):
    """Rough seconds of the hot loop: 112 us per (term, realisation) at 256^3 in single precision."""
    return c.get("batch", 1) * shells * 2 * c["n_alpha"] * 112e-6 * (c["N"] / 256) ** 3 * (25 if c["precision"] == 64 else 1)


def draw(rng):
    op = rng.choices(("spectrum", "scan", "jackknife", "fft", "serve"), (9, 3, 2, 3, 1))[0]
    precision = 64 if rng.random() < 0.3 else 32
    if op == "fft":
        noalloc = rng.random() < 0.4
        N = 2 ** rng.randint(3, (6 if precision == 64 else 7) if noalloc else 8)
        return {"op": "fft", "N": N, "precision": precision, "direction": rng.choice((-1, 1)), "noalloc": noalloc}
    n_alpha = rng.choice((50, 50, 50, rng.randint(12, 50)))
    sigma = round(rng.uniform(0.1, 1.0), 3)
    if op == "serve":
        return {"op": "serve", "N": rng.choice((32, 64)), "nmax": rng.choice((64, 128)), "precision": 32, "map": "mixed",
                "requests": rng.randint(3, 9), "n_alpha": n_alpha}
    if op == "scan":
        N = 2 ** rng.randint(4, 7 if precision == 32 else 6)
        return {"op": "scan", "N": N, "precision": precision, "map": rng.choice(("gauss", "local", "usr")),
                "targets": rng.randint(3, 25 if N * precision < 4096 else 9), "n_alpha": n_alpha, "sigma": sigma}
    if op == "jackknife":
        N = 2 ** rng.randint(4, 7 if precision == 32 else 6)
        c = {"op": op, "N": N, "precision": precision, "map": rng.choice(("gauss", "local", "usr", "nonlocal")),
             "batch": rng.randint(1, 3), "n_alpha": n_alpha, "sigma": sigma, "nstar": N / rng.choice((4, 8)),
             "M": rng.choice((2, 4))}
        most = N // 2 - 1
    else:
        N = 2 ** (rng.randint(3, 7) if precision == 64 else rng.choices(range(3, 10), (4, 4, 4, 4, 4, 4, 1))[0])
        c = {"op": op, "N": N, "precision": precision, "map": rng.choice(("gauss", "local", "usr", "nonlocal", "mixed")),
             "batch": rng.randint(1, 5 if N < 256 else 3), "n_alpha": n_alpha, "sigma": sigma,
             "nstar": N / rng.choice((4, 8))}
        if N == 512:
            c |= {"batch": 1, "n_alpha": min(n_alpha, 40)}
        most = N // 2
    while c["batch"] > 1 and _cost(c, 1) > COST_MOST:
        c["batch"] -= 1
    shells = max(1, min(most, int(COST_MOST / _cost(c, 1))))
    if shells > 3 and rng.random() < 0.5:
        shells = rng.randint(1, shells)
    c["shells"] = 0 if shells == most else shells
    return c


def _shells(c):
    """The target shells of a case: None (the library's default) or `shells` of them spread over the range."""
    n = c["shells"]
    if n == 0:
        return None
    return sorted({max(1, int((i + 0.5) * (c["N"] // 2) / n)) for i in range(n)})


def _points(c, seed):
    """One parameter point (lattice, P_zeta, map, noise seed) per realisation or request."""
    rng = random.Random(1000003 * seed + c["N"])
    serve = c["op"] == "serve"
    out = []
    for i in range(c["requests"] if serve else c.get("batch", 1)):
        N = (c["nmax"] if i % 3 == 2 else c["N"]) if serve else c["N"]
        kind, sigma, f_nl = c["map"], c.get("sigma"), 5.0
        if kind == "mixed":
            kind, sigma, f_nl = ("local", "gauss", "usr")[i % 3], rng.uniform(0.1, 1.0), rng.uniform(-5.0, 20.0)
        out.append(SimpleNamespace(
            N=N, L=1.0, A=5e-3 if kind == "usr" else 1e-2, sigma=sigma, kstar=(N / 8 if serve else c["nstar"]) * TWO_PI,
            kind=kind, F_NL=0.6 * f_nl if kind == "local" else 0.0, G_NL=0.0, usr_floor=1e-6,
            alpha_NL=5.0 if kind == "nonlocal" else 0.0, beta_NL=-3.0 if kind == "nonlocal" else 0.0,
            seed=rng.getrandbits(62)))
    return out


def _targets(c):
    return np.geomspace(0.2, 3.0, c["targets"])


def _scan_point(c, seed):
    kind = c["map"]
    return dict(A=5e-3 if kind == "usr" else 1e-2, sigma=c["sigma"], kstar=1.0, kind=kind,
                F_NL=3.0 if kind == "local" else 0.0, seed=random.Random(seed).getrandbits(62))


def _types(c):
    return (torch.float64, torch.complex128) if c["precision"] == 64 else (torch.float32, torch.complex64)


def _fft_input(c, seed):
    """A real field, or the half spectrum of one."""
    N = c["N"]
    real, cplx = _types(c)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((N, N, N), generator=g, device="cuda", dtype=real)
    return x if c["direction"] < 0 else torch.fft.rfftn(x).contiguous()


def prepare(case, seed):
    op, N = case["op"], case["N"]
    if op == "fft":
        real, cplx = _types(case)
        x = _fft_input(case, seed)
        out = torch.empty((N, N, N // 2 + 1), device="cuda", dtype=cplx) if case["direction"] < 0 else \
            torch.empty((N, N, N), device="cuda", dtype=real)
        # a caller of the transform alone keeps the smallest plan
        plan = None if case["noalloc"] else sigw.Plan(N, 1.0, precision=case["precision"], n_modes=2, n_alpha=1)
        return {"case": case, "plan": plan, "in": x, "out": out}
    if op == "serve":
        server = sigw.Server(20e9, max_slots=2, precision=case["precision"], n_alpha=case["n_alpha"], max_batch=4)
        return {"case": case, "server": server, "points": _points(case, seed)}
    plan = sigw.Plan(N, 1.0, precision=case["precision"], n_alpha=case["n_alpha"], max_batch=case.get("batch", 1))
    if op == "scan":
        return {"case": case, "plan": plan, "k": _targets(case), "point": _scan_point(case, seed)}
    return {"case": case, "plan": plan, "points": _points(case, seed), "shells": _shells(case)}


def run(state):
    c = state["case"]
    if c["op"] == "fft":
        x, out = state["in"], state["out"]
        if c["noalloc"]:
            sigw.fft3d_noalloc(c["N"], c["precision"], c["direction"], x.data_ptr(), out.data_ptr())
        else:
            state["plan"].fft3d(c["direction"], x.data_ptr(), out.data_ptr())
        return out
    t = np.float64 if c["precision"] == 64 else np.float32
    if c["op"] == "serve":
        s = state["server"]
        tickets = [s.submit(p) for p in state["points"]]
        return [s.wait(k)[0].astype(t) for k in tickets]
    plan = state["plan"]
    if c["op"] == "scan":
        r = plan.target_scan(state["k"], **state["point"])
        return {"omega": r["omega"].astype(t), "L": r["L"], "n_c": r["n_c"]}
    hits = plan.generate_batch(state["points"])
    if c["op"] == "jackknife":
        r = plan.spectrum_jackknife(state["shells"], M=c["M"])
        return {"hits": hits, **{k: list(v.astype(t)) for k, v in r.items() if k != "n_c"}}
    r = plan.spectrum(state["shells"])
    return {"hits": hits, "Nk": r["Nk"], **{k: list(r[k].astype(t)) for k in ("omega", "PA", "PB")}}


def _fft_flops(N):
    return 2.5 * N ** 3 * math.log2(float(N) ** 3)  # a real transform


def _shell_work(N, n_alpha, shells, size):
    """Per realisation: two kernels a shell, three inverse transforms and 18 product operations a point for each term,
    six forward transforms; Phi~ is read for every (shell, kernel)."""
    per = (3 * n_alpha + 6) * _fft_flops(N) + 18.0 * n_alpha * N ** 3
    phi = N * N * (N // 2 + 1) * 2 * size
    return shells * 2 * phi, shells * 2 * per


def work(case):
    N, size = case["N"], case["precision"] // 8
    real, half = N ** 3 * size, N * N * (N // 2 + 1) * 2 * size
    if case["op"] == "fft":
        return {"bytes": real + half, "flops": _fft_flops(N)}
    if case["op"] == "serve":
        each = [_shell_work(p.N, case["n_alpha"], p.N // 2, size) for p in _points(case, 0)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    if case["op"] == "scan":
        units, shells, batch = case["targets"], 1, 1
    else:
        units, shells, batch = 1, len(_shells(case) or range(N // 2 - (case["op"] == "jackknife"))), case["batch"]
    b, f = _shell_work(N, case["n_alpha"], shells, size)
    synth = 1 if case["map"] == "gauss" else 3 if case["map"] != "nonlocal" else 6
    if case["op"] == "jackknife":
        f += shells * 2 * (2 * _fft_flops(N) + 2.0 * N ** 3)
    return {"bytes": units * batch * (b + half), "flops": units * batch * (f + synth * _fft_flops(N))}


# ---- the same numbers in 64 bits, in plain numpy and torch

def _kernel(m, u, v):
    a = u * u + v * v - 3.0
    if m == 0:
        return np.where(u + v > math.sqrt(3.0), 27.0 * math.pi * a * a / (32.0 * u ** 3 * v ** 3), 0.0)
    lg = np.log(np.abs((3.0 - (u + v) ** 2) / (3.0 - (u - v) ** 2)))
    return 27.0 * a / (32.0 * u ** 3 * v ** 3) * (a * lg - 4.0 * u * v)


def _separable(n_alpha, n_modes=200, umin=1e-3, umax=15.0, upiv=1.0, sigp=0.5, Ap=10.0):
    """Cell edges of the u-grid and, for both kernels, the n_alpha largest eigen-terms (sigma, phi[term][cell])."""
    erf = np.vectorize(math.erf)
    s2 = math.sqrt(2.0) * sigp

    def R(u):
        return (u - umin) + Ap * sigp * math.sqrt(math.pi / 2) * (erf((u - upiv) / s2) - math.erf((umin - upiv) / s2))

    want = np.arange(n_modes + 1) * R(np.array([umax]))[0] / n_modes
    lo, hi = np.full(n_modes + 1, umin), np.full(n_modes + 1, umax)
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        low = R(mid) < want
        lo, hi = np.where(low, mid, lo), np.where(low, hi, mid)
    edges = 0.5 * (lo + hi)
    edges[0], edges[-1] = umin, umax
    mid, width = 0.5 * (edges[1:] + edges[:-1]), np.diff(edges)
    u, v = mid[:, None], mid[None, :]
    strip = (np.abs(u - v) <= 1.0) & (u + v >= 1.0)
    terms = []
    for m in (0, 1):
        C = np.where(strip, np.sqrt(width[:, None] * width[None, :]) * _kernel(m, u, v), 0.0)
        w, Q = np.linalg.eigh(0.5 * (C + C.T))
        keep = np.argsort(-np.abs(w), kind="stable")[:n_alpha]
        terms.append((w[keep], (Q[:, keep] / np.sqrt(width)[:, None]).T.copy()))
    return edges, terms


def _noise(N, seed):
    """N(0, 1) per cell: Philox4x32-10 (key: the seed, counter: the cell) and Box-Muller, in int64 and float64."""
    mask = 0xFFFFFFFF

    def mulhilo(m, c):
        low, high = m * (c & 0xFFFF), m * (c >> 16)
        return (high + (low >> 16)) >> 16, (low + ((high & mask) << 16)) & mask

    c0 = torch.arange(N ** 3, device="cuda", dtype=torch.int64)
    c1, c2, c3 = (torch.zeros_like(c0) for _ in range(3))
    k0, k1 = seed & mask, (seed >> 32) & mask
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        h0, l0 = mulhilo(0xD2511F53, c0)
        h1, l1 = mulhilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    u1 = (((c0 << 21) | (c1 >> 11)).double() + 1.0) * 2.0 ** -53
    u2 = ((c2 << 21) | (c3 >> 11)).double() * 2.0 ** -53
    return (torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(TWO_PI * u2)).reshape(N, N, N)


def _numbers(N):
    """Lattice wave numbers of the half spectrum along the three axes, index N/2 as +N/2, to broadcast."""
    n = torch.arange(N, device="cuda", dtype=torch.float64)
    n = torch.where(n <= N // 2, n, n - N)
    return n[:, None, None], n[None, :, None], n[None, None, : N // 2 + 1].clone()


def _phi(p, L):
    """Phi~ on the half spectrum: noise, log-normal peak, the map, 2/3."""
    N, dx, kf = p.N, L / p.N, TWO_PI / L
    n = _numbers(N)
    msq = n[0] ** 2 + n[1] ** 2 + n[2] ** 2
    k = kf * torch.sqrt(msq)
    d2 = p.A / math.sqrt(TWO_PI * p.sigma ** 2) * torch.exp(-torch.log(k / p.kstar) ** 2 / (2.0 * p.sigma ** 2))
    amp = torch.sqrt(2.0 * math.pi ** 2 * d2 / k ** 3 * dx ** 3)
    off = (msq == 0) | (n[0] == N // 2) | (n[1] == N // 2) | (n[2] == N // 2)
    zt = torch.where(off, 0.0, amp) * torch.fft.rfftn(_noise(N, p.seed))
    if p.kind == "gauss":
        return zt * (2.0 / 3.0)

    def back(x):
        return torch.fft.irfftn(x, s=(N, N, N)) / dx ** 3

    z = back(zt)
    if p.kind == "local":
        z = z + p.F_NL * (z * z - (z * z).mean()) + p.G_NL * z ** 3
    elif p.kind == "usr":
        z = -torch.log(torch.clamp(1.0 - 3.0 * z, min=p.usr_floor)) / 3.0
    else:
        lap = -kf * kf * msq
        z = z + p.alpha_NL / p.kstar ** 2 * back(lap * torch.fft.rfftn(z * z) * dx ** 3) + \
            p.beta_NL / p.kstar ** 2 * z * back(lap * zt)
    return torch.fft.rfftn(z) * (dx ** 3 * 2.0 / 3.0)


def _tt(n, S):
    """The two TT amplitudes e^l_ij S_ij at the modes n (three vectors) for the six components (00 11 22 01 02 12)."""
    nn = torch.sqrt(n[0] ** 2 + n[1] ** 2 + n[2] ** 2)
    k = [x / nn for x in n]
    flat = k[1] ** 2 + k[2] ** 2 < 1e-24
    zero = torch.zeros_like(nn)
    u = [torch.where(flat, -k[2], zero), torch.where(flat, zero, k[2]), torch.where(flat, k[0], -k[1])]
    un = torch.sqrt(u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    u = [x / un for x in u]
    v = [k[1] * u[2] - k[2] * u[1], k[2] * u[0] - k[0] * u[2], k[0] * u[1] - k[1] * u[0]]
    M = [[S[0], S[3], S[4]], [S[3], S[1], S[5]], [S[4], S[5], S[2]]]

    def dot(a, b):
        return sum(a[i] * M[i][j] * b[j] for i in range(3) for j in range(3))

    return (dot(u, u) - dot(v, v)) / math.sqrt(2.0), math.sqrt(2.0) * dot(u, v)


def _power(Phi, L, edges, term, n_c, M=0):
    """Sum over the shell's modes and both polarisations of |S~|^2, the mode count and, with M, the part of that sum
    each of the M^3 sub-volumes holds (None without M)."""
    N = Phi.shape[0]
    H = N // 2
    n = _numbers(N)
    msq = n[0] ** 2 + n[1] ** 2 + n[2] ** 2
    thr = torch.as_tensor((edges * n_c) ** 2, device="cuda")
    cell = torch.searchsorted(thr, msq, right=True) - 1
    cell = torch.where((cell < 0) | (cell >= len(edges) - 1), len(edges) - 1, cell)
    q = [1j * (TWO_PI / L) * torch.where(x == H, 0.0, x) for x in n]
    sigma, phi = (torch.as_tensor(x, device="cuda") for x in term)
    phi = torch.cat((phi, torch.zeros_like(phi[:, :1])), 1)
    dx3 = (L / N) ** 3
    S = torch.zeros((6, N, N, N), device="cuda", dtype=torch.float64)
    step = max(1, min(len(sigma), 2 ** 22 // N ** 3))
    for a in range(0, len(sigma), step):
        V = phi[a:a + step][:, cell] * Phi
        G = [torch.fft.irfftn(x * V, s=(N, N, N), dim=(1, 2, 3)) / dx3 for x in q]
        del V
        sg = sigma[a:a + step, None, None, None]
        for c, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            S[c] += (sg * G[i] * G[j]).sum(0)
    at = torch.nonzero((msq >= n_c * n_c - n_c + 1) & (msq <= n_c * n_c + n_c), as_tuple=True)
    vals = [torch.fft.rfftn(S[c])[at] * dx3 for c in range(6)]
    modes = [n[0].flatten()[at[0]], n[1].flatten()[at[1]], n[2].flatten()[at[2]]]
    pair = (modes[2] > 0) & (modes[2] < H)  # a stored mode that also stands for its partner -n
    plus, cross = _tt(modes, vals)
    total = (plus.abs() ** 2 + cross.abs() ** 2).sum()
    minus = [torch.where(x == H, x, -x)[pair] for x in modes]
    pp, pc = _tt(minus, [x[pair].conj() for x in vals])
    total = total + (pp.abs() ** 2 + pc.abs() ** 2).sum()
    count = int(len(modes[0]) + pair.sum())
    if not M:
        return float(total), count, None
    e = torch.zeros((N, N, N), device="cuda", dtype=torch.float64)
    for amp in (plus, -1j * cross):
        X = torch.zeros_like(Phi)
        X[at] = amp
        e += torch.fft.irfftn(X, s=(N, N, N)) ** 2
    s = N // M
    return float(total), count, (e.reshape(M, s, M, s, M, s).sum((1, 3, 5)).flatten() * N ** 3).cpu().numpy()


def _spectrum(p, L, dec, shells, M=0):
    """omega, PA, PB over `shells` and, with M, their jackknife errors."""
    edges, terms = dec
    Phi = _phi(p, L)
    V = L ** 3
    keys = ("omega", "PA", "PB") + (("sigma_omega", "sigma_PA", "sigma_PB") if M else ())
    out = {k: [] for k in keys}
    for n_c in shells:
        kc = n_c * TWO_PI / L
        P, rep = [], []
        for m in (0, 1):
            total, count, E = _power(Phi, L, edges, terms[m], n_c, M)
            f = (4.0 / kc ** 2) ** 2 / (V * count)
            P.append(f * total)
            if M:
                rep.append(f * (E.sum() - E) / (1.0 - M ** -3))
        g = kc ** 3 / (48.0 * math.pi ** 2)
        for k, x in zip(("omega", "PA", "PB"), (g * (P[0] + P[1]), P[0], P[1])):
            out[k].append(x)
        if M:
            for k, x in zip(("sigma_omega", "sigma_PA", "sigma_PB"), (g * (rep[0] + rep[1]), rep[0], rep[1])):
                out[k].append(math.sqrt((M ** 3 - 1) / M ** 3 * ((x - x.mean()) ** 2).sum()))
    return {k: np.array(v) for k, v in out.items()}


def _seconds(N, n_alpha, shells):
    """Rough time of _spectrum."""
    return shells * max(2 * (3 * n_alpha + 6) * 3.5e-3 * (N / 256) ** 3, 0.02)


def exact(case, seed):
    op, N = case["op"], case["N"]
    if op == "fft":
        x = _fft_input(case, seed)
        if case["direction"] < 0:
            return torch.fft.rfftn(x.double())
        return torch.fft.irfftn(x.to(torch.complex128), s=(N, N, N)) * N ** 3
    dec = _separable(case["n_alpha"])
    if op == "scan":
        p = SimpleNamespace(N=N, G_NL=0.0, usr_floor=1e-6, **_scan_point(case, seed))
        k, om, Ls = _targets(case), [], []
        kbar = p.kstar * math.exp(p.sigma * math.sqrt(2.0) * float(torch.erfinv(torch.tensor(0.8, dtype=torch.float64))))
        for x in k:
            n_c = max(1, min(N // 2, int(math.floor(x * N / (6.0 * max(x, kbar)) + 0.5))))
            Ls.append(TWO_PI * n_c / x)
            om.append(_spectrum(p, Ls[-1], dec, [n_c])["omega"][0])
        return {"omega": np.array(om), "L": np.array(Ls), "n_c": None}
    points = _points(case, seed)
    if op == "serve":
        out, left = [], 15.0
        for p in points:
            t = _seconds(p.N, case["n_alpha"], p.N // 2)
            out.append(_spectrum(p, p.L, dec, range(1, p.N // 2 + 1))["omega"] if t <= left else None)
            left -= t if t <= left else 0.0
        return out
    M = case.get("M", 0)
    shells = _shells(case) or range(1, N // 2 + (0 if M else 1))
    out, left = None, 15.0
    for p in points:  # as many realisations as the time allows
        t = _seconds(N, case["n_alpha"], len(shells))
        got = _spectrum(p, p.L, dec, shells, M) if t <= left else None
        left -= t if t <= left else 0.0
        if out is None:
            if got is None:
                return None
            out = {k: [] for k in got}
        for k in out:
            out[k].append(None if got is None else got[k])
    return {"hits": None, **({} if M else {"Nk": None}), **out}
