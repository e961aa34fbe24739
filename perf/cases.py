"""The work that a user of this library has it do, as cases to be timed.

Every case goes through the public entry points of paper_2212_05685_gb300 (the
ctypes binding of libkpm.so and the autograd function), with the library's own
defaults: one self-consistency iteration or one KPM pass of a two-vortex cell
of the t-t'-J model, its gradient, its local density of states, or the O(N)
setup calls.  Lattices, orders and temperatures are those of the library's
workloads (inputs.py), its tests and the ranges the paper states (orders 1000
to 2000, 64 to 144 probing vectors, 48 x 48 to 96 x 96 sites).

`exact` restates the method in 64 bits with torch and numpy alone: the
functional's derivatives by automatic differentiation, the Chebyshev recursion
as a sparse matrix times the start vectors, the update, the adjoint recursion
and the resolvent series.
"""
import math

import numpy as np
import torch

from paper_2212_05685_gb300 import autograd, kpm

T_NN, T_NNN, J_EX = 1.0, -0.3, 0.3
MARGIN = 0.01
FWD = ((1, 0), (0, 1), (1, 1), (1, -1))
NN4 = ((1, 0), (0, 1), (-1, 0), (0, -1))
PRECISION = {"fp64": kpm.KPM_FP64, "fp32": kpm.KPM_FP32, "df64": kpm.KPM_DF64}
BATCH_SHAPES = ((24, 12), (32, 16), (48, 24), (64, 32))


def _case(name, kind, nx, ny, M, precision="fp32", doping=0.125, half=False, probe_p=0, temperature=0.0, share=0,
          iterations=0, cells=0, frequencies=0):
    c = dict(kind=kind, nx=nx, ny=ny, M=M, precision=precision, doping=doping, half=half, probe_p=probe_p,
             temperature=temperature, share=share, iterations=iterations, cells=cells, frequencies=frequencies)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the O(N) calls around a pass, as a driver that builds its own loop makes them: latency alone
        _case("setup_100x100", "setup", 100, 100, 0, "fp64"),
        # the smallest workload cell in the precision its trajectories are checked in
        _case("pass_16x16_fp64", "pass", 16, 16, 256, "fp64"),
        # an odd lattice at a finite temperature and an order that is no power of two
        _case("pass_37x29_fp32_warm", "pass", 37, 29, 777, doping=0.15, temperature=0.05),
        # the benchmark cell: every unit vector, vectors far larger than L2
        _case("pass_100x100_fp32", "pass", 100, 100, 1024),
        # one rank's sites of that cell when eight share it
        _case("shard_100x100_fp32", "pass", 100, 100, 1024, share=8),
        # the cell that is taken to self-consistency: most of its iterations run in FP32 ...
        _case("iterate_48x24_fp32", "iterate", 48, 24, 1024, doping=0.15, iterations=3),
        # ... and the last ones in double-float
        _case("iterate_48x24_df64", "iterate", 48, 24, 1024, "df64", doping=0.15, iterations=1),
        # the paper's largest lattice, in the sector that needs half of the unit vectors
        _case("iterate_96x96_half_fp32", "iterate", 96, 96, 1000, half=True, iterations=1),
        # the same lattice with the paper's own estimator: 128 probing vectors
        _case("iterate_96x96_probing_fp32", "iterate", 96, 96, 2000, probe_p=8, iterations=1),
        # a doping series: cells of uneven size solved together
        _case("batched_12_cells_fp32", "batched", 0, 0, 1024, iterations=1, cells=12),
        # forward and backward through the autograd function
        _case("gradient_48x48_fp32", "gradient", 48, 48, 512),
        # a spectrum after convergence, from probing moments
        _case("ldos_100x100_fp32", "ldos", 100, 100, 8192, probe_p=10, frequencies=101),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the kinds in about the listed proportions, the sizes over their whole range."""
    while True:
        kind = rng.choice(("setup", "pass", "pass", "pass", "shard", "iterate", "iterate", "half", "probing",
                           "batched", "gradient", "ldos"))
        nx, ny = _log_int(rng, 8, 100), _log_int(rng, 8, 100)
        M = _log_int(rng, 64, 2048)
        doping = round(rng.uniform(0.05, 0.30), 3)
        prec = rng.choice(("fp32", "fp32", "fp32", "fp64", "df64"))
        p = rng.choice((4, 5, 6, 8, 10))
        px, py = p * max(2, nx // p), p * max(2, ny // p)
        if kind == "setup":
            c = _case(None, "setup", nx, ny, 0, "fp64", doping)
        elif kind == "pass":
            c = _case(None, "pass", nx, ny, M, prec, doping, temperature=rng.choice((0.0, 0.0, 0.02, 0.1)))
        elif kind == "shard":
            c = _case(None, "pass", nx, ny, M, "fp32", doping, share=rng.choice((2, 4, 8)))
        elif kind == "iterate":
            c = _case(None, "iterate", nx, ny, M, prec, doping, iterations=rng.choice((1, 2, 3)))
        elif kind == "half":
            c = _case(None, "iterate", nx, ny, M, prec, doping, half=True, iterations=1)
        elif kind == "probing":
            c = _case(None, "iterate", px, py, M, "fp32", doping, probe_p=p, iterations=rng.choice((1, 2)))
        elif kind == "batched":
            c = _case(None, "batched", 0, 0, M, "fp32", iterations=1, cells=rng.randint(2, 16))
        elif kind == "gradient":
            c = _case(None, "gradient", nx, ny, M, rng.choice(("fp32", "fp32", "fp64")), doping)
        else:
            c = _case(None, "ldos", px, py, _log_int(rng, 1024, 8192), "fp32", doping, probe_p=p,
                      frequencies=rng.randint(20, 120))
        if _seconds(c) <= 0.6:
            return c


def _vectors(c):
    """Start vectors of one pass of the case."""
    D = 2 * c["nx"] * c["ny"]
    if c["probe_p"]:
        return 2 * c["probe_p"] ** 2
    if c["share"]:
        return 2 * (c["nx"] * c["ny"] // c["share"])
    return D // 2 if c["half"] else D


def _batch(c):
    """(nx, ny, doping) of the cells of a batch: a doping series over cells of four sizes."""
    n = c["cells"]
    return [BATCH_SHAPES[(3 * k + 1) % 4] + (round(0.05 + 0.25 * k / max(1, n - 1), 3),) for k in range(n)]


def _row_steps(c):
    """(rows x start vectors x recursion steps) of the case."""
    if c["kind"] == "setup":
        return 0.0
    if c["kind"] == "batched":
        return float(sum((2 * nx * ny) ** 2 for nx, ny, _ in _batch(c))) * (c["M"] - 1) * c["iterations"]
    passes = c["iterations"] if c["kind"] == "iterate" else 3 if c["kind"] == "gradient" else 1
    return 2.0 * c["nx"] * c["ny"] * _vectors(c) * (c["M"] - 1) * passes


def _seconds(c):
    """A rough cost, to keep a drawn case below the largest listed one."""
    rate = {"fp32": 6e-12, "df64": 5e-11, "fp64": 1.2e-10}[c["precision"]]
    return _row_steps(c) * rate + 1e-5 * c["M"] * max(1, c["iterations"])


def work(case):
    """Each input read once and each output written once; a row of a recursion step takes twelve complex
    multiply-adds, one real one and a subtraction (the gradient: a forward and a backward recursion and the
    thirteen products of a row that it sums)."""
    flops = _row_steps(case) * 102.0
    if case["kind"] == "batched":
        sites = sum(nx * ny for nx, ny, _ in _batch(case))
    else:
        sites = case["nx"] * case["ny"]
    words = {"setup": 4 + 26 + 26 + 26 + 3, "pass": 26 + 26, "iterate": 4 + 26 + 26, "batched": 4 + 26 + 26,
             "gradient": 26 + 26 + 26 + 26, "ldos": 26 + 26 + 2 * case["frequencies"]}[case["kind"]]
    if case["kind"] == "setup":
        flops = 1200.0 * sites
    if case["kind"] == "ldos":
        flops += 4.0 * case["M"] * case["frequencies"] * sites
    return {"bytes": 8.0 * words * sites, "flops": flops}


# ---------------------------------------------------------------- inputs

def _cell(nx, ny, doping, seed, pdw=0.0):
    """Order parameters of a two-vortex cell (26 N doubles: n, chi, F), seeded noise on bonds and pairing."""
    N = nx * ny
    rng = np.random.default_rng(seed)
    x, y = np.arange(N) % nx, np.arange(N) // nx
    n = np.full((2, N), 0.5 * (1.0 - doping)) + 0.01 * rng.uniform(-1, 1, size=N)
    chi = 0.2 * (1.0 + 0.05 * rng.uniform(-1, 1, size=(4, N)))
    chi = np.stack([chi, chi]).astype(np.complex128)
    F = np.zeros((4, N), dtype=np.complex128)
    noise = rng.uniform(-1, 1, size=(2, N))
    for b, (dx, dy) in enumerate(((1, 0), (0, 1))):
        X, Y = x + 0.5 * dx, y + 0.5 * dy
        amp, theta = np.ones(N), np.zeros(N)
        for vx, vy in ((nx // 4, ny // 2), ((3 * nx) // 4, ny // 2)):
            rx, ry = X - vx, Y - vy
            rx, ry = rx - nx * np.floor(rx / nx + 0.5), ry - ny * np.floor(ry / ny + 0.5)
            amp *= np.tanh(np.hypot(rx, ry) / 2.0)
            theta += np.arctan2(ry, rx)
        val = 0.1 * amp * np.exp(1j * theta) * (1.0 + 0.1 * noise[b])
        val += pdw * (np.cos(2 * np.pi * X / 8) + np.cos(2 * np.pi * Y / 8))
        val *= 1.0 if b == 0 else -1.0
        F[b] = val
        F[b + 2][(x + dx) % nx + nx * ((y + dy) % ny)] = val
    return np.concatenate([n.reshape(-1), chi.reshape(-1).view(np.float64), F.reshape(-1).view(np.float64)])


def _params(c, seed):
    return _cell(c["nx"], c["ny"], c["doping"], seed, 0.02 if c["nx"] >= 96 else 0.0)


def _site_range(c):
    N = c["nx"] * c["ny"]
    k = N // c["share"]
    return k, 2 * k  # the second rank's sites


def _opts(c):
    begin, end = _site_range(c) if c["share"] else (0, 0)
    return kpm.make_opts(c["M"], PRECISION[c["precision"]], flags=kpm.KPM_FLAG_PH_HALF if c["half"] else 0,
                         probe_p=c["probe_p"], probe_seed=7, temperature=c["temperature"], site_begin=begin,
                         site_end=end)


def _omegas(c):
    return np.linspace(-0.5, 0.5, c["frequencies"])


def _gradient_seed(N, seed):
    rng = np.random.default_rng(seed + 1000003)
    return rng.standard_normal(26 * N), float(rng.uniform(0.1, 0.5))


def _empty(n):
    return torch.empty(n, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    """The library context and the device arrays a user's program has before the call."""
    c = case
    ctx = kpm.kpm_create(0)
    if c["kind"] == "batched":
        s = dict(case=c, ctx=ctx, models=[], phis=[], seeds=[], params=[], ropts=[])
        for k, (nx, ny, doping) in enumerate(_batch(c)):
            model, phi = kpm.make_model(nx, ny, T_NN, T_NNN, J_EX), _empty(4 * nx * ny)
            kpm.kpm_peierls_phases(ctx, model, phi)
            s["models"].append(model)
            s["phis"].append(phi)
            s["seeds"].append(torch.tensor(_cell(nx, ny, doping, 64 * seed + k), device="cuda"))
            s["params"].append(_empty(26 * nx * ny))
            s["ropts"].append(kpm.make_rmft_opts(1.0 - doping, tol=1e-9))
        s["mu"] = _empty(c["cells"])
        s["opts"] = kpm.make_opts(c["M"], PRECISION[c["precision"]])
        return s
    N = c["nx"] * c["ny"]
    model = kpm.make_model(c["nx"], c["ny"], T_NN, T_NNN, J_EX)
    s = dict(case=c, ctx=ctx, model=model, phi=_empty(4 * N), seed=torch.tensor(_params(c, seed), device="cuda"))
    if c["kind"] == "setup":
        s.update(fields=_empty(26 * N), w=_empty(1), ab=_empty(2), delta=_empty(2 * N), mag=_empty(N))
        return s
    kpm.kpm_peierls_phases(ctx, model, s["phi"])
    s["opts"] = _opts(c)
    if c["kind"] == "iterate":
        s.update(params=_empty(26 * N), mu=_empty(1), ropts=kpm.make_rmft_opts(1.0 - c["doping"], tol=1e-9))
        return s
    s.update(fields=_empty(26 * N), ab=_empty(2), obs=_empty(26 * N), omega=_empty(1))
    kpm.kpm_build_H(ctx, model, s["phi"], s["seed"], 0.1, s["fields"])
    kpm.kpm_bounds(ctx, model, s["fields"], MARGIN, s["ab"])
    if c["kind"] == "gradient":
        g, s["g_omega"] = _gradient_seed(N, seed)
        s["g"] = torch.tensor(g, device="cuda")
        s["fields"].requires_grad_(True)
    elif c["kind"] == "ldos":
        s["ldos"] = _empty(2 * c["frequencies"] * N)
        s["freq"] = torch.tensor(_omegas(c), device="cuda")
    return s


def run(s):
    c, ctx = s["case"], s["ctx"]
    if c["kind"] == "setup":
        kpm.kpm_peierls_phases(ctx, s["model"], s["phi"])
        kpm.kpm_build_H(ctx, s["model"], s["phi"], s["seed"], 0.1, s["fields"], s["w"])
        kpm.kpm_bounds(ctx, s["model"], s["fields"], MARGIN, s["ab"])
        kpm.kpm_order_parameters(ctx, s["model"], s["phi"], s["seed"], s["delta"], s["mag"])
        return [s["phi"], s["fields"], s["w"], s["ab"], s["delta"], s["mag"]]
    if c["kind"] == "pass":
        kpm.kpm_observables(ctx, s["model"], s["opts"], s["fields"], s["ab"], s["obs"], s["omega"])
        return [s["obs"], s["omega"]]
    if c["kind"] == "iterate":
        s["params"].copy_(s["seed"])
        s["mu"].zero_()
        _, st = kpm.rmft_iterate(ctx, s["model"], s["opts"], s["ropts"], s["phi"], s["params"], s["mu"],
                                 c["iterations"])
        return [s["params"], s["mu"], st.residual, st.mu, st.omega]
    if c["kind"] == "batched":
        for p, q in zip(s["params"], s["seeds"]):
            p.copy_(q)
        s["mu"].zero_()
        _, st = kpm.rmft_iterate_batched(ctx, s["models"], s["opts"], s["ropts"], s["phis"], s["params"], s["mu"],
                                         c["iterations"])
        return [s["params"], s["mu"], [x.omega for x in st]]
    if c["kind"] == "gradient":
        s["fields"].grad = None
        obs, omega = autograd.observables(ctx, s["model"], s["opts"], s["fields"], s["ab"])
        ((obs * s["g"]).sum() + s["g_omega"] * omega.sum()).backward()
        return [obs.detach(), omega.detach(), s["fields"].grad]
    kpm.kpm_ldos(ctx, s["model"], s["opts"], s["fields"], s["ab"], s["seed"], s["freq"], s["ldos"])
    return [s["ldos"]]


# ---------------------------------------------------------------- the same in 64 bits

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Lattice:
    """Neighbour tables, Peierls phases and local rows of an nx x ny torus with one flux quantum."""

    def __init__(self, nx, ny):
        self.nx, self.ny, self.N = nx, ny, nx * ny
        dev = _device()
        x, y = np.arange(self.N) % nx, np.arange(self.N) // nx

        def to(d):
            return torch.tensor((x + d[0]) % nx + nx * ((y + d[1]) % ny), device=dev)

        self.fwd, self.nn = [to(d) for d in FWD], [to(e) for e in NN4]
        f = 2.0 * math.pi / self.N
        phi = []
        for dx, dy in FWD:
            ph = -f * dy * (x + 0.5 * dx)
            phi.append(np.where(x + dx >= nx, ph + 2.0 * math.pi * ((y + dy) % ny) / ny, ph))
        self.phi = torch.tensor(np.array(phi), device=dev)
        # rows read off column (i, beta): itself, the forward neighbours, the other component of the nn sites
        i = torch.arange(self.N, device=dev)
        self.rows = [torch.stack([2 * i + b] + [2 * j + b for j in self.fwd] + [2 * j + 1 - b for j in self.nn])
                     for b in (0, 1)]


def _split(p, N):
    return (p[:2 * N].reshape(2, N), torch.view_as_complex(p[2 * N:18 * N].reshape(2, 4, N, 2)),
            torch.view_as_complex(p[18 * N:].reshape(4, N, 2)))


def _join(n, chi, F):
    return torch.cat([n.reshape(-1), torch.view_as_real(chi.contiguous()).reshape(-1),
                      torch.view_as_real(F.contiguous()).reshape(-1)])


def _factors(n):
    """g^t of both spins and g^{s,xy} (n_up = n_dn: g^{s,z} = g^{s,xy})."""
    delta, m = 1.0 - n[0] - n[1], 0.5 * (n[0] - n[1])
    P = 1.0 - delta ** 2 + 4.0 * m ** 2
    gt = [torch.sqrt(2.0 * delta * (1.0 - delta) / P * (1.0 + delta + 2.0 * s * m) / (1.0 + delta - 2.0 * s * m))
          for s in (1.0, -1.0)]
    return gt, 2.0 * (1.0 - delta) / P, m


def _fields(L, p, mu):
    """(dW/d(n, chi, F*), W) of the renormalised functional."""
    p = p.detach().clone().requires_grad_(True)
    n, chi, F = _split(p, L.N)
    gt, gxy, m = _factors(n)
    W = -mu * n.sum()
    for d, t in enumerate((T_NN, T_NN, T_NNN, T_NNN)):
        hop = t * torch.exp(1j * L.phi[d])
        for s in (0, 1):
            W = W - 2.0 * (gt[s] * gt[s][L.fwd[d]] * (hop * chi[s, d]).real).sum()
    for d in (0, 1):
        j = L.fwd[d]
        Fij, Fji, cu, cd = F[d], F[d + 2][j], chi[0, d], chi[1, d]
        S = cu.abs() ** 2 + cd.abs() ** 2 + Fij.abs() ** 2 + Fji.abs() ** 2
        Q = (cu * cd.conj() + Fij.conj() * Fji).real
        W = W + J_EX * (gxy * gxy[j] * (m * m[j] - 0.25 * S - Q)).sum()
    g, = torch.autograd.grad(W, p)
    eps, T, D = _split(g, L.N)
    return _join(eps, 0.5 * T.conj(), 0.5 * D), W.detach()


def _entries(L, fields):
    """(rows, columns, values) of the Nambu matrix."""
    eps, T, D = _split(fields, L.N)
    i = torch.arange(L.N, device=fields.device)
    r, c, v = [2 * i, 2 * i + 1], [2 * i, 2 * i + 1], [eps[0] + 0j, -eps[1] + 0j]
    for d, j in enumerate(L.fwd):
        r += [2 * i, 2 * j, 2 * i + 1, 2 * j + 1]
        c += [2 * j, 2 * i, 2 * j + 1, 2 * i + 1]
        v += [T[0, d], T[0, d].conj(), -T[1, d].conj(), -T[1, d]]
    for e, j in enumerate(L.nn):
        r += [2 * i, 2 * j + 1]
        c += [2 * j + 1, 2 * i]
        v += [-D[e], -D[e].conj()]
    return torch.cat(r), torch.cat(c), torch.cat([x.resolve_conj() for x in v])


def _bounds(L, fields, symmetric=False):
    r, c, v = _entries(L, fields)
    D = 2 * L.N
    R = torch.zeros(D, dtype=torch.float64, device=v.device).index_add_(0, r[D:], v[D:].abs())
    diag = torch.zeros_like(R).index_add_(0, r[:D], v[:D].real)
    hi, lo = float((diag + R).max()), float((diag - R).min())
    if symmetric:
        return (1.0 + MARGIN) * max(hi, -lo), 0.0
    return (1.0 + MARGIN) * 0.5 * (hi - lo), 0.5 * (hi + lo)


def _matrix(L, fields, a, b):
    r, c, v = _entries(L, fields)
    D = 2 * L.N
    v = v.clone()
    v[:D] -= b
    return torch.sparse_coo_tensor(torch.stack([r, c]), v / a, (D, D)).coalesce().to_sparse_csr()


def _coefficients(M, a, b, T):
    m, q = np.arange(M, dtype=np.float64), math.pi / (M + 1)
    g = ((M - m + 1) * np.cos(q * m) + np.sin(q * m) / math.tan(q)) / (M + 1)
    if T > 0.0:
        th = math.pi * (np.arange(4 * M) + 0.5) / (4 * M)
        e = a * np.cos(th) + b
        cosines = np.cos(m[:, None] * th[None, :])
        c = cosines @ (0.5 * (1.0 - np.tanh(0.5 * e / T))) / (4 * M)
        co = cosines @ (-T * np.logaddexp(0.0, -e / T) / a) / (4 * M)
    else:
        x0 = -b / a
        th = math.acos(x0)

        def S(k):
            k = np.abs(k)
            return np.where(k == 0, math.pi - th, -np.sin(k * th) / np.where(k == 0, 1.0, k))

        c, co = S(m) / math.pi, (0.5 * (S(m + 1) + S(m - 1)) - x0 * S(m)) / math.pi
    two = np.where(m == 0, 1.0, 2.0)
    return two * g * c, two * g * co


def _recursion(h, V, M):
    """T_m(h) V for m = 0 .. M - 1, in turn."""
    yield V
    if M < 2:
        return
    U, V = V, h @ V
    yield V
    for _ in range(2, M):
        U, V = V, 2.0 * (h @ V) - U
        yield V


def _phases(D, seed):
    k = np.arange(D, dtype=np.uint64) + (np.uint64(seed) << np.uint64(32))
    z = k + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    u = ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    return torch.tensor(np.exp(2j * math.pi * u), device=_device())


def _start(L, c):
    """(start vectors, sources J, their columns, their weights) of a pass."""
    D, dev = 2 * L.N, _device()
    if c["probe_p"]:
        p, K = c["probe_p"], torch.arange(D, device=dev)
        x, y = (K // 2) % L.nx, (K // 2) // L.nx
        colour = K % 2 + 2 * (x % p + p * (y % p))
        xi = _phases(D, 7)
        V = torch.zeros(D, 2 * p * p, dtype=torch.complex128, device=dev)
        V[K, colour] = xi
        return V, K, colour, xi.conj().resolve_conj()
    begin, end = _site_range(c) if c["share"] else (0, L.N)
    J = torch.arange(2 * begin, 2 * end, device=dev)
    V = torch.zeros(D, len(J), dtype=torch.complex128, device=dev)
    V[J, J - 2 * begin] = 1.0
    return V, J, J - 2 * begin, torch.ones(len(J), dtype=torch.complex128, device=dev)


def _pass(L, c, fields, a, b):
    am, ao = _coefficients(c["M"], a, b, c["temperature"])
    V, J, col, w = _start(L, c)
    rows = torch.stack([L.rows[0][:, J[0::2] // 2], L.rows[1][:, J[1::2] // 2]], dim=2).reshape(9, -1)
    acc = torch.zeros(9, len(J), dtype=torch.complex128, device=V.device)
    om = torch.zeros((), dtype=torch.float64, device=V.device)
    for m, T in enumerate(_recursion(_matrix(L, fields, a, b), V, c["M"])):
        e = w * T[rows, col]
        acc += am[m] * e
        om += ao[m] * e[0].real.sum()
    begin, end = _site_range(c) if c["share"] else (0, L.N)
    n = torch.zeros(2, L.N, dtype=torch.float64, device=V.device)
    chi = torch.zeros(2, 4, L.N, dtype=torch.complex128, device=V.device)
    F = torch.zeros(4, L.N, dtype=torch.complex128, device=V.device)
    n[0, begin:end], n[1, begin:end] = acc[0, 0::2].real, 1.0 - acc[0, 1::2].real
    chi[0, :, begin:end], chi[1, :, begin:end] = acc[1:5, 0::2], -acc[1:5, 1::2].conj()
    F[:, begin:end] = -acc[5:9, 0::2].conj()
    return _join(n, chi, F), a * om


def _iterate(L, c, p):
    mu_eff, N = 0.0, L.N
    for _ in range(c["iterations"]):
        fields, _ = _fields(L, p, 0.0)
        mean = float(fields[:2 * N].mean())
        fields[:2 * N] -= mean + mu_eff
        a, b = _bounds(L, fields, c["half"])
        o, omega = _pass(L, c, fields, a, b)
        mu = mu_eff + mean
        o[:2 * N] = (0.5 * (o[:N] + o[N:2 * N])).repeat(2)
        e = float(o[:2 * N].sum()) / N - (1.0 - c["doping"])
        o[:2 * N] -= 0.5 * e
        residual = float((o - p).abs().max())
        q = 0.5 * p + 0.5 * o
        q[:2 * N] = 0.95 * p[:2 * N] + 0.05 * o[:2 * N]
        p, mu_eff = q, mu_eff - 0.5 * e
    return p, mu_eff, residual, mu, omega


def _gradient(L, c, fields, a, b, g, g_omega):
    """d(<g, obs> + g_omega Omega)/d fields at fixed (a, b), by the backward recursion; the forward vectors
    are run backwards from the last two."""
    N, M, D = L.N, c["M"], 2 * L.N
    am, ao = _coefficients(M, a, b, c["temperature"])
    gn, gc, gF = _split(g, N)
    W = torch.zeros(9, D, dtype=torch.complex128, device=g.device)
    W[0, 0::2], W[0, 1::2] = gn[0] + 0j, -gn[1] + 0j
    W[1:5, 0::2], W[1:5, 1::2], W[5:9, 0::2] = gc[0], -gc[1].conj(), -gF.conj()
    rows = torch.stack([L.rows[0], L.rows[1]], dim=2).reshape(9, D)
    J = torch.arange(D, device=g.device)
    h = _matrix(L, fields, a, b)
    V, *_ = _start(L, c)
    hi = lo = None
    for T in _recursion(h, V, M):
        hi, lo = T, hi
    r, k, _ = _entries(L, fields)
    G = torch.zeros(len(r), dtype=torch.complex128, device=g.device)
    lam, lam1 = torch.zeros_like(V), torch.zeros_like(V)
    for m in range(M - 1, 0, -1):
        if m < M - 1:
            hi, lo = lo, 2.0 * (h @ lo) - hi
        lam, lam1 = 2.0 * (h @ lam) - lam1, lam
        for s in range(9):
            lam[rows[s], J] += am[m] * W[s]
        lam[J, J] += ao[m] * a * g_omega
        f = 1.0 if m == 1 else 2.0
        for at in range(0, len(r), D):
            q = slice(at, at + D)
            G[q] += f * torch.linalg.vecdot(lo[k[q]], lam[r[q]])
    # the blocks of _entries: diagonals, then per bond the entry and its mirror image (two spins), then the pairings
    G = (G / a).reshape(-1, N)
    eps = torch.stack([G[0].real, -G[1].real])
    T = torch.stack([torch.stack([G[2 + 4 * d] + G[3 + 4 * d].conj() for d in range(4)]),
                     torch.stack([-(G[4 + 4 * d].conj() + G[5 + 4 * d]) for d in range(4)])])
    P = torch.stack([-(G[18 + 2 * e] + G[19 + 2 * e].conj()) for e in range(4)])
    return _join(eps, T.resolve_conj(), P.resolve_conj())


def _ldos(L, c, p, fields, a, b):
    M, om = c["M"], _omegas(c)
    V, J, col, w = _start(L, c)
    mu = torch.empty(M, 2 * L.N, dtype=torch.float64, device=V.device)
    for m, T in enumerate(_recursion(_matrix(L, fields, a, b), V, M)):
        mu[m] = (w * T[J, col]).real
    gt = _factors(_split(p, L.N)[0])[0]
    out = []
    for s, sign in ((0, 1.0), (1, -1.0)):
        z = (sign * om + 1j * (0.25 * np.abs(om) + 3e-4) - b) / a
        root = np.sqrt(z * z - 1.0 + 0j)
        root = np.where(np.abs(z - root) > 1.0, -root, root)
        k = 2.0 * (z - root)[:, None] ** np.arange(M)[None, :] / root[:, None]
        k[:, 0] *= 0.5
        out.append(-(torch.tensor(k.imag / a, device=mu.device) @ mu[:, s::2]) / math.pi * gt[s] ** 2)
    return torch.stack(out).reshape(-1)


def exact(case, seed):
    c = case
    steps = _row_steps(c)
    if steps * (3 if c["kind"] == "gradient" else 1) > 1.1e11:
        return None  # minutes in 64 bits
    dev = _device()
    if c["kind"] == "batched":
        got = []
        for k, (nx, ny, doping) in enumerate(_batch(c)):
            one = dict(c, nx=nx, ny=ny, doping=doping, kind="iterate")
            got.append(_iterate(_Lattice(nx, ny), one, torch.tensor(_cell(nx, ny, doping, 64 * seed + k), device=dev)))
        return [[x[0] for x in got], torch.tensor([x[1] for x in got], dtype=torch.float64),
                [float(x[4]) for x in got]]
    L = _Lattice(c["nx"], c["ny"])
    p = torch.tensor(_params(c, seed), device=dev)
    if c["kind"] == "iterate":
        q, mu_eff, residual, mu, omega = _iterate(L, c, p)
        return [q, torch.tensor([mu_eff], dtype=torch.float64), residual, mu, float(omega)]
    fields, W = _fields(L, p, 0.1)
    a, b = _bounds(L, fields)
    if c["kind"] == "setup":
        n, chi, F = _split(p, L.N)
        gt = _factors(n)[0]
        delta = torch.zeros(L.N, dtype=torch.complex128, device=dev)
        for e, (dx, dy) in enumerate(NN4):
            j = L.nn[e]
            ph = L.phi[e] if e < 2 else -L.phi[e - 2][j]
            delta += (1.0 if dy == 0 else -1.0) * torch.exp(1j * ph) * (
                gt[0] * gt[0][j] * F[e] + gt[1] * gt[1][j] * F[(e + 2) % 4][j]) / 8.0
        return [L.phi.reshape(-1), fields, W.reshape(1), torch.tensor([a, b], dtype=torch.float64),
                torch.view_as_real(delta).reshape(-1), torch.zeros(L.N, dtype=torch.float64)]
    if c["kind"] == "pass":
        obs, omega = _pass(L, c, fields, a, b)
        return [obs, omega.reshape(1)]
    if c["kind"] == "gradient":
        g, g_omega = _gradient_seed(L.N, seed)
        obs, omega = _pass(L, c, fields, a, b)
        return [obs, omega.reshape(1), _gradient(L, c, fields, a, b, torch.tensor(g, device=dev), g_omega)]
    return [_ldos(L, c, p, fields, a, b)]
