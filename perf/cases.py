"""The work that users of this library have it do, as cases that can be timed and compared.

Every case goes through the public entry points of paper_2210_01837_gb300.binding, with what a user's
program keeps between calls (a Plan, a Lanczos handle) made in prepare().  The sizes are those of the
workload generators (paper_2210_01837_gb300.workloads), of the benchmark and of the tests.

Mixed-precision plans compute in 32 bits and deliver 32-bit results in 64-bit arrays; their cases
hand the results on in 32 bits, the precision that they have.  FP64 plans' results stay 64-bit.
"""

import math

import numpy as np
import torch

from paper_2210_01837_gb300 import binding, workloads

# (height of the box, lowest and highest particle height) per wall mode: the served population's
DOMAINS = {"bottom_wall": (12.0, 1.2, 10.0), "slit": (20.0, 1.2, 18.8), "free": (20.0, 2.0, 18.0)}
LAYER_H = 8.0                # sedimented rollers: heights max(|N(1.6, 0.3)|, 1.05) above one wall
BETA5 = (5 * 1.305, 5 * 2.232)   # monopole and dipole kernels of 5 points (force and torque)
CACHE_BYTES = 129e6


def listed():
    return [
        # The smallest call in double precision: 100 spheres above a wall, forces only, the
        # accuracy reference's own configuration.  Latency and launches count.
        _case("spheres_100_fp64", "apply", "bottom_wall", "fp64", "none", 100, 128, 65, L=64.0, m=6, beta=10.2),
        # One of the small systems of a batch or a served stream: a few hundred particles in a slit.
        _case("slit_317_mixed", "apply", "slit", "mixed", "spectral_curl", 317, 120, 33),
        # The slit suspension with forces and torques: the ordinary product ...
        _case("slit_16k_mixed", "apply", "slit", "mixed", "spectral_curl", 16384, 384, 97, L=256.0),
        # ... and the same in double precision, for users who need all digits.
        _case("slit_16k_fp64", "apply", "slit", "fp64", "spectral_curl", 16384, 384, 97, L=256.0),
        # Sedimented microrollers above a wall, gravity and torque: a tile of the layer ...
        _case("rollers_64k_mixed", "apply", "bottom_wall", "mixed", "spectral_curl", 65536, 768, 65, L=512.0,
              fill="layer"),
        # ... and the whole layer of a million, the largest call.
        _case("rollers_1m_mixed", "apply", "bottom_wall", "mixed", "spectral_curl", 1048576, 3072, 65, L=2048.0,
              fill="layer"),
        # The second torque route (kernel derivatives: three fields instead of six), a quarter layer.
        _case("rollers_256k_derivative", "apply", "bottom_wall", "mixed", "kernel_derivative", 262144, 1536, 65,
              L=1024.0, fill="layer"),
        # An open box through host arrays, as a served request comes: copies in and out, odd sizes.
        _case("free_9k_host", "host", "free", "mixed", "spectral_curl", 9001, 630, 65),
        # The largest force-only scaling system: 663,552 spheres in two layers, 2700^2 x 19.
        _case("forces_663k_mixed", "apply", "bottom_wall", "mixed", "none", 663552, 2700, 19, L=18 * 128.8, m=4,
              beta=4 * 1.87, fill="lattice", H=9.1),
        # Brownian increments of such a layer: Lanczos iterations on the product, to three digits.
        _case("brownian_32k_mixed", "lanczos", "bottom_wall", "mixed", "none", 32768, 600, 19, L=4 * 128.8, m=4,
              beta=4 * 1.87, fill="lattice", H=7.5),
        # Independent systems of uneven size in one call (N log-uniform in [100, 50000]).
        dict(name="batch_12_mixed", call="batch", count=12, sizes=4),
        # The stochastic drift of a small suspension in double precision: two products, ragged box.
        _case("drift_1k_fp64", "drift", "bottom_wall", "fp64", "spectral_curl", 1001, 210, 33),
    ]


def _case(name, call, mode, precision, route, n, nx, nz, L=None, m=5, beta=None, fill="uniform", H=None, ny=None):
    c = dict(call=call, mode=mode, precision=precision, route=route, n=n, nx=nx, ny=ny or nx, nz=nz,
             L=float(L) if L else 4.0 * math.sqrt(n), m=m, beta=float(beta) if beta else BETA5[0], fill=fill,
             H=float(H) if H else (LAYER_H if fill == "layer" else DOMAINS[mode][0]))
    if name:
        c = dict(name=name, **c)
    return c


_SMOOTH = workloads.smooth7_sizes(4096)


def _smooth(x):
    return min(_SMOOTH, key=lambda s: abs(s - x))


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("small", "curl", "layer", "forces", "fp64", "host", "derivative", "batch", "lanczos"))
    mode = ("bottom_wall", "slit", "free")[rng.randrange(3)]
    nz = rng.choice((33, 48, 49, 65, 81, 97))
    if kind == "batch":
        c, most = dict(call="batch", count=rng.randint(4, 14), sizes=rng.randrange(1 << 20)), work(listed()[5])["bytes"]
        while c["count"] > 1 and sum(work(s)["bytes"] for s in _systems(c)) > 0.8 * most:
            c["count"] -= 1
        return c
    if kind in ("layer", "derivative"):
        n = _logu(rng, 4000, 600000)
        nx = _smooth(1.5 * math.sqrt(4 * n))
        route = "kernel_derivative" if kind == "derivative" else "spectral_curl"
        return _case("", "apply", "bottom_wall", "mixed", route, n, nx, 65, L=nx / 1.5, fill="layer")
    if kind in ("forces", "lanczos"):
        n = _logu(rng, 2000, 500000 if kind == "forces" else 40000)
        L = 2.846 * math.sqrt(n)
        call, wall = ("apply", "bottom_wall") if kind == "forces" else ("lanczos", rng.choice(("bottom_wall", "slit")))
        return _case("", call, wall, "mixed", "none", n, _smooth(L * 150 / 128.8), 19, L=L, m=4, beta=4 * 1.87,
                     fill="lattice", H=7.5)
    n = {"small": _logu(rng, 100, 2500), "fp64": _logu(rng, 100, 7000)}.get(kind) or _logu(rng, 2500, 50000)
    L = 4.0 * math.sqrt(n)
    nx = _smooth(L / 0.6)
    ny = nx
    if kind in ("small", "fp64") and rng.random() < 0.4:      # boxes need not be square
        ny = _smooth(nx * rng.uniform(0.5, 0.9))
    call = "host" if kind == "host" else "apply"
    if kind == "fp64" and rng.random() < 0.3:
        call = "drift"
    route = rng.choice(("spectral_curl", "spectral_curl", "kernel_derivative", "none")) if kind != "curl" else "spectral_curl"
    return _case("", call, mode, "fp64" if kind == "fp64" else "mixed", route, n, nx, nz, L=L, ny=ny)


# ---- what a program has in hand before the call -----------------------------------------------
def _params(c):
    torque = c["route"] != "none"
    return dict(Lx=c["L"], Ly=c["L"] * c["ny"] / c["nx"], zmin=0.0, zmax=c["H"], mode=c["mode"], nx=c["nx"],
                ny=c["ny"], nz=c["nz"], m_M=c["m"], beta_M=c["beta"], m_D=c["m"] if torque else 0,
                beta_D=BETA5[1] if torque else 0.0, eta=1.0)


def _particles(c, seed):
    """(positions, forces, torques or None) as numpy float64 [n][3]."""
    rng = np.random.default_rng(seed)
    n, Lx, Ly = c["n"], c["L"], c["L"] * c["ny"] / c["nx"]
    pos = np.empty((n, 3))
    F = rng.standard_normal((n, 3))
    T = rng.standard_normal((n, 3)) if c["route"] != "none" else None
    if c["fill"] == "lattice":   # spheres that do not overlap: a jittered lattice with vacancies, two layers
        s = math.ceil(math.sqrt(1.03 * n))
        at = rng.permutation(s * s)[:n]
        a = Lx / s
        jit = rng.uniform(-0.12, 0.12, (n, 2))
        pos[:, 0] = (at % s + 0.5 + jit[:, 0]) * a
        pos[:, 1] = (at // s + 0.5 + jit[:, 1]) * a
        low = rng.random(n) < 0.5
        pos[:, 2] = np.clip(np.where(low, rng.normal(1.1, 0.05, n), rng.normal(2.2, 0.1, n)), 1.0, 3.0)
        return pos, F, T
    pos[:, 0] = rng.uniform(0.0, Lx, n)
    pos[:, 1] = rng.uniform(0.0, Ly, n)
    if c["fill"] == "layer":     # gravity and a rotating field's torque, with their small spread
        pos[:, 2] = np.maximum(np.abs(rng.normal(1.6, 0.3, n)), 1.05)
        F = 0.05 * F + np.array([0.0, 0.0, -1.0])
        T = None if T is None else 0.05 * T + np.array([0.0, 1.0, 0.0])
    else:
        _, lo, hi = DOMAINS[c["mode"]]
        pos[:, 2] = rng.uniform(lo, hi, n)
    return pos, F, T


def _systems(c):
    """The systems of a batch: sizes from the case, N log-uniform in [100, 50000], nz in {33, 65, 97}."""
    rng = np.random.default_rng(workloads.SEED_BASE + c["sizes"])
    out = []
    for i in range(c["count"]):
        n = int(round(math.exp(rng.uniform(math.log(100), math.log(50000)))))
        out.append(_case("", "apply", ("bottom_wall", "slit")[i % 2], "mixed", "spectral_curl", n,
                         _smooth(4.0 * math.sqrt(n) / 0.6), int(rng.choice((33, 65, 97)))))
    return out


def _dev(a):
    return None if a is None else torch.from_numpy(a).cuda()


def _pinned(a):
    if a is None:
        return None, None
    t = torch.from_numpy(a).pin_memory()
    return t, t.numpy()


def _plan(c):
    return binding.Plan.from_params(_params(c), c["route"], c["precision"], c["n"])


def prepare(case, seed):
    c = case
    if c["call"] == "batch":
        items = []
        for i, s in enumerate(_systems(c)):
            pos, F, T = (_dev(a) for a in _particles(s, seed * 1000 + i))
            items.append((_plan(s), pos, F, T, torch.empty_like(pos), torch.empty_like(pos)))
        return dict(call="batch", items=items, mixed=True)
    pos, F, T = _particles(c, seed)
    st = dict(call=c["call"], plan=_plan(c), mixed=c["precision"] == "mixed")
    if c["call"] == "host":
        st["keep"], st["args"] = zip(*(_pinned(a) for a in (pos, F, T)))
        keep, st["out"] = zip(*(_pinned(np.zeros((c["n"], 3))) if k == 0 or T is not None else (None, None)
                                for k in range(2)))
        st["keep"] += keep
        return st
    st["args"] = (_dev(pos), _dev(F), _dev(T))
    if c["call"] == "lanczos":
        st["lanczos"] = binding.Lanczos(st["plan"], max_iter=32)
    if c["call"] == "drift":
        st["delta"] = 0.1 * c["L"] / c["nx"]
    return st


# ---- one pass -----------------------------------------------------------------------------------
def _hand_on(state, *outs):
    return [o.float() if state["mixed"] else o for o in outs if o is not None]


def run(state):
    call = state["call"]
    if call == "batch":
        binding.apply_batch(state["items"])
        return [_hand_on(state, U, W) for _, _, _, _, U, W in state["items"]]
    plan = state["plan"]
    if call == "host":
        U, W = plan.apply_host(*state["args"], *state["out"])
        return [o.astype(np.float32) if state["mixed"] else o for o in (U, W) if o is not None]
    pos, F, T = state["args"]
    if call == "lanczos":
        g, iterations, _ = state["lanczos"].sample(pos, F.reshape(-1), tol=1e-3)
        return dict(g=_hand_on(state, g)[0], iterations=iterations)
    if call == "drift":
        return binding.rfd_drift(plan, pos, F, state["delta"])
    return _hand_on(state, *plan.apply(pos, F, T))


# ---- what a pass cannot do without --------------------------------------------------------------
def _nodes(c):
    s = np.cos(np.pi * np.arange(c["nz"]) / (c["nz"] - 1))
    return 0.5 * c["H"] * (1.0 + s)


def _occupied(c):
    """Node planes that some envelope reaches."""
    a = 0.5 * c["m"] * c["L"] / c["nx"]
    lo, hi = {"layer": (1.05, 2.9), "lattice": (1.0, 2.6)}.get(c["fill"], DOMAINS[c["mode"]][1:])
    z = _nodes(c)
    return int(np.count_nonzero((z >= lo - a) & (z <= hi + a)))


def work(case):
    """Particle arrays in and out; the grids cross memory only where they do not fit the cache: then
    each field leaves its x transform, passes the y transform (read and write) and enters the z
    stage, and the same back.  Operations: transforms of 2.5 n log2 n, 64 per wavenumber and node
    for the boundary-value problems, a multiply-add per field and support node of the transfer."""
    c = case
    if c["call"] == "batch":
        w = [work(s) for s in _systems(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    word = 8 if c["precision"] == "fp64" else 4
    torque = c["route"] != "none"
    fields = 6 if c["route"] == "spectral_curl" else 3
    planes, nxy, K = _occupied(c), c["nx"] * c["ny"], (c["nx"] // 2 + 1) * c["ny"]
    grid = fields * planes * nxy * word
    a = 0.5 * c["m"] * c["L"] / c["nx"]
    support = c["m"] ** 2 * planes * min(1.0, 2 * a / (c["H"] * planes / c["nz"]))
    flops = (2 * fields * planes * 2.5 * nxy * math.log2(nxy) + 2 * fields * 2 * K * 2.5 * c["nz"] * math.log2(c["nz"])
             + 64.0 * K * c["nz"] + 2 * 2 * fields * support * c["n"])
    bytes_ = c["n"] * 8 * (18 if torque else 9) + (8 * grid if grid > CACHE_BYTES else 0)
    products = {"lanczos": 9, "drift": 2}.get(c["call"], 1)
    return {"bytes": float(products * bytes_), "flops": float(products * flops)}


# ---- the same in 64 bits, from the equations, in plain torch --------------------------------------
def _es(t, alpha, beta):
    x, w = np.polynomial.legendre.leggauss(128)
    th = 0.5 * np.pi * x
    Z = alpha * 0.5 * np.pi * float(np.dot(w, np.exp(beta * (np.cos(th) - 1.0)) * np.cos(th)))
    r = t / alpha
    inside = r.abs() <= 1.0
    s = torch.sqrt(torch.where(inside, 1.0 - r * r, torch.zeros_like(r)))
    return torch.where(inside, torch.exp(beta * (s - 1.0)) / Z, torch.zeros_like(r))


def _es_prime(t, alpha, beta):
    lo, hi = 2.0 / 3.0, 1.0      # |phi'| is smallest where beta v sqrt(1 - v) = 1, v > 2/3: cut there
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if beta * mid * math.sqrt(1.0 - mid) > 1.0 else (lo, mid)
    cut = alpha * math.sqrt(0.5 * (lo + hi))
    inside = t.abs() <= cut
    r = torch.where(inside, t / alpha, torch.zeros_like(t))
    return torch.where(inside, -beta * r / (alpha * torch.sqrt(1.0 - r * r)) * _es(t, alpha, beta), torch.zeros_like(t))


class _Exact:
    """The product [U; Omega] = M [F; T] of one case in 64 bits."""

    def __init__(self, c):
        self.c = c
        N, H = c["nz"], c["H"]
        n1, i = N - 1, np.arange(N)
        C = np.cos(np.pi * np.outer(i, i) / n1) * (2.0 / n1)
        C[:, [0, -1]] *= 0.5
        C[[0, -1], :] *= 0.5
        B = np.zeros((N + 2, N + 2))             # antiderivative of a Chebyshev series
        for n in range(1, N + 2):
            B[n, n - 1] = (2.0 if n == 1 else 1.0) / (2.0 * n)
            if n + 1 < N + 2:
                B[n, n + 1] = -1.0 / (2.0 * n)
        D = np.zeros((N, N))                     # derivative
        for n in range(N):
            D[[m for m in range(n) if (n - m) % 2], n] = 2.0 * n
        D[0] *= 0.5
        Y = np.zeros((N, N + 2))                 # y = trunc(B B c) + a0 + a1 T1
        Y[:, :N] = (B[:, :N + 1] @ B[:N + 1, :N])[:N]
        Y[0, N] = Y[1, N + 1] = 1.0
        integ = np.where(i % 2 == 0, 2.0 / (1.0 - np.where(i % 2 == 0, i, 0).astype(float) ** 2), 0.0)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        self.C, self.IC, self.D, self.Y = t(C), t(np.cos(np.pi * np.outer(i, i) / n1)), t(2.0 / H * D), t(Y)
        self.z, self.wz = t(_nodes(c)), t(0.5 * H * (C.T @ integ))
        self.top, self.bot = t(np.ones(N)), t((-1.0) ** i)
        self.dtop, self.dbot = t(2.0 / H * i.astype(float) ** 2), t(-2.0 / H * (-1.0) ** i * i.astype(float) ** 2)
        self.h = c["L"] / c["nx"]
        self.Ly = c["L"] * c["ny"] / c["nx"]
        self.sides = {"free": (), "bottom_wall": (0.0,), "slit": (0.0, H)}[c["mode"]]

    # particles <-> grid
    def _axis(self, x, L, n, alpha, beta, prime):
        first = torch.floor((x - alpha) / self.h).long()
        at = first[:, None] + torch.arange(self.c["m"] + 2, device=x.device)
        t = at.double() * self.h - x[:, None]
        return at % n, _es(t, alpha, beta), _es_prime(t, alpha, beta) if prime else None

    def _factors(self, pos, beta, prime):
        c, a = self.c, 0.5 * self.c["m"] * self.h
        ix, fx, dx = self._axis(pos[:, 0] % c["L"], c["L"], c["nx"], a, beta, prime)
        iy, fy, dy = self._axis(pos[:, 1] % self.Ly, self.Ly, c["ny"], a, beta, prime)
        t = self.z - pos[:, 2:3]
        fz, dz = _es(t, a, beta), _es_prime(t, a, beta) if prime else None
        for w in self.sides:
            t = self.z - (2.0 * w - pos[:, 2:3])
            fz = fz - _es(t, a, beta)
            dz = dz - _es_prime(t, a, beta) if prime else None
        at = (iy[:, :, None] * c["nx"] + ix[:, None, :]).reshape(len(pos), 1, -1)
        at = at + (torch.arange(c["nz"], device=pos.device) * (c["nx"] * c["ny"]))[:, None]
        prod = lambda z, y, x: z[:, :, None] * (y[:, :, None] * x[:, None, :]).reshape(len(pos), 1, -1)  # noqa: E731
        env = prod(fz, fy, fx)
        return at, env, (prod(fz, fy, dx), prod(fz, dy, fx), prod(dz, fy, fx)) if prime else None

    def _chunks(self, n):
        s = max(64, int(3e7 // (self.c["nz"] * (self.c["m"] + 2) ** 2)))
        return [slice(a, min(n, a + s)) for a in range(0, n, s)]

    def _spread(self, grid, pos, v, beta, prime):
        for s in self._chunks(len(pos)):
            at, env, grad = self._factors(pos[s], beta, prime)
            q = v[s]
            for f in range(3):
                if prime:
                    a, b = (f + 1) % 3, (f + 2) % 3
                    val = 0.5 * (grad[a] * q[:, b, None, None] - grad[b] * q[:, a, None, None])
                else:
                    val = env * q[:, f, None, None]
                grid[f].view(-1).index_add_(0, at.reshape(-1), val.reshape(-1))

    def _interpolate(self, grid, pos, beta, prime):
        out = torch.empty_like(pos)
        for s in self._chunks(len(pos)):
            at, env, grad = self._factors(pos[s], beta, prime)
            w = self.h * self.h * self.wz[:, None]
            u = [grid[f].view(-1)[at] * w for f in range(3)]
            for f in range(3):
                a, b = (f + 1) % 3, (f + 2) % 3
                val = 0.5 * (u[a] * grad[b] - u[b] * grad[a]) if prime else u[f] * env
                out[s, f] = val.sum(dim=(1, 2))
        return out

    # one block of wavenumbers: force coefficients [3][k][N] -> velocity coefficients
    def _bvp(self, k, r, gt, gb):
        """(D^2 - k^2) y = r with y' + k y = gt above and y' - k y = gb below; r [R][k][N] complex."""
        N = self.c["nz"]
        A = (-(k * k))[:, None, None] * self.Y
        A[:, :, :N] += (2.0 / self.c["H"]) ** 2 * torch.eye(N, dtype=A.dtype, device=A.device)
        rows = torch.stack([(self.dtop @ self.Y) + k[:, None] * (self.top @ self.Y),
                            (self.dbot @ self.Y) - k[:, None] * (self.bot @ self.Y)], dim=1)
        rhs = torch.cat([r, gt[:, :, None], gb[:, :, None]], dim=2).permute(1, 2, 0)
        R = rhs.shape[2]
        sol = torch.linalg.solve(torch.cat([A, rows], dim=1), torch.cat([rhs.real, rhs.imag], dim=2))
        y = torch.einsum("nm,kmr->rkn", self.Y, sol)
        return torch.complex(y[:R], y[R:])

    def _correct(self, k, kx, ky, v):
        """Node values of the homogeneous flow that cancels the velocity at the walls."""
        kc = k[:, None]
        bot = -(v * self.bot).sum(-1)
        z = self.z[None, :]
        Eb = torch.exp(-kc * z)
        if self.c["mode"] == "bottom_wall":
            u0, v0, w0 = (b[:, None] for b in bot)
            com = 1j * kc * w0 + kx[:, None] * u0 + ky[:, None] * v0
            return torch.stack([(u0 - kx[:, None] / kc * com * z) * Eb, (v0 - ky[:, None] / kc * com * z) * Eb,
                                (w0 + (kc * w0 - 1j * kx[:, None] * u0 - 1j * ky[:, None] * v0) * z) * Eb])
        H, E = self.c["H"], torch.exp(-k * self.c["H"])
        top = -(v * self.top).sum(-1)
        A = torch.zeros((len(k), 8, 8), dtype=torch.complex128, device=k.device)
        o = torch.ones_like(k)
        # unknowns C0, D0, then (C, D) of u, v, w; D multiplies e^{-k (H - z)}; eta = 1
        for f, q in enumerate((-1j * kx / (2 * k), -1j * ky / (2 * k), o / 2)):
            A[:, f, 2 + 2 * f], A[:, f, 3 + 2 * f] = o + 0j, E + 0j
            A[:, 3 + f, 0], A[:, 3 + f, 1] = q * H * E, (-q if f < 2 else q) * H
            A[:, 3 + f, 2 + 2 * f], A[:, 3 + f, 3 + 2 * f] = E + 0j, o + 0j
        for row, (p, q) in ((6, (o, E)), (7, (E, o))):
            for col, val in enumerate((0.5, 1j * kx, 1j * ky)):
                A[:, row, 2 * col], A[:, row, 2 * col + 1] = val * p, val * q
            A[:, row, 6], A[:, row, 7] = -k * p, k * q
        x = torch.linalg.solve(A, torch.cat([bot, top, torch.zeros_like(bot[:2])]).T[:, :, None])[:, :, 0]
        Et = torch.exp(-kc * (H - z))
        out = []
        for f, q in enumerate((-1j * kx / (2 * k), -1j * ky / (2 * k), o / 2)):
            q = q[:, None]
            out.append(x[:, 0:1] * q * z * Eb + x[:, 1:2] * (-q if f < 2 else q) * z * Et
                       + x[:, 2 + 2 * f, None] * Eb + x[:, 3 + 2 * f, None] * Et)
        return torch.stack(out)

    def _zero(self, f):
        """k = 0: u'' = -f with u = 0 at the walls, u' = 0 at an open top above a wall; no flow in an open box."""
        N, s = self.c["nz"], 2.0 / self.c["H"]
        if self.c["mode"] == "free":
            return torch.zeros_like(f)
        A = torch.zeros((N + 2, N + 2), dtype=torch.float64, device=f.device)
        A[:N, :N] = s * s * torch.eye(N, dtype=A.dtype, device=A.device)
        A[N] = (self.top if self.c["mode"] == "slit" else self.dtop) @ self.Y
        A[N + 1] = self.bot @ self.Y
        rhs = torch.zeros((N + 2, 2), dtype=f.dtype, device=f.device)
        rhs[:N] = -f[:2].T
        y = self.Y @ torch.linalg.solve(A, rhs.real)
        return torch.cat([y.T + 0j, torch.zeros_like(f[:1])])

    def product(self, pos, F, T):
        c, N, nx, ny = self.c, self.c["nz"], self.c["nx"], self.c["ny"]
        curl, prime = c["route"] == "spectral_curl", c["route"] == "kernel_derivative"
        grid = torch.zeros((6 if curl else 3, N, ny, nx), dtype=torch.float64, device=pos.device)
        self._spread(grid[:3], pos, F, c["beta"], False)
        if T is not None:
            self._spread(grid[3:] if curl else grid, pos, T, BETA5[1], prime)
        nk = nx // 2 + 1
        spec = torch.stack([torch.fft.rfft2(g) for g in grid]).view(len(grid), N, ny * nk)
        grid = None
        KX = (2 * math.pi / c["L"] * torch.arange(nk, dtype=torch.float64, device=pos.device)).repeat(ny)
        nyv = torch.fft.fftfreq(ny, 1.0 / ny, dtype=torch.float64, device=pos.device)
        KY = (2 * math.pi / self.Ly * nyv).repeat_interleave(nk)
        live = torch.ones((ny, nk), dtype=torch.bool, device=pos.device)
        if nx % 2 == 0:
            live[:, nx // 2] = False
        if ny % 2 == 0:
            live[ny // 2] = False
        live[0, 0] = False
        idx = live.view(-1).nonzero()[:, 0]
        out = torch.zeros_like(spec)

        def half_curl(a, ikx, iky):
            d = a @ self.D.T.to(a.dtype)
            return 0.5 * torch.stack([iky * a[2] - d[1], d[0] - ikx * a[2], ikx * a[1] - iky * a[0]])

        step = max(256, int(1.5e8 // (N * N * 8)) * 4)
        for s in [torch.zeros(1, dtype=torch.long, device=pos.device)] + list(idx.split(step)):
            a = torch.einsum("nc,fck->fkn", self.C + 0j, spec[:, :, s])
            kx, ky = KX[s], KY[s]
            ikx, iky = 1j * kx[:, None], 1j * ky[:, None]
            f = a[:3] + half_curl(a[3:], ikx, iky) if curl else a
            if int(s[0]) == 0:
                v = self._zero(f[:, 0])[:, None]
            else:
                k = torch.hypot(kx, ky)
                DT = self.D.T + 0j
                zero = torch.zeros_like(f[:1, :, 0])
                p = self._bvp(k, (ikx * f[0] + iky * f[1] + f[2] @ DT)[None], zero, zero)[0]
                pt, pb = (p * self.top).sum(-1), (p * self.bot).sum(-1)
                gt = torch.stack([-1j * kx / (2 * k) * pt, -1j * ky / (2 * k) * pt, pt / 2])
                gb = torch.stack([1j * kx / (2 * k) * pb, 1j * ky / (2 * k) * pb, pb / 2])
                v = self._bvp(k, torch.stack([ikx * p - f[0], iky * p - f[1], p @ DT - f[2]]), gt, gb)
                if self.sides:
                    v = v + self._correct(k, kx, ky, v) @ (self.C.T + 0j)
            o = torch.cat([v, half_curl(v, ikx, iky)]) if curl else v
            out[:, :, s] = torch.einsum("cn,fkn->fck", self.IC + 0j, o)
        spec = None
        grid = torch.stack([torch.fft.irfft2(g.view(N, ny, nk), s=(ny, nx)) for g in out])
        U = self._interpolate(grid[:3], pos, c["beta"], False)
        if T is None:
            return U, None
        return U, self._interpolate(grid[3:] if curl else grid, pos, BETA5[1], prime)

    def lanczos(self, pos, w, tol):
        """M^{1/2} w by the Lanczos process, to a relative change of `tol` between iterates."""
        norm, V, alpha, beta, y = float(w.norm()), [w / w.norm()], [], [], None
        while True:
            v = self.product(pos, V[-1].view(-1, 3), None)[0].reshape(-1)
            alpha.append(float(V[-1] @ v))
            for _ in range(2):
                for q in V:
                    v = v - (q @ v) * q
            lam, Q = np.linalg.eigh(np.diag(alpha) + np.diag(beta, 1) + np.diag(beta, -1))
            last, y = y, Q @ (np.sqrt(np.maximum(lam, 0.0)) * Q[0])
            if last is not None and np.linalg.norm(y - np.append(last, 0.0)) <= tol * np.linalg.norm(last):
                return norm * sum(float(a) * q for a, q in zip(y, V)), len(alpha)
            beta.append(float(v.norm()))
            V.append(v / v.norm())


def exact(case, seed):
    c = case
    if c["call"] == "batch":
        out = []
        for i, s in enumerate(_systems(c)):
            out.append(list(_Exact(s).product(*(_dev(a) for a in _particles(s, seed * 1000 + i)))))
        return out
    if c["nx"] * c["ny"] * c["nz"] > 2.2e8:   # the million-roller layer: over the time allowed
        return None
    pos, F, T = (_dev(a) for a in _particles(c, seed))
    e = _Exact(c)
    if c["call"] == "lanczos":
        g, iterations = e.lanczos(pos, F.reshape(-1), 1e-3)
        return dict(g=g, iterations=iterations)
    if c["call"] == "drift":
        d = 0.1 * c["L"] / c["nx"]
        T = torch.zeros_like(F) if T is not None else None
        P, M = e.product(pos + 0.5 * d * F, F, T), e.product(pos - 0.5 * d * F, F, T)
        return torch.cat([(p - m) / d for p, m in zip(P, M) if p is not None])
    return [o for o in e.product(pos, F, T) if o is not None]
