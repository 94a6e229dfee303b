"""Performance cases: the work that users of this framework have it do, each one
pass through its public entry points.

Four kinds of pass:

``steps``        a running simulation (``Context``): a number of time steps
                 (``step``, or ``step_sums_async`` where every step's mass and
                 momentum are wanted), then the state into a device tensor; with
                 ``snapshot`` also the mode variances and the structure factor.
``ensemble``     many uneven replicas (``Batch``): the steps between two snapshots,
                 the mode variances of all replicas and every replica's density
                 structure factor added to its accumulator (one is read back).
``adjoint``      gradients through many steps (``adjoint.run``): forward, spectral
                 loss, backward to the initial populations and the parameters.
``observables``  one snapshot of a large state: mode variances, conserved totals
                 and the structure factor.

``exact`` restates the update in 64-bit torch operations (moment matrices, the
counter-based noise, FFTs) and shares nothing with the package.
"""
import math

import numpy as np
import torch

from paper_1012_3632_gb300 import D2Q9, D3Q19, MODE_VAR, Batch, Context
from paper_1012_3632_gb300.adjoint import density_spectrum_loss
from paper_1012_3632_gb300.adjoint import run as adjoint_run

DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "bf16": torch.bfloat16}

# Fluids: the ideal gas; the one-phase force-model fluid of the 256^3 workload;
# the Landau double well as total bulk free energy (capillary workload); the same
# in the modified-equilibrium model.
MODELS = {
    "ideal": dict(fe=None, kT=1e-5, omega=(1.2, 1.0, 1.0)),
    "calibration": dict(fe=None, kT=1e-4, omega=(1.0, 1.0, 1.0)),
    "force": dict(fe=dict(A=-0.01, B=0.1, rho_c=1.0, kappa=0.02), kT=1e-6, omega=(1.0, 1.0, 1.0)),
    "stripe": dict(fe=dict(A=-0.025, B=0.4, rho_c=0.75, kappa=0.08, total=True), kT=1e-7, omega=(1.0, 1.0, 1.0)),
    "swift": dict(fe=dict(A=-0.025, B=0.4, rho_c=0.75, kappa=0.08, total=True, model=1), kT=1e-7,
                  omega=(1.0, 1.0, 1.0)),
}


def _steps(name, lattice, x, y, z, precision, model, steps, sums=False, snapshot=False):
    c = dict(kind="steps", lattice=lattice, x=x, y=y, z=z, precision=precision, model=model, steps=steps, sums=sums,
             snapshot=snapshot)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest run: the FP64 calibration lattice, 100 steps and its observables, 1024 sites.
        _steps("d2q9_ideal_32_fp64", "D2Q9", 32, 32, 1, "fp64", "calibration", 100, snapshot=True),
        # A small 3-D ideal gas, a replica of the ensemble run alone.
        _steps("d3q19_ideal_32_fp32", "D3Q19", 32, 32, 32, "fp32", "ideal", 50),
        # The shear-wave / FDT run at 128^3.
        _steps("d3q19_ideal_128_fp32", "D3Q19", 128, 128, 128, "fp32", "ideal", 20),
        # The headline: 256^3 force-model fluid, every step's mass and momentum recorded.
        _steps("d3q19_force_256_fp32", "D3Q19", 256, 256, 256, "fp32", "force", 8, sums=True),
        # The same with BF16 storage.
        _steps("d3q19_force_256_bf16", "D3Q19", 256, 256, 256, "bf16", "force", 8),
        # A ragged odd lattice (no even row length), force model.
        _steps("d3q19_force_odd_fp32", "D3Q19", 129, 95, 67, "fp32", "force", 10),
        # FP64 reference run of the force model at the adjoint workload's size.
        _steps("d3q19_force_64_fp64", "D3Q19", 64, 64, 64, "fp64", "force", 4),
        # Capillary waves: the 1024 x 400 liquid stripe, force model with the total free energy.
        _steps("d2q9_stripe_1024x400_fp32", "D2Q9", 1024, 400, 1, "fp32", "stripe", 100),
        # The same stripe in the modified-equilibrium model (noise coloured in Fourier space).
        _steps("d2q9_swift_1024x400_fp32", "D2Q9", 1024, 400, 1, "fp32", "swift", 20),
        # 64 uneven ideal-gas replicas: one snapshot interval of the ensemble run.
        dict(name="ensemble_64", kind="ensemble", replicas=64, steps=20),
        # Gradients of the spectral loss through 40 steps of the 64^3 force-model fluid.
        dict(name="adjoint_64_fp32", kind="adjoint", x=64, y=64, z=64, precision="fp32", steps=40, every=20),
        # A snapshot of the 128^3 run: mode temperatures, conserved totals, S(k).
        dict(name="observables_128_fp32", kind="observables", x=128, y=128, z=128, precision="fp32"),
    ]


def _edge(rng, lo, hi, odd=0.3):
    """A length spread over the logarithm of [lo, hi]; odd with probability `odd`, else even."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    n += (n & 1) != (1 if rng.random() < odd else 0)
    return min(max(n, lo), hi)


def draw(rng):
    kind = rng.choice(["ideal", "ideal", "force", "force", "force", "fp64", "calibration", "stripe", "swift",
                       "ensemble", "adjoint", "observables"])
    if kind in ("ideal", "force"):
        dims = [_edge(rng, 16, 256) for _ in range(3)]
        steps = max(2, min(50, int(1.2e8 / (dims[0] * dims[1] * dims[2]))))
        return _steps(None, "D3Q19", *dims, rng.choice(["fp32", "fp32", "bf16"]), kind,
                      rng.randint(max(2, steps // 2), steps), sums=rng.random() < 0.4)
    if kind == "fp64":
        return _steps(None, "D3Q19", *[_edge(rng, 8, 64) for _ in range(3)], "fp64",
                      rng.choice(["ideal", "force"]), rng.randint(2, 5))
    if kind == "calibration":
        precision = rng.choice(["fp64", "fp32"])
        return _steps(None, "D2Q9", _edge(rng, 16, 128), _edge(rng, 16, 128), 1, precision, "calibration",
                      rng.randint(20, 100), snapshot=precision == "fp64")
    if kind == "stripe":
        return _steps(None, "D2Q9", _edge(rng, 128, 1024), _edge(rng, 96, 400), 1, rng.choice(["fp32", "fp32", "fp64"]),
                      "stripe", rng.randint(10, 60))
    if kind == "swift":
        return _steps(None, "D2Q9", rng.choice([128, 225, 256, 360, 512, 1024]), rng.choice([96, 135, 200, 243, 400]),
                      1, "fp32", "swift", rng.randint(5, 20))
    if kind == "ensemble":
        return dict(kind="ensemble", replicas=rng.randint(2, 64), steps=rng.randint(2, 20))
    if kind == "adjoint":
        every = rng.randint(3, 20)
        return dict(kind="adjoint", x=_edge(rng, 16, 64), y=_edge(rng, 16, 64), z=_edge(rng, 16, 64),
                    precision=rng.choice(["fp32", "fp32", "fp64"]), steps=rng.randint(4, 2 * every), every=every)
    return dict(kind="observables", x=_edge(rng, 16, 96, 0.0), y=_edge(rng, 16, 96, 0.0), z=_edge(rng, 16, 96, 0.0),
                precision=rng.choice(["fp32", "fp32", "fp64"]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _weights(Q):
    return [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4 if Q == 9 else [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _velocities(Q):
    if Q == 9:
        c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        return [(a, b, 0) for a, b in c]
    return [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
            (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
            (0, 1, -1), (0, -1, 1)]


def _initial(case, seed, device):
    """Deviations g = f - w (rho0 = 1), shape (Q, Z, Y, X), in the case's storage type."""
    X, Y, Z = case["x"], case["y"], case.get("z", 1)
    model = MODELS[case.get("model", "force" if case["kind"] == "adjoint" else "ideal")]
    Q = 9 if case.get("lattice") == "D2Q9" else 19
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    dtype = DTYPE[case["precision"]]
    w, c = _weights(Q), _velocities(Q)
    g = torch.empty((Q, Z, Y, X), dtype=dtype, device=device)
    drho, ux = 0.0, None
    if model["fe"] and model["fe"].get("total"):
        # a liquid stripe of thickness Y / 2 between two tanh interfaces, shifted by a few rows
        fe = model["fe"]
        gap = 2 * math.sqrt(-fe["A"] / fe["B"])
        width = math.sqrt(8 * fe["kappa"] / (fe["B"] / 4)) / gap
        shift = 4 * torch.rand((), generator=gen, device=device, dtype=torch.float64)
        y = torch.arange(Y, device=device, dtype=torch.float64) - shift
        p = torch.tanh(2 * (y - 0.25 * Y) / width) - torch.tanh(2 * (y - 0.75 * Y) / width)
        drho = (fe["rho_c"] - gap / 2 + gap / 2 * p - 1.0)[None, :, None].expand(Z, Y, X)
    elif model["fe"]:
        # rho = rho_c + U(-0.01, 0.01) per site
        drho = 0.02 * torch.rand((Z, Y, X), generator=gen, device=device, dtype=torch.float32) - 0.01
    elif Q == 19:
        # a shear wave u_x(z) on the thermal state
        z = torch.arange(Z, device=device, dtype=torch.float32)
        ux = (1e-3 * torch.sin(2 * math.pi * z / Z))[:, None, None]
    for i in range(Q):
        gi = w[i] * drho
        if not model["fe"]:
            # thermal state: independent populations of variance rho0 kT w_i / cs^2
            gi = math.sqrt(3 * model["kT"] * w[i]) * torch.randn((Z, Y, X), generator=gen, device=device,
                                                                 dtype=torch.float32)
            if ux is not None:
                gi = gi + w[i] * (3 * c[i][0] * ux + 4.5 * c[i][0] ** 2 * ux * ux - 1.5 * ux * ux)
        g[i] = gi.to(dtype)
    return g


def _replicas(case, seed):
    """Edges, shear rates and keys of the ensemble: one fixed draw of sizes, rates and keys from the seed."""
    n = case["replicas"]
    rng = np.random.default_rng(4)
    edges = [int(v) for v in rng.choice(np.asarray((32, 48, 64, 96, 128)), size=64)][:n]
    om = np.random.default_rng(seed).uniform(0.8, 1.6, n)
    return edges, om, [1000 * (seed % 1000003) + r for r in range(n)]


def _shown(edges):
    """The replica whose structure factor is read back: the first of the smallest size."""
    return edges.index(min(edges))


def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "ensemble":
        edges, om, keys = _replicas(case, seed)
        n = len(edges)
        b = Batch([(e, e, e) for e in edges], om, [1e-5] * n, keys, stream=stream)
        b.init(thermal=True)
        return dict(case=case, batch=b, shown=_shown(edges))
    g = _initial(case, seed, "cuda")
    if case["kind"] == "adjoint":
        m = MODELS["force"]
        theta = [*m["omega"], m["fe"]["kappa"], m["fe"]["A"], m["fe"]["B"]]
        cfg = dict(dims=(case["x"], case["y"], case["z"]), kT=m["kT"], seed=seed, precision=case["precision"],
                   nsteps=case["steps"], every=case["every"], nonideal=True, rho_c=m["fe"]["rho_c"])
        return dict(case=case, g0=g.reshape(19, -1).requires_grad_(True), cfg=cfg,
                    theta=torch.tensor(theta, dtype=DTYPE[case["precision"]], requires_grad=True))
    m = MODELS[case.get("model", "ideal")]
    lattice = D2Q9 if case.get("lattice") == "D2Q9" else D3Q19
    ctx = Context(lattice, (case["x"], case["y"], case.get("z", 1)), *m["omega"], kT=m["kT"], free_energy=m["fe"],
                  seed=seed, precision=case["precision"], stream=stream)
    ctx.set_state_device(g.data_ptr())
    s = dict(case=case, ctx=ctx)
    if case["kind"] == "steps":
        s["out"] = g.reshape(g.shape[0], -1)  # the user's state buffer, reused for what comes out
        if case["sums"]:
            s["sums"] = torch.empty((case["steps"], 4), dtype=torch.float64, pin_memory=True)
    else:
        torch.cuda.synchronize()  # g is read before it is freed
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "ensemble":
        b = s["batch"]
        b.step(case["steps"])
        var = b.mode_variance()
        S = None
        for r in range(case["replicas"]):
            got = b.structure_factor(r, 0, accumulate=True, fetch=r == s["shown"])
            S = got if r == s["shown"] else S
        return dict(var=var, S=S)
    if case["kind"] == "adjoint":
        g0, theta = s["g0"], s["theta"]
        g0.grad = theta.grad = None
        gN = adjoint_run(g0, theta, s["cfg"])
        density_spectrum_loss(gN, s["cfg"]["dims"]).backward()
        return dict(gN=gN.detach(), g0=g0.grad, theta=theta.grad)
    ctx = s["ctx"]
    if case["kind"] == "observables":
        return dict(var=ctx.moments(MODE_VAR), totals=ctx.conservation(),
                    S=ctx.structure_factor(0, accumulate=True))
    out = {}
    if case["sums"]:
        ctx.step_sums_async(case["steps"], s["sums"].numpy())
        out["sums"] = s["sums"]
    else:
        ctx.step(case["steps"])
    ctx.get_state_device(s["out"].data_ptr())
    out["g"] = s["out"]
    if case["snapshot"]:
        out["var"] = ctx.moments(MODE_VAR)
        out["S"] = ctx.structure_factor(0, accumulate=True)
    return out


def work(case):
    if case["kind"] == "ensemble":
        sites = sum(e ** 3 for e in _replicas(case, 0)[0])
        # steps, then the populations once more for the statistics and one S(k) each
        return {"bytes": sites * (case["steps"] * 152 + 76 + 8), "flops": sites * (case["steps"] * 420 + 300)}
    Q = 9 if case.get("lattice") == "D2Q9" else 19
    e = {"fp64": 8, "fp32": 4, "bf16": 2}[case["precision"]]
    V = case["x"] * case["y"] * case.get("z", 1)
    n = case.get("steps", 0)
    flops = 420 if Q == 19 else 170  # transforms, relaxation and Box-Muller of a site
    if case["kind"] == "observables":
        return {"bytes": V * (Q * e + 8), "flops": V * 300}
    if case["kind"] == "adjoint":
        # the steps, and per step back the adjoint state in and out and the state it is taken at
        return {"bytes": V * n * Q * e * (2 + 3), "flops": V * n * 1300}
    if case["model"] != "ideal" and case["model"] != "calibration":
        flops += 120
    extra = V * (Q * e + 8) if case["snapshot"] else 0
    return {"bytes": V * n * 2 * Q * e + V * 2 * Q * e + extra, "flops": V * n * flops}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _basis(Q):
    """(T, N): moment polynomials at the velocities and their weighted norms."""
    c = np.array(_velocities(Q), dtype=float)
    x, y, z = c.T
    c2 = (c * c).sum(1)
    if Q == 9:
        T = [1 + 0 * x, x, y, 3 * c2 - 2, x * x - y * y, x * y, (3 * c2 - 4) * x, (3 * c2 - 4) * y,
             9 * c2 ** 2 - 15 * c2 + 2]
    else:
        T = [1 + 0 * x, x, y, z, c2 - 1, 3 * x * x - c2, y * y - z * z, x * y, y * z, z * x, (c2 - 5 / 3) * x,
             (c2 - 5 / 3) * y, (c2 - 5 / 3) * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z,
             c2 ** 2 - 2 * c2 + 1 / 3, (c2 - 1.5) * (3 * x * x - c2), (c2 - 1.5) * (y * y - z * z)]
    T = np.array(T)
    return T, (T * T * np.array(_weights(Q))).sum(1)


def _philox(site, step, call_tag, replica, key):
    """Philox4x32-10 of (site, step, call_tag, replica) under a 64-bit key, as four int64 tensors."""
    low = 0xFFFFFFFF
    a, b = site & low, torch.full_like(site, step & low)
    c, d = torch.full_like(site, call_tag), torch.full_like(site, replica)
    k0, k1 = key & low, (key >> 32) & low
    m0, m1 = 0xD2511F53, 0xCD9E8D57
    for _ in range(10):
        p, q = a * m0, c * m1  # 64-bit products, kept modulo 2^64
        a, b, c, d = ((q >> 32) & low) ^ b ^ k0, q & low, ((p >> 32) & low) ^ d ^ k1, p & low
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return a, b, c, d


def _normals(shape, count, step, key, device, replica=0, tag=0):
    """`count` standard normals per site: normal k is number k % 4 of call k // 4."""
    V = shape[0] * shape[1] * shape[2]
    site = torch.arange(V, device=device, dtype=torch.int64)
    z = []
    for call in range((count + 3) // 4):
        r = _philox(site, step, call | tag << 8, replica, key)
        for a, b in ((r[0], r[1]), (r[2], r[3])):
            radius = torch.sqrt(-2 * torch.log((a.double() + 0.5) * 2.0 ** -32))
            angle = 2 * math.pi * ((b.double() + 0.5) * 2.0 ** -32)
            z += [(radius * torch.cos(angle)).reshape(shape), (radius * torch.sin(angle)).reshape(shape)]
    return z[:count]


def _shift(f, c):
    """f(r + c) on the periodic lattice (z, y, x)."""
    return torch.roll(f, (-c[2], -c[1], -c[0]), (-3, -2, -1))


class _Exact:
    """The update of one lattice in 64-bit torch operations; state g of shape (Q, Z, Y, X)."""

    def __init__(self, Q, omega, kT, fe, key, device, replica=0):
        self.Q, self.key, self.replica, self.kT, self.device = Q, key, replica, kT, device
        T, N = _basis(Q)
        self.T = torch.tensor(T, device=device)
        self.N = N
        self.w, self.c = _weights(Q), _velocities(Q)
        # populations of moments: f_i = w_i sum_a T_ai m_a / N_a
        self.inv = torch.tensor((T / N[:, None] * np.array(self.w)).T.copy(), device=device)
        self.fe = fe
        D = 2 if Q == 9 else 3
        self.cons = D + 1
        s, b, gh = omega
        n = D * (D + 1) // 2
        self.rates = [b] + [s] * (n - 1) + [gh] * (Q - D - 1 - n)

    def force(self, drho):
        fe, w, c = self.fe, self.w, self.c
        lap = 6 * sum(w[i] * (_shift(drho, c[i]) - drho) for i in range(1, self.Q))
        d = drho + (1.0 - fe["rho_c"])
        mu = fe["A"] * d + fe["B"] * d ** 3 - fe["kappa"] * lap
        F = []
        for k in range(3):
            pairs = [i for i in range(1, self.Q) if c[i][k]]
            gr = 3 * sum(w[i] * c[i][k] * _shift(mu, c[i]) for i in pairs) if pairs else 0 * mu
            f = -(1 + drho) * gr
            if fe.get("total") and pairs:
                f = f + sum(w[i] * c[i][k] * _shift(drho, c[i]) for i in pairs)
            F.append(f)
        return F

    def coloured(self, z, drho):
        """xi_e and xi_eps of the modified-equilibrium model around rho0 = 1."""
        fe = self.fe
        Y, X = drho.shape[1:]
        kx = 2 * math.pi * torch.arange(X, device=self.device, dtype=torch.float64) / X
        ky = (2 * math.pi * torch.arange(Y, device=self.device, dtype=torch.float64) / Y)[:, None]
        K2 = 6 * sum(self.w[i] * (1 - torch.cos(kx * self.c[i][0] + ky * self.c[i][1])) for i in range(9))
        d = 1.0 - fe["rho_c"]
        c2 = fe["A"] + 3 * fe["B"] * d * d + (0 if fe.get("total") else 1 / 3) + fe["kappa"] * K2
        oe, op = self.rates[0], self.rates[5]
        le, lp, se, sp = 2 * oe / (2 - oe), 2 * op / (2 - op), 1 - oe / 2, 1 - op / 2
        P = 6 * self.kT
        a = se * se * P * 4 * (2 - 3 * c2) * le
        cc = sp * sp * P * 16 * (1.25 - 0.75 * c2) * lp
        b = se * sp * P * 6 * (c2 - 1 / 3) * (le + lp)
        c11 = torch.sqrt(a)
        c21 = b / c11
        c22 = torch.sqrt(torch.clamp(cc - c21 * c21, min=0))
        E, H = torch.fft.fft2(z[0][0]), torch.fft.fft2(z[5][0])
        return torch.fft.ifft2(c11 * E).real[None], torch.fft.ifft2(c21 * E + c22 * H).real[None]

    def step(self, g, t):
        Q, k0 = self.Q, self.cons
        shape = tuple(g.shape[1:])
        m = (self.T @ g.reshape(Q, -1)).reshape(g.shape)
        drho = m[0]
        rho = 1 + drho
        swift = self.fe is not None and self.fe.get("model") == 1
        F = self.force(drho) if self.fe is not None and not swift else [0.0, 0.0, 0.0]
        u = [(m[1 + d] + 0.5 * F[d]) / rho for d in range(k0 - 1)] + [0.0] * (4 - k0)
        x, y, z = u
        if Q == 9:
            eq = [3 * rho * (x * x + y * y), rho * (x * x - y * y), rho * x * y]
            fm = [6 * (x * F[0] + y * F[1]), 2 * (x * F[0] - y * F[1]), x * F[1] + y * F[0]]
        else:
            uu, uF = x * x + y * y + z * z, x * F[0] + y * F[1] + z * F[2]
            eq = [rho * uu, rho * (3 * x * x - uu), rho * (y * y - z * z), rho * x * y, rho * y * z, rho * z * x]
            fm = [2 * uF, 2 * (3 * x * F[0] - uF), 2 * (y * F[1] - z * F[2]), x * F[1] + y * F[0],
                  y * F[2] + z * F[1], z * F[0] + x * F[2]]
        normals = _normals(shape, Q - k0, t, self.key, self.device, self.replica) if self.kT else None
        if swift:
            fe, w, c = self.fe, self.w, self.c
            d = drho + (1.0 - fe["rho_c"])
            lap = 6 * sum(w[i] * (_shift(drho, c[i]) - drho) for i in range(1, 9))
            gx = 3 * sum(w[i] * c[i][0] * _shift(drho, c[i]) for i in range(1, 9) if c[i][0])
            gy = 3 * sum(w[i] * c[i][1] * _shift(drho, c[i]) for i in range(1, 9) if c[i][1])
            psi = d * d * (fe["A"] / 2 + fe["B"] / 4 * d * d)
            pex = rho * (fe["A"] * d + fe["B"] * d ** 3) - psi - fe["kappa"] * rho * lap
            if fe.get("total"):
                pex = pex - rho / 3
            eq = [eq[0] + 6 * pex, eq[1] + fe["kappa"] * (gx * gx - gy * gy), eq[2] + fe["kappa"] * gx * gy]
            xe, xp = self.coloured(normals, drho)
        out = [drho] + [m[1 + d] + F[d] for d in range(k0 - 1)]
        for k in range(Q - k0):
            a, om = k0 + k, self.rates[k]
            e = eq[k] if k < len(eq) else (-6 * pex if swift and k == 5 else 0.0)
            v = m[a] - om * (m[a] - e)
            if self.fe is not None and not swift and k < len(fm):
                v = v + (1 - om / 2) * fm[k]
            if normals is not None:
                if swift and k in (0, 5):
                    v = v + torch.sqrt(rho) * (xe if k == 0 else xp)
                else:
                    amp = 3 * self.kT * (2 - om) * om * self.N[a]
                    v = v + (amp ** 0.5) * torch.sqrt(rho) * normals[k]
            out.append(v)
        g = (self.inv @ torch.stack(out).reshape(Q, -1)).reshape((Q,) + shape)
        return torch.stack([_shift(g[i], tuple(-v for v in self.c[i])) for i in range(Q)])


def _variances(T, g):
    m = (T @ g.reshape(g.shape[0], -1))
    return m.var(1, unbiased=False)


def _spectrum(drho):
    S = torch.fft.fftn(drho - drho.mean()).abs() ** 2 / drho.numel()
    S.view(-1)[0] = 0
    return S.reshape(-1)


def _exact_ensemble(case, seed, device):
    edges, om, keys = _replicas(case, seed)
    if sum(e ** 3 for e in edges) * case["steps"] > 1.2e9:
        return None
    var, S = [], None
    for r, e in enumerate(edges):
        x = _Exact(19, (float(om[r]), 1.0, 1.0), 1e-5, None, keys[r], device, replica=r)
        z = _normals((e, e, e), 19, 0, keys[r], device, r, tag=1)
        m = torch.stack([math.sqrt(3e-5 * x.N[a]) * z[a] for a in range(19)])
        g = (x.inv @ m.reshape(19, -1)).reshape(19, e, e, e)
        for t in range(case["steps"]):
            g = x.step(g, t)
        var.append(_variances(x.T, g))
        if r == _shown(edges):
            S = _spectrum(g.sum(0)).cpu().numpy()
    return dict(var=torch.stack(var).cpu().numpy(), S=S)


def _exact_adjoint(case, seed, device):
    from torch.utils.checkpoint import checkpoint

    dtype = DTYPE[case["precision"]]
    m = MODELS["force"]
    th = torch.tensor([*m["omega"], m["fe"]["kappa"], m["fe"]["A"], m["fe"]["B"]], dtype=dtype).double()
    th.requires_grad_(True)
    g0 = _initial(case, seed, device).double().requires_grad_(True)

    def one(g, theta, t):
        # the oracle's parameters as 0-d tensors on the device: gradients flow through them
        v = [p.to(device) for p in theta]
        fe = dict(m["fe"], kappa=v[3], A=v[4], B=v[5])
        return _Exact(19, (v[0], v[1], v[2]), m["kT"], fe, seed, device).step(g, t)

    g = g0
    for t in range(case["steps"]):
        g = checkpoint(one, g, th, t, use_reentrant=False)
    rho = g.sum(0)
    k = [2 * math.pi * torch.fft.fftfreq(n, device=device, dtype=torch.float64) for n in g.shape[1:]]
    k2 = k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2
    (torch.exp(-k2 / 0.5) * torch.fft.fftn(rho - rho.mean()).abs() ** 2).sum().backward()
    return dict(gN=g.detach().reshape(19, -1), g0=g0.grad.reshape(19, -1), theta=th.grad.cpu())


def exact(case, seed, device="cuda"):
    if case["kind"] == "ensemble":
        return _exact_ensemble(case, seed, device)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed, device)
    m = MODELS[case.get("model", "ideal")]
    Q = 9 if case.get("lattice") == "D2Q9" else 19
    x = _Exact(Q, m["omega"], m["kT"], m["fe"], seed, device)
    g = _initial(case, seed, device).double()
    V = g[0].numel()

    def totals():
        c = torch.tensor(x.c, dtype=torch.float64, device=device)
        return torch.cat([(V + g.sum()).reshape(1), c.T @ g.reshape(Q, -1).sum(1)])

    if case["kind"] == "observables":
        return dict(var=_variances(x.T, g).cpu().numpy(), totals=totals().cpu().numpy(),
                    S=_spectrum(g.sum(0)).cpu().numpy())
    sums = []
    for t in range(case["steps"]):
        if case["sums"]:
            sums.append(totals())
        g = x.step(g, t)
    out = dict(g=g.reshape(Q, -1))
    if case["sums"]:
        out["sums"] = torch.stack(sums).cpu()
    if case["snapshot"]:
        out["var"] = _variances(x.T, g).cpu().numpy()
        out["S"] = _spectrum(g.sum(0)).cpu().numpy()
    return out
