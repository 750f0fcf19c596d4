"""Measured workloads of the lattice-QCD library, through its public Python entry points.

Each case is one call (or one short sequence of calls) that a user of the library makes:
operators, solves, gauge generation and observables, from the smallest lattice, where
launches count, to the largest of the benchmark. Lattice sizes, kappas, tolerances and
storage precisions are those of the repository's benchmark, tests and README; inputs are
drawn on the GPU from the seed alone. `exact` restates the operators in plain complex128
torch and shares no code with the library.

A user's program keeps one context, and keeps resident gauge fields, sources and result
tensors between calls; `prepare` makes these, `run` is the call.
"""
import math

import torch

from paper_1112_5280_gb300 import lqcd

DEV = "cuda"
C128 = torch.complex128
GAMMAS = ["1", "g5", "gx", "gy", "gz", "gt", "g5gx", "g5gy", "g5gz", "g5gt"]
REAL_BYTES = {"f64": 8, "df64": 8, "f32": 4, "f16": 2, "bf16": 2}
HOP_FLOPS = 1320  # one even-odd hop per output site, the usual count of the Wilson term

_context = None


def context():
    global _context
    if _context is None:
        _context = lqcd.Context(0)
    return _context


# ---------------------------------------------------------------- the cases


def _case(name, op, dims, **options):
    lx, ly, lz, lt = dims
    c = {"op": op, "lx": lx, "ly": ly, "lz": lz, "lt": lt}
    if name:
        c["name"] = name
    c.update(options)
    return c


def listed():
    return [
        # one application of the Schur operator on the smallest lattice that is solved and
        # served in earnest: launches and call overhead are all there is
        _case("mhat_8x8_f32", "mhat", (8, 8, 8, 8), prec="f32", compress=12, kappa=0.15, mu=0.0, reps=1),
        # the benchmark's headline: ten independent field sets per launch, ten launches
        _case("dslash_batch_16x32_f32", "dslash_batch", (16, 16, 16, 32), prec="f32", compress=18, sets=10, reps=10),
        # the inner operator of the mixed solvers at the largest lattice: M^dag M, four times
        _case("mhat_32x64_f16", "mhat", (32, 32, 32, 64), prec="f16", compress=12, kappa=0.155, mu=0.0, reps=8),
        # the FP64-class twisted-mass operator (residuals, outer corrections, force fields)
        _case("mhat_tm_24x48_df64", "mhat", (24, 24, 24, 48), prec="df64", compress=18, kappa=0.15, mu=0.01, reps=4),
        # a configuration and a source taken from torch tensors, the full FP64 operator, and
        # the result back in a torch tensor; extents of no round number
        _case("load_apply_ragged_f64", "load", (22, 18, 14, 38), prec="f64", compress=18, kappa=0.14, mu=0.0),
        # one propagator column at the largest lattice, the recommended mixed-precision CG
        _case("solve_cg_32x64_f16", "solve", (32, 32, 32, 64), solver="cg", prec="f16", kappa=0.155, mu=0.0, eps=0.8),
        # the other solver, on a twisted-mass operator and a lattice that does not fill the GPU
        _case("solve_bicgstab_tm_16x32_f32", "solve", (16, 16, 16, 32), solver="bicgstab", prec="f32", kappa=0.15,
              mu=0.01, eps=0.5),
        # a whole point-source propagator: 12 right-hand sides on one configuration
        _case("propagator_24x48_f32", "propagator", (24, 24, 24, 48), prec="f32", kappa=0.14, mu=0.0, eps=0.5,
              sources=12),
        # many small systems of uneven size, each on its own configuration, in one call
        _case("solve_batch_mixed_f32", "solve_batch", (16, 16, 16, 32), systems=18, prec="f32", eps=0.5),
        # pure-gauge generation: heatbath sweeps, then the configuration to the host
        _case("heatbath_24x48", "heatbath", (24, 24, 24, 48), beta=6.0, sweeps=2),
        # a short N_f = 2 twisted-mass HMC trajectory from a stored configuration and fresh
        # momenta: force solves, gauge and fermion forces, link updates
        _case("hmc_16x32", "hmc", (16, 16, 16, 32), beta=5.6, kappa=0.14, mu=0.01, tau=0.2, nsteps=4, ngauge=4,
              prec="f16"),
        # the meson two-point functions of a propagator, all ten Dirac structures
        _case("meson_24x48", "meson", (24, 24, 24, 48), gammas=10),
    ]


def _draw_dims(rng, lo, hi):
    """Even extents with lo <= volume <= hi, the volume spread over its logarithm."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        base = (v / 2) ** 0.25
        l3 = [max(2, 2 * round(base * rng.uniform(0.7, 1.4) / 2)) for _ in range(3)]
        lt = max(2, 2 * round(v / (l3[0] * l3[1] * l3[2]) / 2))
        if lo <= l3[0] * l3[1] * l3[2] * lt <= hi and lt <= 8 * max(l3):
            return (*l3, lt)


def draw(rng):
    op = rng.choice(["mhat", "mhat", "dslash_batch", "load", "solve", "solve", "propagator", "solve_batch",
                     "heatbath", "hmc", "meson"])
    small, mid, large = 8 ** 4, 24 ** 3 * 48, 32 ** 3 * 64
    kappa = round(rng.uniform(0.12, 0.155), 4)
    mu = rng.choice([0.0, 0.0, round(rng.uniform(0.005, 0.05), 4)])
    if op == "mhat":
        prec = rng.choice(["f64", "df64", "f32", "f32", "f16", "f16", "bf16"])
        dims = _draw_dims(rng, small, mid if prec in ("f64", "df64") else large)
        return _case("", op, dims, prec=prec, compress=18 if prec == "df64" else rng.choice([12, 18]), kappa=kappa,
                     mu=mu, reps=rng.randint(1, 8))
    if op == "dslash_batch":
        dims = _draw_dims(rng, small, 16 ** 3 * 32)
        return _case("", op, dims, prec=rng.choice(["f32", "f32", "f16", "f64"]), compress=rng.choice([12, 18]),
                     sets=rng.randint(2, 16), reps=rng.randint(1, 10))
    if op == "load":
        return _case("", op, _draw_dims(rng, small, mid), prec=rng.choice(["f64", "f32", "f16"]),
                     compress=rng.choice([12, 18]), kappa=kappa, mu=mu)
    if op == "solve":
        solver = rng.choice(["cg", "cg", "bicgstab"])
        prec = rng.choice(["f16", "f32", "bf16"]) if solver == "cg" else "f32"
        return _case("", op, _draw_dims(rng, small, mid), solver=solver, prec=prec, kappa=kappa, mu=mu,
                     eps=rng.choice([0.5, 0.8]))
    if op == "propagator":
        return _case("", op, _draw_dims(rng, small, 16 ** 3 * 32), prec=rng.choice(["f32", "f16"]), kappa=kappa, mu=mu,
                     eps=0.5, sources=rng.choice([4, 12]))
    if op == "solve_batch":
        return _case("", op, _draw_dims(rng, 4 * small, 16 ** 3 * 32), systems=rng.randint(3, 24),
                     prec=rng.choice(["f32", "f16"]), eps=0.5)
    if op == "heatbath":
        return _case("", op, _draw_dims(rng, small, mid), beta=round(rng.uniform(5.0, 7.0), 2),
                     sweeps=rng.randint(1, 2))
    if op == "hmc":
        return _case("", op, _draw_dims(rng, small, 16 ** 3 * 32), beta=5.6, kappa=0.14, mu=mu, tau=0.1,
                     nsteps=rng.randint(1, 3), ngauge=rng.randint(2, 4), prec=rng.choice(["f16", "f32"]))
    return _case("", op, _draw_dims(rng, small, mid), gammas=rng.randint(1, 10))


def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


# ---------------------------------------------------------------- inputs


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _gaussian(shape, gen):
    return torch.randn(shape, dtype=C128, device=DEV, generator=gen) * math.sqrt(2.0)


def _links(dims, eps, gen):
    """SU(3) links around the identity: the rows of 1 + i eps H, H Gaussian Hermitian and
    traceless, made orthonormal, with determinant 1; [V, 4, 3, 3]."""
    a = _gaussian((_volume(dims), 4, 3, 3), gen)
    h = 0.5 * (a + a.mH)
    del a
    one = torch.eye(3, dtype=C128, device=DEV)
    h = h - (h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3)[..., None, None] * one
    m = one + 1j * eps * h
    del h
    r0 = m[..., 0, :] / torch.linalg.vector_norm(m[..., 0, :], dim=-1, keepdim=True)
    r1 = m[..., 1, :] - (r0.conj() * m[..., 1, :]).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], dim=-2).contiguous()


def _momenta(dims, gen):
    a = _gaussian((_volume(dims), 4, 3, 3), gen)
    h = 0.5 * (a + a.mH)
    tr = h.diagonal(dim1=-2, dim2=-1).sum(-1) / 3
    return 1j * (h - tr[..., None, None] * torch.eye(3, dtype=C128, device=DEV))


def _point_source(dims, site, spin, colour):
    b = torch.zeros((_volume(dims), 4, 3), dtype=C128, device=DEV)
    b[site, spin, colour] = 1.0
    return b


def _propagator_like(dims, gen):
    """Twelve solutions as they look in earnest: noise that falls off from a time slice."""
    lt = dims[3]
    t = torch.arange(_volume(dims), device=DEV) // (dims[0] * dims[1] * dims[2])
    fall = torch.exp(-0.4 * torch.minimum(t, lt - t).double())
    return [_gaussian((_volume(dims), 4, 3), gen) * fall[:, None, None] for _ in range(12)]


def _systems(case):
    """The lattices and kappas of a solve_batch case: the case's own extents, and smaller
    ones as the benchmark mixes them."""
    lx, ly, lz, lt = _dims(case)
    sizes = [(lx, ly, lz, lt)]
    for f in (0.75, 0.5):
        sizes.append(tuple(max(2, 2 * round(f * e / 2)) for e in (lx, ly, lz)) + (max(2, 2 * round(f * lt / 2)),))
    n = case["systems"]
    return [(sizes[(2 - i) % 3], 0.12 + 0.035 * ((7 * i) % n) / n) for i in range(n)]


def _options(case):
    solver = lqcd.BICGSTAB if case.get("solver") == "bicgstab" else lqcd.CG
    return lqcd.solve_opts(solver=solver, sloppy_prec=case["prec"], sloppy_compress=12, mu=case.get("mu", 0.0))


TOL = 1e-11  # of the solves: propagators and forces are compared to about ten digits


def _tensors(case, seed):
    """The case's inputs as torch tensors, from the seed alone."""
    dims, gen, op = _dims(case), _generator(seed), case["op"]
    shape = (_volume(dims), 4, 3)
    if op in ("mhat", "load"):
        return {"U": _links(dims, 0.5, gen), "src": _gaussian(shape, gen)}
    if op == "dslash_batch":
        return {"U": [_links(dims, 0.5, gen) for _ in range(case["sets"])],
                "src": [_gaussian(shape, gen) for _ in range(case["sets"])]}
    if op == "solve":
        return {"U": _links(dims, case["eps"], gen), "src": _gaussian(shape, gen)}
    if op == "propagator":
        site = int(seed) % _volume(dims)
        return {"U": _links(dims, case["eps"], gen),
                "src": [_point_source(dims, site, k // 3, k % 3) for k in range(case["sources"])]}
    if op == "solve_batch":
        systems = _systems(case)
        return {"U": [_links(d, case["eps"], gen) for d, _ in systems],
                "src": [_gaussian((_volume(d), 4, 3), gen) for d, _ in systems]}
    if op == "heatbath":
        return {"U": _links(dims, 0.35, gen)}
    if op == "hmc":
        # as rough as an equilibrium configuration at beta = 5.6 (plaquette about 0.53)
        return {"U": _links(dims, 0.41, gen), "P": _momenta(dims, gen), "eta": _gaussian(shape, gen)}
    return {"props": _propagator_like(dims, gen)}


def prepare(case, seed):
    ctx, dims, op = context(), _dims(case), case["op"]
    t = _tensors(case, seed)
    torch.cuda.synchronize()  # the library works on a stream of its own
    s = {"case": case, "dims": dims}
    v = _volume(dims)
    if op == "mhat":
        s["g"] = ctx.gauge(dims, t["U"], case["prec"], case["compress"])
        s["in"] = ctx.field(dims, case["prec"], lqcd.EVEN, t["src"])
        s["tmp"] = [ctx.field(dims, case["prec"], lqcd.EVEN) for _ in range(2)]
        s["out"] = torch.zeros((v, 4, 3), dtype=C128, device=DEV)
    elif op == "dslash_batch":
        s["g"] = [ctx.gauge(dims, u, case["prec"], case["compress"]) for u in t["U"]]
        s["in"] = [ctx.field(dims, case["prec"], lqcd.ODD, b) for b in t["src"]]
        s["res"] = [ctx.field(dims, case["prec"], lqcd.EVEN) for _ in t["src"]]
        s["batch"] = lqcd.DslashBatch(s["g"], s["in"], s["res"], lqcd.EVEN)
        s["out"] = [torch.zeros((v, 4, 3), dtype=C128, device=DEV) for _ in t["src"]]
    elif op == "load":
        s["U"], s["src"] = t["U"], t["src"]
        s["a"], s["b"] = ctx.field(dims, case["prec"]), ctx.field(dims, case["prec"])
        s["out"] = torch.zeros((v, 4, 3), dtype=C128, device=DEV)
    elif op == "solve":
        s["g"] = ctx.gauge(dims, t["U"])
        s["src"], s["x"] = ctx.field(dims, data=t["src"]), ctx.field(dims)
        s["opts"] = _options(case)
        s["out"] = torch.zeros((v, 4, 3), dtype=C128, device=DEV)
    elif op == "propagator":
        s["g"] = ctx.gauge(dims, t["U"])
        s["src"] = [ctx.field(dims, data=b) for b in t["src"]]
        s["x"] = [ctx.field(dims) for _ in t["src"]]
        s["opts"] = _options(case)
        s["out"] = [torch.zeros((v, 4, 3), dtype=C128, device=DEV) for _ in t["src"]]
    elif op == "solve_batch":
        systems = _systems(case)
        s["g"] = [ctx.gauge(d, u) for (d, _), u in zip(systems, t["U"])]
        s["src"] = [ctx.field(d, data=b) for (d, _), b in zip(systems, t["src"])]
        s["x"] = [ctx.field(d) for d, _ in systems]
        s["kappas"] = [k for _, k in systems]
        s["opts"] = _options(case)
        s["out"] = [torch.zeros((_volume(d), 4, 3), dtype=C128, device=DEV) for d, _ in systems]
    elif op == "heatbath":
        s["g"] = ctx.gauge(dims, t["U"])
        s["seed"], s["sweep"] = int(seed), 0
        s["out"] = torch.zeros((v, 4, 3, 3), dtype=C128, pin_memory=True).numpy()
    elif op == "hmc":
        s["U"], s["P"], s["mom"] = t["U"], t["P"].cpu().pin_memory().numpy(), ctx.mom(dims)
        eta, s["phi"] = ctx.field(dims, data=t["eta"]), ctx.field(dims)
        lqcd.apply_Mhat(ctx.gauge(dims, t["U"]), case["kappa"], eta, s["phi"], dagger=True, mu=case["mu"])
        s["params"] = lqcd.hmc_params(beta=case["beta"], kappa=case["kappa"], mu=case["mu"], tau=case["tau"],
                                      nsteps=case["nsteps"], ngauge=case["ngauge"], scheme=lqcd.TWO_MN, chrono=2,
                                      tol=TOL)
        s["opts"] = _options(case)
        s["out"] = torch.zeros((v, 4, 3, 3), dtype=C128, pin_memory=True).numpy()
    else:
        s["props"] = [ctx.field(dims, data=p) for p in t["props"]]
    ctx.sync()
    return s


# ---------------------------------------------------------------- one pass


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "mhat":
        cur = s["in"]
        for i in range(case["reps"]):
            nxt = s["tmp"][i % 2]
            lqcd.apply_Mhat(s["g"], case["kappa"], cur, nxt, dagger=i % 2 == 1, mu=case["mu"])
            cur = nxt
        return cur.download(s["out"])
    if op == "dslash_batch":
        for _ in range(case["reps"]):
            s["batch"].apply()
        return [f.download(o) for f, o in zip(s["res"], s["out"])]
    if op == "load":
        g = context().gauge(s["dims"], s["U"], case["prec"], case["compress"])
        s["a"].upload(s["src"])
        lqcd.apply_M(g, case["kappa"], s["a"], s["b"], mu=case["mu"])
        return s["b"].download(s["out"])
    if op == "solve":
        lqcd.solve_fields(s["g"], s["src"], case["kappa"], TOL, s["x"], s["opts"])
        return s["x"].download(s["out"])
    if op == "propagator":
        lqcd.solve_multi(s["g"], s["src"], case["kappa"], TOL, s["x"], s["opts"])
        return [x.download(o) for x, o in zip(s["x"], s["out"])]
    if op == "solve_batch":
        lqcd.solve_batch(s["g"], s["src"], s["kappas"], TOL, s["x"], s["opts"])
        return [x.download(o) for x, o in zip(s["x"], s["out"])]
    if op == "heatbath":  # each pass continues the Markov chain
        fails = s["g"].heatbath(case["beta"], case["sweeps"], seed=s["seed"], sweep0=s["sweep"])
        s["sweep"] += case["sweeps"]
        return {"fails": fails, "plaquette": s["g"].plaquette(), "links": s["g"].download(s["out"])}
    if op == "hmc":
        g = context().gauge(s["dims"], s["U"])
        s["mom"].upload(s["P"])
        info = lqcd.hmc_trajectory(g, s["params"], s["mom"], s["phi"], s["opts"])
        return {"H": info["H1"], "plaquette": info["plaquette"], "links": g.download(s["out"]),
                "momenta": s["mom"].download()}
    return lqcd.meson_correlator(s["props"], GAMMAS[: case["gammas"]])


# ---------------------------------------------------------------- necessary work

ITERATIONS = 40  # conjugate-gradient steps that these kappas and tolerance take, nominal


def _hop_bytes(vh, prec, reals):
    """One even-odd hop: eight links, one spinor in and one out per output site."""
    return vh * (8 * reals + 48) * REAL_BYTES[prec]


def work(case):
    dims, op = _dims(case), case["op"]
    v = _volume(dims)
    vh = v // 2
    spinor, links = v * 24 * 8, v * 4 * 18 * 8  # FP64, in the host layout
    if op == "mhat":
        n = 2 * case["reps"]
        return {"bytes": n * _hop_bytes(vh, case["prec"], case["compress"]) + spinor // 2,
                "flops": n * vh * HOP_FLOPS}
    if op == "dslash_batch":
        n = case["sets"] * case["reps"]
        return {"bytes": n * _hop_bytes(vh, case["prec"], case["compress"]) + case["sets"] * spinor // 2,
                "flops": n * vh * HOP_FLOPS}
    if op == "load":
        return {"bytes": links + 2 * spinor + 2 * _hop_bytes(vh, case["prec"], case["compress"]),
                "flops": v * HOP_FLOPS}
    if op in ("solve", "propagator", "solve_batch"):
        sizes = [d for d, _ in _systems(case)] if op == "solve_batch" else [dims] * case.get("sources", 1)
        sites = sum(_volume(d) for d in sizes)
        hops = 4 * ITERATIONS * sites // 2
        return {"bytes": 4 * ITERATIONS * _hop_bytes(sites // 2, case["prec"], 12) + 2 * sites * 24 * 8,
                "flops": hops * HOP_FLOPS}
    if op == "heatbath":  # six staples of two SU(3) products, one more product, three SU(2) rotations
        return {"bytes": (2 * case["sweeps"] + 1) * links, "flops": case["sweeps"] * 4 * v * (13 * 198 + 810)}
    if op == "hmc":
        solves = 2 * case["nsteps"] + 1
        kicks = 4 * case["nsteps"] * case["ngauge"]
        hops = solves * 4 * ITERATIONS // 2
        return {"bytes": hops * _hop_bytes(vh, case["prec"], 12) + kicks * 4 * links,
                "flops": hops * vh * HOP_FLOPS + kicks * 4 * v * 16 * 198}
    return {"bytes": 12 * spinor, "flops": v * 144 * 6 * 2}


# ---------------------------------------------------------------- the same in 64 bits

_I2, _Z2 = torch.eye(2, dtype=C128), torch.zeros((2, 2), dtype=C128)
_PAULI = [torch.tensor(m, dtype=C128) for m in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]


def _block(a, b, c, d):
    return torch.cat([torch.cat([a, b], 1), torch.cat([c, d], 1)], 0)


# chiral basis: gamma_k = [[0, -i sigma_k], [i sigma_k, 0]], gamma_t = [[0, 1], [1, 0]]
GAMMA = [_block(_Z2, -1j * p, 1j * p, _Z2) for p in _PAULI] + [_block(_Z2, _I2, _I2, _Z2)]
GAMMA5 = _block(_I2, _Z2, _Z2, -_I2)


class _Wilson:
    """M = A - kappa D with A = 1 + 2 i kappa mu g5, antiperiodic in t; fields are
    [Lt, Lz, Ly, Lx, 4, 3] and the links [Lt, Lz, Ly, Lx, 4, 3, 3]."""

    def __init__(self, dims, U, kappa=0.0, mu=0.0):
        lx, ly, lz, lt = dims
        self.shape = (lt, lz, ly, lx)
        u = U.reshape(*self.shape, 4, 3, 3)
        self.u = [u[..., k, :, :].contiguous() for k in range(4)]
        self.dev = U.device
        self.kappa, self.a = kappa, 2.0 * kappa * mu
        x = [torch.arange(n, device=self.dev) for n in self.shape]
        grid = x[0][:, None, None, None] + x[1][:, None, None] + x[2][:, None] + x[3]
        self.even = ((grid % 2) == 0)[..., None, None]
        self.g5 = torch.tensor([1, 1, -1, -1], dtype=torch.float64, device=self.dev)[:, None]
        self.one = torch.eye(4, dtype=C128, device=self.dev)
        self.gamma = [g.to(self.dev) for g in GAMMA]

    def field(self, psi):
        return psi.reshape(*self.shape, 4, 3)

    def hop(self, psi, dagger=False):
        """D psi (or D^dag psi)."""
        out = torch.zeros_like(psi)
        for k in range(4):
            dim = 3 - k
            forward, backward = self.one - self.gamma[k], self.one + self.gamma[k]
            if dagger:
                forward, backward = backward, forward
            w = torch.roll(psi, -1, dim)
            if k == 3:
                w[-1] = -w[-1]
            w = torch.einsum("...ij,...sj->...si", self.u[k], torch.matmul(forward, w))
            out += w
            w = torch.einsum("...ji,...sj->...si", self.u[k].conj(), torch.matmul(backward, psi))
            w = torch.roll(w, 1, dim)
            if k == 3:
                w[0] = -w[0]
            out += w
        return out

    def diag(self, psi, dagger=False, inverse=False):
        """A psi, A^dag psi or their inverses."""
        if self.a == 0.0:
            return psi
        a = -self.a if dagger else self.a
        if inverse:
            return (psi - 1j * a * self.g5 * psi) / (1.0 + a * a)
        return psi + 1j * a * self.g5 * psi

    def m(self, psi):
        return self.diag(psi) - self.kappa * self.hop(psi)

    def mhat(self, psi, dagger=False):
        """The Schur operator on a field that vanishes on the odd sites."""
        t = self.diag(self.hop(psi, dagger), dagger, inverse=True)
        return self.diag(psi, dagger) - self.kappa ** 2 * self.hop(t, dagger)

    def solve(self, b):
        """M x = b by conjugate gradients on the Schur operator's normal equations, begun again
        from the true residual until that is at rounding."""
        zero = torch.zeros_like(b)
        be, bo = torch.where(self.even, b, zero), torch.where(self.even, zero, b)
        bhat = be + self.kappa * self.hop(self.diag(bo, inverse=True))
        x, u = zero, bhat
        for _ in range(4):
            r = p = self.mhat(u, dagger=True)
            first = rr = float((r.conj() * r).real.sum())
            e = zero
            for _ in range(1000):
                q = self.mhat(p)
                alpha = rr / float((q.conj() * q).real.sum())
                e = e + alpha * p
                r = r - alpha * self.mhat(q, dagger=True)
                rr, last = float((r.conj() * r).real.sum()), rr
                if rr <= 1e-16 * first:
                    break
                p = r + (rr / last) * p
            x = x + e
            u = bhat - self.mhat(x)
            if float(torch.linalg.vector_norm(u)) <= 1e-14 * float(torch.linalg.vector_norm(bhat)):
                break
        xo = self.diag(bo + self.kappa * self.hop(x), inverse=True)
        return x + torch.where(self.even, zero, xo)


def _flat(psi):
    return psi.reshape(-1, 4, 3)


def _exact_meson(dims, props, n):
    """C(t) = sum_x -Tr[S^dag g5 G S G g5], S[(spin, colour), (source spin, source colour)]."""
    lt = dims[3]
    s = torch.stack(props, dim=-1).reshape(lt, -1, 4, 3, 4, 3)
    g5 = GAMMA5.to(s.device)
    g = [x.to(s.device) for x in GAMMA]
    structures = [torch.eye(4, dtype=C128, device=s.device), g5, *g, *[g5 @ x for x in g]]
    # spin content of conj(S) S summed over space and colours
    gram = torch.stack([torch.einsum("xaibj,xcidj->abcd", s[t].conj(), s[t]) for t in range(lt)])
    corr = []
    for gm in structures[:n]:
        left, right = g5 @ gm, gm @ g5
        corr.append(-torch.einsum("ac,db,tabcd->t", left, right, gram))
    return torch.stack(corr).cpu().numpy()


def exact(case, seed):
    op, dims = case["op"], _dims(case)
    if op in ("heatbath", "hmc"):
        return None
    t = _tensors(case, seed)
    if op == "meson":
        return _exact_meson(dims, t["props"], case["gammas"])
    if op == "mhat":
        w = _Wilson(dims, t["U"], case["kappa"], case["mu"])
        psi = w.field(t["src"])
        psi = torch.where(w.even, psi, torch.zeros_like(psi))
        for i in range(case["reps"]):
            psi = w.mhat(psi, dagger=i % 2 == 1)
        return _flat(torch.where(w.even, psi, torch.zeros_like(psi)))
    if op == "dslash_batch":
        out = []
        for u, b in zip(t["U"], t["src"]):
            w = _Wilson(dims, u)
            psi = w.hop(w.field(b))
            out.append(_flat(torch.where(w.even, psi, torch.zeros_like(psi))))
        return out
    if op == "load":
        w = _Wilson(dims, t["U"], case["kappa"], case["mu"])
        return _flat(w.m(w.field(t["src"])))
    if op == "solve":
        w = _Wilson(dims, t["U"], case["kappa"], case["mu"])
        return _flat(w.solve(w.field(t["src"])))
    if op == "propagator":  # the first two sources; the others are the same work again
        w = _Wilson(dims, t["U"], case["kappa"], case["mu"])
        return [_flat(w.solve(w.field(b))) if k < 2 else None for k, b in enumerate(t["src"])]
    out = []
    for k, ((d, kappa), u, b) in enumerate(zip(_systems(case), t["U"], t["src"])):
        w = _Wilson(d, u, kappa)
        out.append(_flat(w.solve(w.field(b))) if k < 6 else None)
    return out
