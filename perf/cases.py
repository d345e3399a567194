"""Cases by which the speed of the library is measured.

Each case is work that a program using the library has it do through its public entry points (``fg.Lattice``,
``fg.Batch`` and the C ABI that they wrap): HMC trajectories of one lattice in the precisions and link formats
that are run in earnest, trajectories of many chains at once, solves of the Wilson normal equations, a dynamical-fermion
trajectory and the action sums on caller-owned device arrays.  Sizes, couplings, step sizes and integrators are
those of the repository's benchmark, tests and workloads.

Inputs.  Links are independent SU(3) matrices spread around the unit matrix so far that the mean plaquette is near
the one of the coupling (0.6 at beta = 6), momenta are unit Gaussians and spinors complex Gaussians.  Trajectories
are always accepted (``u_accept = 0``) and go on from the momenta at the end of the last one, so that a state can be
passed again and every pass does the same work.

Outputs.  A trajectory gives what the call reports and the new links, as the program reads them for its next
measurement or for a stored configuration: FP64 for the FP64 and double-float fields, single precision on the GPU
for the FP32 ones.  H at both ends is among them and dH is not given a second time where the fields are FP32.
"""

import ctypes
import math
import random

import numpy as np
import torch

from paper_0910_2950_gb300 import fg

# Spread of the links: mean plaquette 0.60 (gauge runs), and rougher ones on which the hopping parameter of the
# repository's fermion workloads, 0.158, lies just below the critical one (a solve takes about 100 iterations, as on
# its thermalised fields).  The dynamical trajectory starts at the plaquette of its coupling instead.
SPREAD = 0.225
SPREAD_SOLVE = 0.40
SPREAD_NF2 = 0.235


def listed():
    return [
        # The smallest call: a 4^4 test chain in FP64, all latency and launches.
        {"name": "hmc fp64 4^4", "kind": "hmc", "precision": "fp64", "reals": 18, "lx": 4, "ly": 4, "lz": 4, "lt": 4,
         "beta": 6.0, "integrator": "fg", "steps": 8, "tau": 1.0},
        # A small pure-gauge chain as a trajectory server holds many of.
        {"name": "hmc fp32 8^4", "kind": "hmc", "precision": "fp32", "reals": 18, "lx": 8, "ly": 8, "lz": 8, "lt": 8,
         "beta": 5.9, "integrator": "fg", "steps": 8, "tau": 1.0},
        # An ordinary chain at the accuracy that dH needs.
        {"name": "hmc df64 16^4", "kind": "hmc", "precision": "df64", "reals": 18, "lx": 16, "ly": 16, "lz": 16,
         "lt": 16, "beta": 6.0, "integrator": "fg", "steps": 4, "tau": 1.0},
        # The same on unequal extents that fill no tile, with the other integrator in use.
        {"name": "hmc df64 ragged", "kind": "hmc", "precision": "df64", "reals": 18, "lx": 10, "ly": 14, "lz": 12,
         "lt": 26, "beta": 6.0, "integrator": "omelyan", "steps": 8, "tau": 1.0},
        # The headline: 32^4 in FP32 with the force-gradient integrator at the step that gives 75% acceptance.
        {"name": "hmc fp32 32^4", "kind": "hmc", "precision": "fp32", "reals": 18, "lx": 32, "ly": 32, "lz": 32,
         "lt": 32, "beta": 6.0, "integrator": "fg", "steps": 6, "tau": 1.0},
        # Compressed links, Omelyan's integrator, a lattice whose fields exceed the L2 cache.
        {"name": "hmc fp32 12 reals 24^4", "kind": "hmc", "precision": "fp32", "reals": 12, "lx": 24, "ly": 24,
         "lz": 24, "lt": 24, "beta": 6.0, "integrator": "omelyan", "steps": 16, "tau": 1.0},
        # Many small chains of mixed sizes at once: the accurate batch, and a smaller FP32 one.
        {"name": "batch df64 64 chains", "kind": "batch", "precision": "df64", "reals": 18, "chains": 64, "lmin": 4,
         "lmax": 12, "sizes": 4, "integrator": "fg", "steps": 4, "tau": 1.0},
        {"name": "batch fp32 24 chains", "kind": "batch", "precision": "fp32", "reals": 18, "chains": 24, "lmin": 4,
         "lmax": 10, "sizes": 7, "integrator": "omelyan", "steps": 8, "tau": 1.0},
        # One solve of Mhat^dagger Mhat x = b to the tolerance of an action evaluation: fields within the L2 cache,
        # and beyond it with the inner precision that the library chooses by size.
        {"name": "solve fp32 16^3x32", "kind": "solve", "precision": "fp32", "reals": 18, "lx": 16, "ly": 16, "lz": 16,
         "lt": 32, "kappa": 0.158},
        {"name": "solve auto 24^3x48", "kind": "solve", "precision": "fp32_autocg", "reals": 18, "lx": 24, "ly": 24,
         "lz": 24, "lt": 48, "kappa": 0.158},
        # A whole dynamical-fermion trajectory of a served chain: some 26 solves with the forces between them.
        {"name": "nf2 fp32 8^3x16", "kind": "nf2", "precision": "fp32", "reals": 18, "lx": 8, "ly": 8, "lz": 8,
         "lt": 16, "beta": 5.6, "kappa": 0.13, "integrator": "fg", "steps": 8, "tau": 1.0},
        # The measurement on arrays that the caller holds on the device.
        {"name": "action sums 32^4", "kind": "action", "lx": 32, "ly": 32, "lz": 32, "lt": 32, "beta": 6.0},
    ]


def _extents(rng, low, high, most):
    """Four even extents, each spread over the logarithm of its range, of at most `most` sites."""
    while True:
        e = [2 * round(0.5 * math.exp(rng.uniform(math.log(low), math.log(high)))) for _ in range(4)]
        if math.prod(e) <= most:
            return dict(zip(("lx", "ly", "lz", "lt"), e))


def draw(rng):
    kind = rng.choices(("hmc", "batch", "solve", "nf2", "action"), (8, 3, 4, 2, 1))[0]
    integrator = rng.choice(("fg", "fg", "omelyan", "leapfrog"))
    steps = {"fg": (4, 10), "omelyan": (12, 24), "leapfrog": (16, 28)}
    run = {"integrator": integrator, "steps": rng.randint(*steps[integrator]), "tau": rng.choice((0.5, 1.0, 1.0))}
    reals = rng.choice((18, 18, 12))
    if kind == "hmc":
        precision = rng.choice(("fp32", "fp32", "df64", "df64", "fp64"))
        most = {"fp32": 30 ** 4, "df64": 16 ** 4, "fp64": 10 ** 4}[precision]
        return {"kind": kind, "precision": precision, "reals": reals, **_extents(rng, 4, 40, most),
                "beta": round(rng.uniform(5.7, 6.2), 3), **run}
    if kind == "batch":
        precision = rng.choice(("fp32", "df64"))
        reals = 18 if precision == "df64" else reals  # double-float batches hold full links
        low = rng.choice((4, 6, 8))
        run["steps"] = min(run["steps"], 12)
        return {"kind": kind, "precision": precision, "reals": reals, "chains": rng.randint(4, 40), "lmin": low,
                "lmax": rng.choice((low, 8, 10)), "sizes": rng.randint(0, 999), **run}
    if kind == "solve":
        precision = rng.choice(("fp32", "fp32", "fp32_autocg", "fp32_fp16cg", "fp64"))
        return {"kind": kind, "precision": precision, "reals": reals,
                **_extents(rng, 6, 40, 8 ** 4 if precision == "fp64" else 22 ** 4),
                "kappa": round(rng.uniform(0.152, 0.158), 4)}
    if kind == "nf2":
        run["steps"] = min(run["steps"], {"fg": 6, "omelyan": 10}.get(integrator, 16))
        return {"kind": kind, "precision": "fp32", "reals": 18, **_extents(rng, 4, 16, 4096), "beta": 5.6,
                "kappa": round(rng.uniform(0.125, 0.132), 4), **run}
    return {"kind": kind, **_extents(rng, 6, 40, 30 ** 4), "beta": round(rng.uniform(5.7, 6.2), 3)}


# ---------------------------------------------------------------------------------------------------- inputs

def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _gaussian(shape, g):
    return torch.randn(shape, generator=g, dtype=torch.float64, device=_device())


def _links(volume, g, spread):
    """complex128[volume, 4, 3, 3]: the rows of 1 + i spread H, H Gaussian, made orthonormal."""
    z = torch.view_as_complex(_gaussian((volume, 4, 2, 3, 2), g)) * (1j * spread)
    z[..., 0, 0] += 1.0
    z[..., 1, 1] += 1.0
    a = z[..., 0, :] / torch.linalg.vector_norm(z[..., 0, :], dim=-1, keepdim=True)
    b = z[..., 1, :] - (a.conj() * z[..., 1, :]).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    c = torch.stack([(a[..., (k + 1) % 3] * b[..., (k + 2) % 3] - a[..., (k + 2) % 3] * b[..., (k + 1) % 3]).conj()
                     for k in range(3)], -1)
    return torch.stack([a, b, c], -2).contiguous()


def _spinor(volume, g):
    """complex128[volume / 2, 4, 3] on the even sites, density exp(-|chi|^2)."""
    return torch.view_as_complex(_gaussian((volume // 2, 4, 3, 2), g)) * math.sqrt(0.5)


def _chains(case):
    """Extents and couplings of a batch: hypercubes of mixed sizes, fixed by the case."""
    r = random.Random(case["sizes"])
    ext = [r.choice(range(case["lmin"], case["lmax"] + 1, 2)) for _ in range(case["chains"])]
    return [(n,) * 4 for n in ext], [round(r.uniform(5.7, 6.2), 4) for _ in ext]


def _lattice_inputs(case, seed, spread, spinor=False):
    g = _generator(seed)
    volume = math.prod(_dims(case))
    links = _links(volume, g, spread)
    momenta = _gaussian((volume, 4, 8), g)
    return links, momenta, _spinor(volume, g) if spinor else None


def _batch_inputs(case, seed):
    g = _generator(seed)
    out = []
    for dims in _chains(case)[0]:
        volume = math.prod(dims)
        out.append((_links(volume, g, SPREAD), _gaussian((volume, 4, 8), g)))
    return out


def _pinned(n):
    return torch.empty(n, dtype=torch.float64, pin_memory=True)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "hmc":
        links, momenta, _ = _lattice_inputs(case, seed, SPREAD)
        lat = fg.Lattice(_dims(case), beta=case["beta"], precision=case["precision"], link_reals=case["reals"])
        lat.set_gauge(links.cpu().numpy())
        lat.set_momenta(momenta.cpu().numpy())
        s.update(lat=lat, links=_pinned(links.numel() * 2))
    elif kind == "batch":
        dims, beta = _chains(case)
        b = fg.Batch(dims, beta, precision=case["precision"], link_reals=case["reals"])
        at = [0]
        for c, (links, momenta) in enumerate(_batch_inputs(case, seed)):
            b.set_gauge(c, links.cpu().numpy())
            b.set_momenta(c, momenta.cpu().numpy())
            at.append(at[-1] + links.numel() * 2)
        s.update(batch=b, links=_pinned(at[-1]), at=at)
    elif kind == "solve":
        links, _, b = _lattice_inputs(case, seed, SPREAD_SOLVE, spinor=True)
        lat = fg.Lattice(_dims(case), kappa=case["kappa"], precision=case["precision"], link_reals=case["reals"],
                         cg_tol=1e-12)
        lat.set_gauge(links.cpu().numpy())
        s.update(lat=lat, b=b.cpu().numpy())
    elif kind == "nf2":
        links, momenta, chi = _lattice_inputs(case, seed, SPREAD_NF2, spinor=True)
        lat = fg.Lattice(_dims(case), beta=case["beta"], kappa=case["kappa"], precision=case["precision"],
                         link_reals=case["reals"])
        lat.set_gauge(links.cpu().numpy())
        lat.set_momenta(momenta.cpu().numpy())
        lat.set_pseudofermion(chi.cpu().numpy())
        s.update(lat=lat, links=_pinned(links.numel() * 2))
    else:
        links, momenta, _ = _lattice_inputs(case, seed, SPREAD)
        s.update(lib=fg.load(), links=torch.view_as_real(links), momenta=momenta,
                 dims=(ctypes.c_int * 4)(*_dims(case)))
    return s


# ---------------------------------------------------------------------------------------------------- one pass

REPORTED = ("H0", "H1", "S_gauge0", "S_gauge1", "T0", "T1", "accepted", "n_force")


def _as_held(host, precision):
    """Links as the program goes on with them: FP32 fields in single precision on the GPU."""
    if precision in ("fp64", "df64"):
        return host
    return host.to("cuda", non_blocking=True).to(torch.float32)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "solve":
        return s["lat"].cg_solve(s["b"])[0]
    if kind == "action":
        out = torch.empty(2, dtype=torch.float64, device="cuda")
        status = s["lib"].fg_action_sums_noalloc(s["links"].data_ptr(), s["momenta"].data_ptr(), s["dims"],
                                                 case["beta"], out.data_ptr(),
                                                 torch.cuda.current_stream().cuda_stream or None)
        if status != fg.FG_OK:
            raise RuntimeError("fg_action_sums_noalloc: status %d" % status)
        return out
    dt = case["tau"] / case["steps"]
    if kind == "batch":
        b = s["batch"]
        res = b.trajectory(case["integrator"], dt, case["tau"], refresh=False, always_accept=True)
        # chain by chain into one pinned array, through the C call that Batch.get_gauge wraps
        base = s["links"].data_ptr()
        for c in range(b.n):
            at = ctypes.cast(base + 8 * s["at"][c], ctypes.POINTER(ctypes.c_double))
            status = b._lib.fg_batch_get_gauge(b._h, c, at)
            if status != fg.FG_OK:
                raise RuntimeError("fg_batch_get_gauge: status %d" % status)
        kept = np.float32 if case["precision"] == "fp32" else np.float64
        out = {k: np.array([r[k] for r in res], dtype=kept) for k in REPORTED[:6]}
        out["accepted"] = np.array([r["accepted"] for r in res])
        out["links"] = _as_held(s["links"], case["precision"])
        return out
    r = s["lat"].trajectory(case["integrator"], dt, case["tau"], refresh=False, u_accept=0.0)
    s["lat"].get_gauge(out=s["links"].numpy())
    out = {k: r[k] for k in REPORTED}
    if case["precision"] in ("fp64", "df64"):
        out["dH"] = r["dH"]
    if kind == "nf2":
        out["S_ferm0"], out["S_ferm1"] = r["S_ferm0"], r["S_ferm1"]
    out["links"] = _as_held(s["links"], case["precision"])
    return out


# ---------------------------------------------------------------------------------------------------- work

def _n_force(case):
    n = case["steps"]
    return {"fg": 3 * n + 1, "omelyan": 2 * n + 1, "leapfrog": n + 1}[case["integrator"]]


def _n_exp(case):
    n = case["steps"]
    return {"fg": 3 * n, "omelyan": 2 * n, "leapfrog": n}[case["integrator"]]


# Operations a site: a 3x3 complex product is 198; every plaquette once (three products), its force carried to the
# two links that do not start at its corner (276 each); an exponential and its product with a link 520 a link; the
# two action sums, two products and a trace for each plaquette.
FORCE = 6 * 3 * 198 + 12 * 276
EXP = 4 * 520
ACTION = 6 * (2 * 198 + 36)


def work(case):
    """Links, momenta and spinors in and out once, in the type the caller holds them in on the far side."""
    if case["kind"] == "batch":
        volume = sum(math.prod(d) for d in _chains(case)[0])
    else:
        volume = math.prod(_dims(case))
    if case["kind"] == "action":
        return {"bytes": volume * (576 + 256), "flops": volume * (ACTION + 64)}
    wide = 4 if case["precision"].startswith("fp32") else 8
    field = 4 * case["reals"] * wide
    if case["kind"] == "solve":
        # iterations of about 100 sweeps of the operator, four hops of half the sites each
        return {"bytes": volume * (field + 2 * 96), "flops": volume * 100 * 4 * 1320 / 2}
    flops = volume * (_n_force(case) * FORCE + _n_exp(case) * EXP + 2 * ACTION)
    read = volume * (2 * field + 2 * 32 * wide + 576)
    if case["kind"] == "nf2":
        flops += volume * (_n_force(case) + 1) * 60 * 4 * 1320 / 2
    return {"bytes": read, "flops": flops}


# ---------------------------------------------------------------------------------------------------- 64 bits

class Plain:
    """The trajectories and solves in complex128 with plain tensors: links (4, 3, 3, t, z, y, x), momenta
    (4, 8, t, z, y, x), spinors (4, 3, t, z, y, x); forces as derivatives of the actions."""

    S3 = 1.0 / math.sqrt(3.0)

    def __init__(self, dims, beta=6.0, kappa=0.0):
        self.dims, self.beta, self.kappa = dims, beta, kappa
        self.sites = tuple(reversed(dims))
        x = [torch.arange(n, device=_device()) for n in self.sites]
        self.even = (sum(torch.meshgrid(*x, indexing="ij")) % 2 == 0)
        g = torch.zeros(4, 4, 4, dtype=torch.complex128)
        for m, row in enumerate((((3, 1j), (2, 1j), (1, -1j), (0, -1j)), ((3, -1), (2, 1), (1, 1), (0, -1)),
                                 ((2, 1j), (3, -1j), (0, -1j), (1, 1j)), ((2, 1), (3, 1), (0, 1), (1, 1)))):
            for i, (j, v) in enumerate(row):
                g[m, i, j] = v
        one = torch.eye(4, dtype=torch.complex128)
        self.minus, self.plus = (one - g).to(_device()), (one + g).to(_device())
        self.g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=_device()).view(4, 1, 1, 1, 1, 1)
        self.phi = None

    def links(self, u):
        return u.view(self.sites + (4, 3, 3)).permute(4, 5, 6, 0, 1, 2, 3).contiguous()

    def links_out(self, u):
        return torch.view_as_real(u.permute(3, 4, 5, 6, 0, 1, 2).contiguous()).reshape(-1)

    def momenta(self, p):
        return p.view(self.sites + (4, 8)).permute(4, 5, 0, 1, 2, 3).contiguous()

    def spinor(self, v):
        full = torch.zeros(self.sites + (4, 3), dtype=torch.complex128, device=_device())
        full[self.even] = v
        return full.permute(4, 5, 0, 1, 2, 3).contiguous()

    def spinor_out(self, v):
        return v.permute(2, 3, 4, 5, 0, 1)[self.even]

    @staticmethod
    def mul(a, b):
        return (a.unsqueeze(2) * b.unsqueeze(0)).sum(1)

    @staticmethod
    def dag(a):
        return a.transpose(0, 1).conj()

    @staticmethod
    def shift(f, mu, step):
        return torch.roll(f, -step, -1 - mu)

    def plane(self, u, mu, nu):
        a = self.mul(u[mu], self.shift(u[nu], mu, 1))
        b = self.mul(u[nu], self.shift(u[mu], nu, 1))
        return (a * b.conj()).real.sum((0, 1))

    def gauge_action(self, u):
        return sum(self.beta * (1.0 - self.plane(u, mu, nu) / 3.0).sum() for mu in range(4) for nu in range(mu))

    def hop(self, u, v):
        out = torch.zeros_like(v)
        for mu in range(4):
            fwd, back = self.shift(v, mu, 1), (u[mu].conj().unsqueeze(0) * v.unsqueeze(2)).sum(1)
            fwd = (u[mu].unsqueeze(0) * fwd.unsqueeze(1)).sum(2)
            out = out + torch.einsum("st,tc...->sc...", self.minus[mu], fwd)
            out = out + torch.einsum("st,tc...->sc...", self.plus[mu], self.shift(back, mu, -1))
        return out

    def bounded(self, u):
        """Links with the antiperiodic boundary in t."""
        sign = torch.ones(self.sites, dtype=torch.float64, device=_device())
        sign[-1] = -1.0
        return torch.stack([u[0], u[1], u[2], u[3] * sign])

    def mhat(self, ub, v):
        return v - self.kappa ** 2 * self.hop(ub, self.hop(ub, v))

    def mhat_dag(self, ub, v):
        return self.g5 * self.mhat(ub, self.g5 * v)

    def solve(self, u, b, tol=1e-13):
        ub = self.bounded(u)
        x, r = torch.zeros_like(b), b.clone()
        p, rr = r.clone(), (r.conj() * r).real.sum()
        stop = tol * tol * rr
        for k in range(5000):
            ap = self.mhat_dag(ub, self.mhat(ub, p))
            alpha = rr / (p.conj() * ap).real.sum()
            x, r = x + alpha * p, r - alpha * ap
            new = (r.conj() * r).real.sum()
            if k % 8 == 7 and new <= stop:
                break
            p, rr = r + (new / rr) * p, new
        self.iterations = k + 1
        return x

    def ferm_action(self, u):
        return (self.phi.conj() * self.solve(u, self.phi)).real.sum()

    def force(self, u):
        u = u.detach().requires_grad_(True)
        for mu in range(4):
            for nu in range(mu):
                (-self.beta / 3.0 * self.plane(u, mu, nu).sum()).backward()
        if self.phi is not None:
            with torch.no_grad():
                x = self.solve(u, self.phi)
                y = self.mhat(self.bounded(u), x)
            (-2.0 * (y.conj() * self.mhat(self.bounded(u), x)).real.sum()).backward()
        g, u = u.grad, u.detach()
        f = torch.empty((4, 8) + self.sites, dtype=torch.float64, device=_device())
        for mu in range(4):
            w = self.mul(u[mu], self.dag(g[mu]))
            f[mu] = -0.5 * torch.stack([w[0, 1].imag + w[1, 0].imag, w[0, 1].real - w[1, 0].real,
                                        w[0, 0].imag - w[1, 1].imag, w[0, 2].imag + w[2, 0].imag,
                                        w[0, 2].real - w[2, 0].real, w[1, 2].imag + w[2, 1].imag,
                                        w[1, 2].real - w[2, 1].real,
                                        (w[0, 0].imag + w[1, 1].imag - 2.0 * w[2, 2].imag) * self.S3])
        return f

    def moved(self, u, p, c):
        """exp(i c P) U: the series on a quarter of the exponent, squared twice."""
        out = torch.empty_like(u)
        for mu in range(4):
            q, z = p[mu] * (0.125 * c), torch.zeros_like(p[mu, 0])
            a = torch.stack([torch.stack([torch.complex(q[2] + self.S3 * q[7], z), torch.complex(q[0], -q[1]),
                                          torch.complex(q[3], -q[4])]),
                             torch.stack([torch.complex(q[0], q[1]), torch.complex(-q[2] + self.S3 * q[7], z),
                                          torch.complex(q[5], -q[6])]),
                             torch.stack([torch.complex(q[3], q[4]), torch.complex(q[5], q[6]),
                                          torch.complex(-2.0 * self.S3 * q[7], z)])]) * 1j
            one = torch.eye(3, dtype=torch.complex128, device=_device()).view(3, 3, 1, 1, 1, 1)
            e = one + a / 16.0
            for k in range(15, 0, -1):
                e = one + self.mul(a, e) / k
            e = self.mul(e, e)
            out[mu] = self.mul(self.mul(e, e), u[mu])
        return out

    def trajectory(self, u, p, integrator, steps, tau):
        dt, al = tau / steps, 0.1932
        seq = {"leapfrog": (("P", 0.5), ("Q", 1.0), ("P", 0.5)),
               "omelyan": (("P", al), ("Q", 0.5), ("P", 1.0 - 2.0 * al), ("Q", 0.5), ("P", al)),
               "fg": (("P", 1.0 / 6.0), ("Q", 0.5), ("G", 2.0 / 3.0), ("Q", 0.5), ("P", 1.0 / 6.0))}[integrator]
        s0, t0 = self.gauge_action(u), 0.5 * (p * p).sum()
        f0 = self.ferm_action(u) if self.phi is not None else 0.0
        ops = [list(o) for _ in range(steps) for o in seq]
        for i in range(len(ops) - 1, 0, -1):  # a kick after a kick is one kick
            if ops[i][0] == ops[i - 1][0] == "P":
                ops[i - 1][1] += ops.pop(i)[1]
        for op, c in ops:
            if op == "Q":
                u = self.moved(u, p, c * dt)
            else:
                f = self.force(u)
                if op == "G":
                    f = self.force(self.moved(u, f, -dt * dt / 24.0))
                p = p - c * dt * f
        s1, t1 = self.gauge_action(u), 0.5 * (p * p).sum()
        out = {"S_gauge0": float(s0), "S_gauge1": float(s1), "T0": float(t0), "T1": float(t1)}
        f1 = self.ferm_action(u) if self.phi is not None else 0.0
        if self.phi is not None:
            out["S_ferm0"], out["S_ferm1"] = float(f0), float(f1)
        out["H0"], out["H1"] = float(s0 + t0 + f0), float(s1 + t1 + f1)
        out["dH"] = out["H1"] - out["H0"]
        out["links"] = self.links_out(u)
        return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        dims, beta = _chains(case)
        all_of = []
        for d, b, (links, momenta) in zip(dims, beta, _batch_inputs(case, seed)):
            m = Plain(d, b)
            all_of.append(m.trajectory(m.links(links), m.momenta(momenta), case["integrator"], case["steps"],
                                       case["tau"]))
        out = {k: np.array([r[k] for r in all_of]) for k in REPORTED[:6]}
        return {**out, "accepted": None, "links": torch.cat([r["links"] for r in all_of])}
    spread = {"solve": SPREAD_SOLVE, "nf2": SPREAD_NF2}.get(kind, SPREAD)
    links, momenta, chi = _lattice_inputs(case, seed, spread, spinor=kind in ("solve", "nf2"))
    m = Plain(_dims(case), case.get("beta", 6.0), case.get("kappa", 0.0))
    u = m.links(links)
    if kind == "solve":
        return m.spinor_out(m.solve(u, m.spinor(chi)))
    if kind == "action":
        return torch.stack([m.gauge_action(u), 0.5 * (momenta * momenta).sum()])
    if kind == "nf2":
        m.phi = m.mhat_dag(m.bounded(u), m.spinor(chi))
    out = m.trajectory(u, m.momenta(momenta), case["integrator"], case["steps"], case["tau"])
    if case["precision"] not in ("fp64", "df64"):
        del out["dH"]
    return {**out, "accepted": None, "n_force": None}
