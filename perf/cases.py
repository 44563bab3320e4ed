"""The work that users of this package have it do, as measurable cases: heat-bath
chains on one lattice, batches of lattices (ensembles and finite-temperature
scans) and the measurement of stored configurations, through the public
entry points of ``paper_1104_5432_gb300.su2``.

A case is one call sequence of a user's program on one handle.  Programs that
run long chains tune the launch shape once per lattice and keep the choice in
the tuning cache (``SU2_AUTOTUNE_CACHE``), as the benchmark and the scan
runner do; short one-off calls use the handle as it comes (``tuned``).
"""
import math
import os
import tempfile

import numpy as np
import torch

from paper_1104_5432_gb300 import inputs, su2

# the tuning cache of this process: a handle of a shape tuned before takes its
# launch shape from it
if "SU2_AUTOTUNE_CACHE" not in os.environ:
    os.environ["SU2_AUTOTUNE_CACHE"] = os.path.join(tempfile.mkdtemp(prefix="su2_tune_"), "shapes")


def listed():
    return [
        # a one-off look at a small ragged lattice: latency and launches
        _chain("short 10^3x6 f32", 10, 6, "f32", 2.4, 5, tuned=False),
        # the paper's performance test (hot start, 100 sweeps, plaquette after
        # each) at its smallest size
        _chain("8^4 f32", 8, 8, "f32", 6.0, 100),
        # the small FP64 workload (20 sweeps: a last-bit difference grows with
        # every sweep, and the links of longer chains cannot be compared)
        _chain("8^4 f64", 8, 8, "f64", 2.3, 20),
        # the FP64 arm of the equal-accuracy comparison; a thermalising run
        # takes no plaquette
        _chain("16^4 f64", 16, 16, "f64", 2.5, 20, plaq="none"),
        # the medium workload in both precisions
        _chain("32^4 f32", 32, 32, "f32", 6.0, 100, plaq="device"),
        _chain("32^4 f64", 32, 32, "f64", 6.0, 10),
        # the headline workload in both precisions
        _chain("64^4 f32", 64, 64, "f32", 2.5, 40, plaq="device"),
        _chain("64^4 f64", 64, 64, "f64", 2.5, 4),
        # the largest workload: 16 GiB of links
        _chain("128^4 f32", 128, 128, "f32", 2.5, 8, plaq="device"),
        # one bin of the finite-temperature scan: 21 couplings at 48^3 x 4,
        # Polyakov loop and correlator after every sweep
        {"name": "scan 21x48^3x4 f32", "kind": "scan", "Ns": 48, "Nt": 4, "n": 21, "dtype": "f32",
         "sweeps": 50, "rmax": 24, "tuned": True},
        # the ensemble of uneven lattices in one batch
        {"name": "ensemble 64 uneven f32", "kind": "ensemble", "n": 64, "dtype": "f32",
         "draw": 5, "sweeps": 20, "tuned": True},
        # a stored configuration: links in, every observable, links out
        {"name": "config 48^3x8 f32", "kind": "config", "Ns": 48, "Nt": 8, "dtype": "f32",
         "rmax": 24},
    ]


def _chain(name, Ns, Nt, dtype, beta, sweeps, plaq="host", tuned=True):
    return {"name": name, "kind": "chain", "Ns": Ns, "Nt": Nt, "dtype": dtype, "beta": beta,
            "sweeps": sweeps, "plaq": plaq, "tuned": tuned}


def _even(rng, lo, hi):
    """An even extent, spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)))


def draw(rng):
    kind = rng.choice(["chain"] * 6 + ["ensemble", "scan", "config", "config"])
    dtype = rng.choice(["f32", "f64"])
    if kind == "chain":
        Ns = _even(rng, 4, 64)
        Nt = rng.choice([Ns, _even(rng, 4, 64)])
        # at most the link updates of the largest listed case of the precision
        most = (5.0e9 if dtype == "f32" else 2.5e8) / (4.0 * Ns ** 3 * Nt)
        long = 100.0 if dtype == "f32" else 20.0
        sweeps = max(1, int(min(most, math.exp(rng.uniform(0.0, math.log(long))))))
        c = _chain("", Ns, Nt, dtype, round(rng.uniform(2.2, 6.0), 3), sweeps,
                   rng.choice(["host", "device", "none"]), rng.random() < 0.75)
        del c["name"]
        return c
    if kind == "ensemble":
        return {"kind": kind, "n": rng.randrange(3, 65), "dtype": dtype, "draw": rng.randrange(1000),
                "sweeps": rng.randrange(1, 21) if dtype == "f32" else rng.randrange(1, 4),
                "tuned": rng.random() < 0.75}
    Ns = _even(rng, 8, 48)
    if kind == "scan":
        return {"kind": kind, "Ns": Ns, "Nt": rng.choice([4, 6, 8]), "n": rng.randrange(2, 13),
                "dtype": dtype, "sweeps": rng.randrange(5, 51) if dtype == "f32" else 4,
                "rmax": rng.randrange(1, Ns // 2 + 1), "tuned": rng.random() < 0.75}
    return {"kind": kind, "Ns": Ns, "Nt": _even(rng, 4, 32), "dtype": dtype,
            "rmax": rng.randrange(1, Ns // 2 + 1)}


# ----------------------------------------------------------------------------
# what a program has in hand before the call, and the call
# ----------------------------------------------------------------------------
def _members(case, seed):
    """(Ns, Nt, betas, seeds) of a batch."""
    if case["kind"] == "scan":
        pts = inputs.temperature_scan(case["n"], case["Ns"], case["Nt"])
    else:
        pts = inputs.batched_ensemble(case["n"], case["draw"])
    return ([p["Ns"] for p in pts], [p["Nt"] for p in pts], [p["beta"] for p in pts],
            [1000 * seed + p["seed"] for p in pts])


def _stored_links(case, seed, dev):
    """Canonical links float64[V][4][4] scattered around the identity: mean
    plaquette about 0.6, as on thermalised lattices."""
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    q = torch.randn((case["Ns"] ** 3 * case["Nt"], 4, 4), dtype=torch.float64, device=dev, generator=g)
    q *= 0.35
    q[:, :, 0] = 1.0
    return q / q.norm(dim=2, keepdim=True)


def prepare(case, seed):
    dtype = su2.F32 if case["dtype"] == "f32" else su2.F64
    s = dict(case)
    if case["kind"] == "chain":
        lat = su2.Lattice(case["Ns"], case["Nt"], dtype)
        if case["tuned"]:
            lat.autotune(beta=case["beta"])
        s["seed"] = seed
        s["out"] = {"host": True, "none": None, "device":
                    torch.zeros(case["sweeps"], dtype=torch.float64, device="cuda")}[case["plaq"]]
    elif case["kind"] == "config":
        lat = su2.Lattice(case["Ns"], case["Nt"], dtype)
        s["stored"] = _stored_links(case, seed, "cuda")
        s["read"] = torch.empty_like(s["stored"])
    else:
        Ns, Nt, s["betas"], s["seeds"] = _members(case, seed)
        lat = su2.Lattice(Ns, Nt, dtype)
        if case["tuned"]:
            lat.autotune(beta=s["betas"])
        if case["kind"] == "scan":  # a run in progress: the first sweeps are behind it
            lat.batch_init(su2.HOT, s["seeds"])
            lat.batch_heatbath(s["betas"], 10, s["seeds"], plaq=None)
    s["lat"] = lat
    s["links"] = lat.links_buf.view(torch.float32 if dtype == su2.F32 else torch.float64)
    return s


def run(s):
    lat = s["lat"]
    if s["kind"] == "chain":
        lat.init(su2.HOT, s["seed"])
        plaq = lat.heatbath(s["beta"], s["sweeps"], s["seed"], plaq=s["out"])
        return {"links": s["links"]} if plaq is None else {"plaq": plaq, "links": s["links"]}
    if s["kind"] == "ensemble":
        lat.batch_init(su2.HOT, s["seeds"])
        plaq = lat.batch_heatbath(s["betas"], s["sweeps"], s["seeds"])
        return {"plaq": plaq, "links": s["links"]}
    if s["kind"] == "scan":
        plaq, poly, corr = lat.batch_heatbath_measure(s["betas"], s["sweeps"], s["seeds"], s["rmax"])
        return {"plaq": plaq, "poly": poly, "corr": corr, "links": s["links"]}
    lat.set_links(s["stored"])
    plaq = lat.plaquette()
    loop, modulus = lat.polyakov_loop()
    corr = lat.polyakov_correlator(s["rmax"])
    lat.get_links(out=s["read"])
    return {"plaq": plaq, "loop": loop, "modulus": modulus, "corr": corr, "read": s["read"]}


# ----------------------------------------------------------------------------
# the work of one pass, and how far correct answers may lie apart
# ----------------------------------------------------------------------------
def work(case):
    link = 16 if case["dtype"] == "f32" else 32
    if case["kind"] == "config":
        V = case["Ns"] ** 3 * case["Nt"]
        # canonical links in and out in double precision; the links stored,
        # read by the measurements and read again by the last call
        return {"bytes": 4.0 * V * (2 * 32 + 3 * link), "flops": 6.0 * V * 63}
    if case["kind"] == "chain":
        sites = case["Ns"] ** 3 * case["Nt"]
    else:
        Ns, Nt, _, _ = _members(case, 0)
        sites = sum(a ** 3 * b for a, b in zip(Ns, Nt))
    updates = 4.0 * sites * case["sweeps"]
    # a checkerboard phase reads seven links for each link it writes: one of
    # its own direction and six of the others; 12 quaternion products, the
    # sums, the draw and the new link
    start = 0.0 if case["kind"] == "scan" else 4.0 * sites * link
    return {"bytes": updates * 8 * link + start, "flops": updates * 430.0}


def tolerance(case):
    # FP32: the chain of one seed is fixed bit by bit (the operations of an
    # update and its random stream do not depend on the launch shape, and one
    # flipped accept decision sends a chain elsewhere); the per-sweep
    # plaquettes sum FP32 products in a grouping of the launch shape (6e-9
    # measured).  FP64: another order of the sums moves the last bits, and
    # every sweep multiplies that (by 1.5 a sweep at beta = 2.2, measured:
    # 2e-10 after 20 sweeps).  Stored configurations: FP32 products with FP64
    # sums, the correlator's smallest terms furthest off.
    if case["kind"] == "config":
        return {"rel": 1e-6 if case["dtype"] == "f32" else 1e-13}
    return {"rel": 1e-7 if case["dtype"] == "f32" else 1e-9}


# ----------------------------------------------------------------------------
# the same in plain torch, in 64 bits
# ----------------------------------------------------------------------------
def exact(case, seed):
    """Chains in FP64 and the measurement of stored configurations; a chain
    in FP32 is not near its FP64 counterpart once an accept decision flips."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "config":
        return _exact_config(case, seed, dev)
    if case["kind"] != "chain" or case["dtype"] != "f64":
        return None
    Ns, Nt = case["Ns"], case["Nt"]
    if 4.0 * Ns ** 3 * Nt * case["sweeps"] > 1.0e9:
        return None
    L = _Exact(Ns, Nt, seed, dev)
    L.hot()
    plaq = []
    for k in range(case["sweeps"]):
        L.sweep(case["beta"], k)
        if case["plaq"] != "none":
            plaq.append(float(L.plaquette()))
    out = {"links": L.device_layout()}
    if case["plaq"] != "none":
        p = np.array(plaq)
        out["plaq"] = p[None, :] if case["plaq"] == "host" else torch.from_numpy(p)
    return out


def _exact_config(case, seed, dev):
    q = _stored_links(case, seed, dev)
    if case["dtype"] == "f32":
        q = q.float().double()
    L = _Exact(case["Ns"], case["Nt"], seed, dev)
    # [lex][mu][component] -> U[mu][component] over (t, z, y, x)
    L.U = [[q[:, mu, c].reshape(L.shape) for c in range(4)] for mu in range(4)]
    P = L.U[3]
    P = [c[0] for c in P]
    for t in range(1, case["Nt"]):
        P = _mul(P, [c[t] for c in L.U[3]])
    loop = P[0]
    corr = [float(sum((loop * loop.roll(-r, d)).sum() for d in range(3)) / (3 * loop.numel()))
            for r in range(case["rmax"] + 1)]
    m = float(loop.mean())
    return {"plaq": np.array([float(L.plaquette())]), "loop": np.array([m]),
            "modulus": np.array([abs(m)]), "corr": np.array([corr]), "read": q}


def _mul(p, q):
    """U = a0 + i a.sigma: (p0 q0 - p.q, p0 q + q0 p - p x q)."""
    return [p[0] * q[0] - p[1] * q[1] - p[2] * q[2] - p[3] * q[3],
            p[0] * q[1] + p[1] * q[0] - (p[2] * q[3] - p[3] * q[2]),
            p[0] * q[2] + p[2] * q[0] - (p[3] * q[1] - p[1] * q[3]),
            p[0] * q[3] + p[3] * q[0] - (p[1] * q[2] - p[2] * q[1])]


def _dag(p):
    return [p[0], -p[1], -p[2], -p[3]]


def _shift(p, mu, s):
    """The links at x + s mu."""
    return [c.roll(-s, 3 - mu) for c in p]


class _Exact:
    """One lattice as FP64 torch arrays over (t, z, y, x)."""

    def __init__(self, Ns, Nt, seed, dev):
        self.Ns, self.Nt, self.seed, self.dev = Ns, Nt, seed, dev
        self.shape = (Nt, Ns, Ns, Ns)
        self.V = Nt * Ns ** 3
        self.lex = torch.arange(self.V, device=dev, dtype=torch.int64)
        x, r = self.lex % Ns, self.lex // Ns
        self.parity = (x + r % Ns + (r // Ns) % Ns + r // (Ns * Ns)) % 2
        self.sites = [torch.nonzero(self.parity == p).reshape(-1) for p in (0, 1)]

    def words(self, link, sweep, tag, trial):
        """The Philox4x32-10 block of counter (link, sweep lo, tag<<24 | trial, sweep hi)."""
        M = 0xFFFFFFFF
        c = [link & M, torch.full_like(link, sweep & M), torch.full_like(link, tag << 24) | trial,
             torch.full_like(link, sweep >> 32)]
        k0, k1 = self.seed & M, (self.seed >> 32) & M
        for _ in range(10):
            a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
            c = [((b >> 32) & M) ^ c[1] ^ k0, b & M, ((a >> 32) & M) ^ c[3] ^ k1, a & M]
            k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
        return c

    @staticmethod
    def uniform(w):
        return ((w >> 9).double() + 0.5) * 2.0 ** -23

    def hot(self):
        self.U = []
        for mu in range(4):
            u = [self.uniform(w) for w in self.words(self.lex * 4 + mu, 0, 2, 0)]
            r0, r1 = (-2 * u[0].log()).sqrt(), (-2 * u[2].log()).sqrt()
            a0, a1 = 2 * math.pi * u[1], 2 * math.pi * u[3]
            self.U.append([c.reshape(self.shape) for c in _unit(
                [r0 * a0.cos(), r0 * a0.sin(), r1 * a1.cos(), r1 * a1.sin()])])

    def staple(self, mu):
        A = None
        for nu in range(4):
            if nu == mu:
                continue
            Unu, Umu = self.U[nu], self.U[mu]
            up = _mul(_mul(_shift(Unu, mu, 1), _dag(_shift(Umu, nu, 1))), _dag(Unu))
            d = _shift(Unu, nu, -1)
            lo = _mul(_mul(_dag(_shift(d, mu, 1)), _dag(_shift(Umu, nu, -1))), d)
            up = [a + b for a, b in zip(up, lo)]
            A = up if A is None else [a + b for a, b in zip(A, up)]
        return A

    def sweep(self, beta, sweep):
        for mu in range(4):
            for p in (0, 1):
                self.phase(beta, mu, p, sweep)

    def phase(self, beta, mu, p, sweep):
        at = self.sites[p]
        A = [c.reshape(-1)[at] for c in self.staple(mu)]
        k = (A[0] ** 2 + A[1] ** 2 + A[2] ** 2 + A[3] ** 2).sqrt()
        link = self.lex[at] * 4 + mu
        w = self.words(link, sweep, 0, 0)
        u1 = ((((w[0] & 511) << 9) | (w[1] & 511)).double() + 0.5) * 2.0 ** -18
        u2 = ((((w[2] & 511) << 9) | (w[3] & 511)).double() + 0.5) * 2.0 ** -18
        delta = torch.zeros_like(k)
        left = torch.arange(len(at), device=self.dev)
        for trial in range(4096):
            r1, r2, r3, r4 = (self.uniform(v) for v in w)
            lam2 = -(r1.log() + (2 * math.pi * r2).cos() ** 2 * r3.log()) / (2 * beta * k[left])
            ok = r4 ** 2 <= 1 - lam2
            delta[left[ok]] = 2 * lam2[ok]
            left = left[~ok]
            if not len(left):
                break
            w = self.words(link[left], sweep, 0, trial + 1)
        cth = 2 * u1 - 1
        sth = ((1 - cth) * (1 + cth)).sqrt()
        v = (delta * (2 - delta)).sqrt()
        phi = 2 * math.pi * u2
        X = [1 - delta, v * sth * phi.cos(), v * sth * phi.sin(), v * cth]
        new = _unit(_mul(X, _dag([a / k for a in A])))
        for c in range(4):
            flat = self.U[mu][c].reshape(-1).clone()
            flat[at] = new[c]
            self.U[mu][c] = flat.reshape(self.shape)

    def plaquette(self):
        tot = 0.0
        for mu in range(4):
            for nu in range(mu + 1, 4):
                a = _mul(self.U[mu], _shift(self.U[nu], mu, 1))
                b = _mul(self.U[nu], _shift(self.U[mu], nu, 1))
                tot = tot + sum((x * y).sum() for x, y in zip(a, b))
        return tot / (6 * self.V)

    def device_layout(self):
        """U[mu][parity][plane][index] in pairs (a0, a1), (a2, a3)."""
        out = []
        for mu in range(4):
            flat = torch.stack([c.reshape(-1) for c in self.U[mu]])
            for p in (0, 1):
                q = flat[:, self.sites[p]]
                out += [q[0:2].t().reshape(-1), q[2:4].t().reshape(-1)]
        return torch.cat(out)


def _unit(q):
    n = (q[0] ** 2 + q[1] ** 2 + q[2] ** 2 + q[3] ** 2).sqrt()
    return [c / n for c in q]
