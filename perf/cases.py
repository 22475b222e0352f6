"""The work that programs give to this package, as cases that can be timed.

Every case goes through the public entry points of ``paper_2510_00193_gb300``
(list build, energies and forces, parameter gradients, force matching, batches,
extrapolation grades, molecular dynamics) on structures that are made on the
device from a seed.  The potentials are the ones under ``potentials/``; sizes
and structures follow the repository's benchmark and tests (BCC and FCC
crystals with thermal displacements, sheared cells, small strained cells with
vacancies).

Results of the mixed path are sums formed in single precision; the programs
modelled here keep them as float32 records (trajectory frames, thermodynamic
output), converted in one go.  Everything computed in FP64 stays FP64.

``exact`` restates the model in plain torch, in FP64, on dense candidate lists.
"""
import functools
import json
import math
import os

import numpy as np
import torch

import paper_2510_00193_gb300 as P
from paper_2510_00193_gb300 import autograd as mtp_autograd

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
F64 = torch.float64
MASSES = (183.84, 95.95, 50.94)              # W, Mo, V, in amu
KB = 8.617333262e-5                          # eV / K
MVV2E = 1.0364269e-4                         # amu A^2 / ps^2 in eV
TAU_SEL, TAU_BRK = 2.0, 10.0                 # selection and break thresholds of the grade


# ---------------------------------------------------------------- the cases

def _case(name, kind, pot, lattice, cells, a, sigma, precision="mixed", **more):
    c = {"kind": kind, "pot": pot, "lattice": lattice, "n1": cells[0], "n2": cells[1], "n3": cells[2], "a": a,
         "sigma": sigma, "tilt": 0.0, "precision": precision}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call a program makes: one energy/force evaluation of a 128-atom box with the
        # smallest potential (a relaxation or a check of a fitted potential).
        _case("efv_l8_128", "efv", "bcc-l8-s1", "bcc", (4, 4, 4), 3.16, 0.05, dtheta=False, fresh=False),
        # A few thousand atoms per GPU, the regime of the block-parallel variant: one step of a small run.
        _case("efv_l16_2000", "efv", "bcc-l16-s3", "bcc", (10, 10, 10), 3.16, 0.08, dtheta=False, fresh=False),
        # A configuration seen for the first time (sheared cell, odd sizes, the wider cutoff): list build and
        # evaluation, as a relaxation with cell changes or a scan over stored structures does it.
        _case("fresh_l16_14858", "efv", "bcc-l16-s3-rc5.6", "bcc", (17, 19, 23), 3.16, 0.08, dtheta=False,
              fresh=True, tilt=0.08),
        # The large-system evaluation (one step of a million-atom run on a list that is reused).
        _case("efv_l16_1024000", "efv", "bcc-l16-s3", "bcc", (80, 80, 80), 3.16, 0.08, dtheta=False, fresh=False),
        # FP64 energies, forces and parameter gradient: the fitting program's reference evaluation.
        _case("fp64_dtheta_l16_48546", "efv", "bcc-l16-s3", "bcc", (27, 29, 31), 3.16, 0.08, "fp64", dtheta=True,
              fresh=False),
        # The high-level potential on a small box (the block-parallel regime of the case studies).
        _case("efv_l20_2016", "efv", "fcc-l20-s4", "fcc", (7, 8, 9), 3.6, 0.1, dtheta=False, fresh=False),
        # The high-level potential on a large box.
        _case("efv_l20_108000", "efv", "fcc-l20-s4", "fcc", (30, 30, 30), 3.6, 0.1, dtheta=False, fresh=False),
        # One force-matching training step through autograd: forward, backward and double backward, FP64.
        _case("force_match_l20_4000", "force_match", "fcc-l20-s4", "fcc", (10, 10, 10), 3.6, 0.1, "fp64"),
        # One pass over a training set of 4096 small cells with energies, forces, virials and dE/dtheta.
        _case("batch_dtheta_4096", "batch", "gas-l16-s2", "bcc", (0, 0, 0), 2.866, 0.1, n_cfg=4096, lo=8, hi=256,
              dtheta=True),
        # A large configuration seen for the first time, with a cheap potential: the list build is most of it.
        _case("fresh_l8_500000", "efv", "bcc-l8-s1", "bcc", (50, 50, 100), 3.16, 0.08, dtheta=False, fresh=True),
        # Active learning: the neighbourhood grade of every atom of a large strongly displaced box.
        _case("grade_500000", "grade", "bcc-l16-s1", "bcc", (50, 50, 100), 3.16, 0.15, "fp64"),
        # Molecular dynamics: 20 velocity-Verlet steps with the displacement check on every step.
        _case("md_l16_16000", "md", "bcc-l16-s3", "bcc", (20, 20, 20), 3.16, 0.04, steps=20, dt=2.5e-4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(rng, lattice, lo, hi, least=2):
    """Three unequal edge lengths (in unit cells) for between lo and hi atoms."""
    per = 4 if lattice == "fcc" else 2
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    edge = (n / per) ** (1.0 / 3.0)
    n1 = max(least, int(round(edge * rng.uniform(0.75, 1.3))))
    n2 = max(least, int(round(edge * rng.uniform(0.75, 1.3))))
    n3 = max(least, int(n / per / (n1 * n2)))
    while per * n1 * n2 * n3 > hi and max(n1, n2, n3) > least:
        n1, n2, n3 = (v - 1 if v == max(n1, n2, n3) else v for v in (n1, n2, n3))
    return n1, n2, n3


def draw(rng):
    kind = rng.choice(["efv"] * 7 + ["force_match", "force_match", "batch", "batch", "grade", "md"])
    if kind == "efv":
        pot = rng.choice(["bcc-l8-s1", "bcc-l16-s3", "bcc-l16-s3", "bcc-l16-s3-rc5.6", "fcc-l20-s4", "fcc-l20-s4"])
        lattice = "fcc" if pot.startswith("fcc") else "bcc"
        precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        hi = {("fcc", "mixed"): 108000, ("fcc", "fp64"): 4000, ("bcc", "mixed"): 1024000, ("bcc", "fp64"): 48000}
        return _case("", kind, pot, lattice, _cells(rng, lattice, 128, hi[lattice, precision]),
                     (3.6 if lattice == "fcc" else 3.16) * rng.uniform(0.99, 1.02), rng.uniform(0.05, 0.1), precision,
                     dtheta=rng.random() < 0.3, fresh=rng.random() < 0.3, tilt=rng.choice([0.0, rng.uniform(0.02, 0.1)]))
    if kind == "force_match":
        pot, lattice, a, hi = rng.choice([("fcc-l20-s4", "fcc", 3.6, 4000), ("bcc-l16-s3", "bcc", 3.16, 16000)])
        return _case("", kind, pot, lattice, _cells(rng, lattice, 128, hi), a, rng.uniform(0.05, 0.1),
                     rng.choice(["fp64", "fp64", "mixed"]), tilt=rng.choice([0.0, 0.05]))
    if kind == "batch":
        precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        lo = rng.randint(4, 16)
        return _case("", kind, "gas-l16-s2", "bcc", (0, 0, 0), 2.866, rng.uniform(0.05, 0.12), precision,
                     n_cfg=_log_int(rng, 16, 4096 if precision == "mixed" else 256), lo=lo,
                     hi=_log_int(rng, 2 * lo, 256), dtheta=rng.random() < 0.7)
    if kind == "grade":
        return _case("", kind, "bcc-l16-s1", "bcc", _cells(rng, "bcc", 250, 500000), 3.16, rng.uniform(0.08, 0.15), "fp64")
    return _case("", kind, "bcc-l16-s3", "bcc", _cells(rng, "bcc", 250, 16000, 4), 3.16, rng.uniform(0.03, 0.05),
                 steps=rng.randint(8, 20), dt=2.5e-4)


# ------------------------------------------------------------------- inputs

@functools.lru_cache(maxsize=None)
def _json(name):
    with open(os.path.join(ROOT, "potentials", name + ".json")) as fh:
        return json.load(fh)


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed, stream):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) * 16 + stream)
    return g


def _species(n, kinds, gen):
    return (torch.randperm(n, generator=gen, device=_dev()) % kinds).to(torch.int32)


def _sites(lattice):
    b = [[0.0, 0.0, 0.0], [0.5, 0.5, 0.5]] if lattice == "bcc" else [[0.0, 0.0, 0.0], [0.0, 0.5, 0.5], [0.5, 0.0, 0.5],
                                                                    [0.5, 0.5, 0.0]]
    return torch.tensor(b, dtype=F64, device=_dev())


def _crystal(case, seed):
    """Displaced lattice: positions before wrapping, the deformation of the unit cube's axes, and the cell."""
    dev, n = _dev(), (case["n1"], case["n2"], case["n3"])
    t = case["tilt"]
    axes = case["a"] * np.array([[1.0, 0.0, 0.0], [t, 1.0 - 0.3 * t, 0.0], [-0.5 * t, 0.7 * t, 1.0 + 0.2 * t]])
    g = torch.stack(torch.meshgrid(*[torch.arange(k, device=dev) for k in n], indexing="ij"), -1).reshape(-1, 3)
    frac = (g[:, None, :] + _sites(case["lattice"])[None]).reshape(-1, 3)
    x = frac @ torch.tensor(axes, device=dev)
    x += case["sigma"] * torch.randn(x.shape, generator=_gen(seed, 1), dtype=F64, device=dev)
    return x, axes, axes * np.array(n, dtype=np.float64)[:, None]


def _wrapped(x, cell):
    h = torch.tensor(cell, dtype=F64, device=x.device)
    s = x @ torch.linalg.inv(h)
    s = s - torch.floor(s)
    return (torch.where(s >= 1.0, torch.zeros_like(s), s) @ h).contiguous()


def _training_set(case, seed):
    """Small strained cells with displacements and vacancies: sizes log-uniform in [lo, hi], the same for every seed."""
    r = np.random.default_rng([case["n_cfg"], case["lo"], case["hi"]])
    sizes = np.floor(np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"] + 1), case["n_cfg"]))).astype(np.int64)
    off = np.concatenate([[0], np.cumsum(sizes)])
    r = np.random.default_rng(int(seed))
    cells = np.zeros((case["n_cfg"], 3, 3))
    x = np.empty((off[-1], 3))
    for k, n in enumerate(sizes):
        pairs = -(-int(n) // 2)
        e = max(1, round(pairs ** (1.0 / 3.0)))
        dims = (e, e, -(-pairs // (e * e)))
        g = np.indices(dims).reshape(3, -1).T
        f = np.concatenate([g, g + 0.5])
        f = f[r.permutation(len(f))[:n]]
        axes = case["a"] * (np.eye(3) + np.tril(r.uniform(-0.05, 0.05, (3, 3))))
        cells[k] = axes * np.array(dims)[:, None]
        x[off[k]:off[k + 1]] = f @ axes
    x += r.normal(0.0, case["sigma"], x.shape)
    return off, cells, x


def _records(n, dtheta_n, rows=1):
    """One FP64 buffer for everything an evaluation returns, and the views of it that the calls fill."""
    sizes = {"forces": (n, 3), "e_atom": (n,), "virial": (rows, 6), "e": (rows,)}
    if dtheta_n:
        sizes["dtheta"] = (rows, dtheta_n)
    at, where = 0, {}
    for k, s in sizes.items():
        where[k] = (at, s)
        at += -(-math.prod(s) // 2) * 2                  # every part starts on 16 bytes
    flat = torch.empty(at, dtype=F64, device=_dev())
    return flat, where


def _parts(flat, where):
    return {k: flat[at:at + math.prod(s)].view(s) for k, (at, s) in where.items()}


def prepare(case, seed):
    pot_json = _json(case["pot"])
    pot = P.Potential.from_dict(pot_json, check_basis=False)
    prec = P.MTP_MIXED if case["precision"] == "mixed" else P.MTP_FP64
    st = {"kind": case["kind"], "pot": pot, "prec": prec, "mixed": case["precision"] == "mixed"}
    if case["kind"] == "batch":
        off, cells, x = _training_set(case, seed)
        st["x"] = torch.tensor(x, dtype=F64, device=_dev())
        st["z"] = _species(x.shape[0], pot.n_species, _gen(seed, 2))
        st["batch"] = P.mtp_batch_create(pot, off, cells, st["x"])
        st["dtheta"] = case["dtheta"]
        st["flat"], st["where"] = _records(x.shape[0], pot.n_params if case["dtheta"] else 0, case["n_cfg"])
        parts = _parts(st["flat"], st["where"])
        st["out"] = {"e_cfg": parts["e"], "e_atom": parts["e_atom"], "forces": parts["forces"],
                     "virial": parts["virial"], "dtheta": parts.get("dtheta")}
        return st
    x, _, cell = _crystal(case, seed)
    st["x"], st["cell"] = _wrapped(x, cell), cell
    n = x.shape[0]
    st["z"] = _species(n, pot.n_species, _gen(seed, 2))
    if case["kind"] == "md":
        m = torch.tensor(MASSES[:pot.n_species], dtype=F64, device=_dev())[st["z"].long()][:, None]
        v = torch.randn(n, 3, generator=_gen(seed, 3), dtype=F64, device=_dev()) * torch.sqrt(300.0 * KB / (m * MVV2E))
        st["v"] = v - (m * v).sum(0) / m.sum()
        st["md"] = P.MD(pot, st["x"], cell)
        st["f"] = P.mtp_compute_efv(pot, st["md"].nlist(), st["x"], st["z"], cell, precision=prec)["forces"]
        st["now"] = [torch.empty_like(st["x"]) for _ in range(3)]
        st["e"] = torch.zeros(2, case["steps"], dtype=F64, device=_dev())
        st["dt"], st["steps"] = case["dt"], case["steps"]
        return st
    st["nl"] = P.mtp_build_neighbors(pot, st["x"], cell)
    if case["kind"] == "efv":
        st["dtheta"], st["fresh"] = case["dtheta"], case["fresh"]
        st["flat"], st["where"] = _records(n, pot.n_params if case["dtheta"] else 0)
        parts = _parts(st["flat"], st["where"])
        st["out"] = {"e_atom": parts["e_atom"], "forces": parts["forces"], "virial": parts["virial"],
                     "e_total": parts["e"], "dtheta": parts.get("dtheta")}
    elif case["kind"] == "force_match":
        st["theta"] = pot.initial_theta().requires_grad_()
        st["target"] = 0.5 * torch.randn(n, 3, generator=_gen(seed, 4), dtype=F64, device=_dev())
    elif case["kind"] == "grade":
        a = _json(case["pot"] + "-active")
        st["a_inv"] = torch.tensor(a["a_inv"], dtype=F64, device=_dev()).view(a["m"], a["m"])
    return st


# --------------------------------------------------------------------- runs

def _kept(st):
    """What the program keeps of an evaluation: FP64 as it is, mixed results as one float32 record."""
    return _parts(st["flat"].float() if st["mixed"] else st["flat"], st["where"])


def _force_match(st):
    x = st["x"].detach().requires_grad_()
    e = mtp_autograd.energy(st["pot"], st["nl"], x, st["z"], st["cell"], st["theta"], precision=st["prec"])
    f = -torch.autograd.grad(e, x, create_graph=True)[0]
    loss = ((f - st["target"]) ** 2).mean()
    grad, = torch.autograd.grad(loss, st["theta"])
    out = {"energy": e.detach(), "loss": loss.detach(), "forces": f.detach(), "theta_grad": grad}
    return {k: v.float() for k, v in out.items()} if st["mixed"] else out


def run(state):
    st, kind = state, state["kind"]
    if kind == "efv":
        if st["fresh"]:
            P.mtp_build_neighbors(st["pot"], st["x"], st["cell"], nlist=st["nl"])
        P.mtp_compute_efv(st["pot"], st["nl"], st["x"], st["z"], st["cell"], precision=st["prec"], dtheta=st["dtheta"],
                          out=st["out"])
        return _kept(st)
    if kind == "batch":
        P.mtp_compute_batch(st["pot"], st["batch"], st["x"], st["z"], precision=st["prec"], dtheta=st["dtheta"],
                            out=st["out"])
        return _kept(st)
    if kind == "force_match":
        return _force_match(st)
    if kind == "grade":
        out = P.mtp_compute_grade(st["pot"], st["nl"], st["x"], st["z"], st["cell"], a_inv=st["a_inv"],
                                  tau_sel=TAU_SEL, tau_brk=TAU_BRK)
        return {"gamma": out["gamma"], "flags": out["flags"], "gamma_max": out["gamma_max"], "status": out["status"]}
    x, v, f = st["now"]                                   # a run that starts from a stored state
    x.copy_(st["x"])
    v.copy_(st["v"])
    f.copy_(st["f"])
    st["md"].run(x, v, st["z"], MASSES[:st["pot"].n_species], st["dt"], st["steps"], f, rebuild_every=-1,
                 precision=st["prec"], e_pot=st["e"][0], e_kin=st["e"][1])
    if st["mixed"]:                                       # one trajectory frame and the thermodynamic lines
        return {"x": x, "v": v.float(), "forces": f.float(), "energies": st["e"].float()}
    return {"x": x, "v": v, "forces": f, "energies": st["e"]}


# --------------------------------------------------------------------- work

#: per level: flops of a pair's moment terms and adjoint (components with a z-exponent of at most 1, which
#: determine the others because the pair vector is a unit vector), and of an atom's contraction with its reverse
_FLOPS = {8: (8 + 16 + 66, 148), 16: (48 + 160 + 530, 7043), 20: (80 + 320 + 1055, 62000)}


def _per_atom(pot, density, forces=True):
    q, mu = pot["n_q"], pot["n_mu"]
    pair, atom = _FLOPS[pot["level"]]
    pairs = density * 4.0 / 3.0 * math.pi * pot["r_cut"] ** 3
    radial = 4 + 2 * mu + (q - 2) * (3 + 2 * mu) + mu
    slope = (q - 2) * (4 + 2 * mu) + 1 + 4 * mu
    if not forces:                                        # moments and basis values alone
        return pairs, pairs * (28 + radial + pair // 3) + atom // 3
    return pairs, pairs * (28 + radial + slope + pair + 24) + atom


def work(case):
    pot = _json(case["pot"])
    per = 4 if case["lattice"] == "fcc" else 2
    density = per / case["a"] ** 3
    n = per * case["n1"] * case["n2"] * case["n3"]
    theta = 8 * (pot["n_species"] + len(pot["radial"]) + pot["m"])
    kind = case["kind"]
    if kind == "batch":
        lo, hi = case["lo"], case["hi"] + 1
        n = int(case["n_cfg"] * ((hi - lo) / math.log(hi / lo) - 0.5))
    pairs, flops = _per_atom(pot, density, kind != "grade")
    read = 28 * n + 8 * n * pairs                         # positions, species, list entries
    if kind == "efv":
        listing = 8 * n * pairs if case["fresh"] else 0   # the list is written before it is read
        return {"bytes": read + listing + 32 * n + theta * (1 + case["dtheta"]),
                "flops": n * (flops + (pairs * 3 * pot["n_q"] * pot["n_mu"] if case["dtheta"] else 0))}
    if kind == "batch":
        return {"bytes": read + 32 * n + case["n_cfg"] * (128 + (theta if case["dtheta"] else 0)),
                "flops": n * (flops + (pairs * 3 * pot["n_q"] * pot["n_mu"] if case["dtheta"] else 0))}
    if kind == "force_match":                             # value and directional derivative: three times one pass
        return {"bytes": read + 72 * n + 3 * theta, "flops": 4.0 * n * flops}
    if kind == "grade":
        m = pot["m"]
        return {"bytes": read + 9 * n + 8 * m * m, "flops": n * (flops + 2.0 * m * m)}
    return {"bytes": case["steps"] * (read + 96 * n), "flops": case["steps"] * n * (flops + 30)}


# -------------------------------------------- the model in plain torch, FP64

def _multi(n):
    return [(a, b, n - a - b) for a in range(n, -1, -1) for b in range(n - a, -1, -1)]


class _Model:
    def __init__(self, name):
        d = _json(name)
        t = lambda v, s: torch.tensor(v, dtype=F64, device=_dev()).view(s)  # noqa: E731
        k = d["n_species"]
        self.s, self.xi = t(d["species_energy"], (k,)), t(d["xi"], (d["m"],))
        self.c = t(d["radial"], (d["n_mu"], d["n_q"], k, k))
        self.r_min, self.r_cut, self.n_q, self.n_mu, self.kinds = d["r_min"], d["r_cut"], d["n_q"], d["n_mu"], k
        self.graphs, self.bases = [], []
        seen = {}
        for b in d["basis"]:
            for g in b:
                key = json.dumps(g)
                if key not in seen:
                    seen[key] = len(self.graphs)
                    self.graphs.append(g)
            self.bases.append([seen[json.dumps(g)] for g in b])
        nu = 0
        for mus, e in self.graphs:
            deg = [0] * len(mus)
            for (i, j), m in zip(((i, j) for i in range(len(mus)) for j in range(i + 1, len(mus))), e):
                deg[i] += m
                deg[j] += m
            nu = max([nu] + deg)
        self.multi = [k for n in range(nu + 1) for k in _multi(n)]
        self.at = {k: i for i, k in enumerate(self.multi)}
        self.plans = [self._plan(mus, e) for mus, e in self.graphs]

    def _plan(self, mus, e):
        """Every edge of multiplicity n is one index over the multi-indices of degree n with multinomial weights."""
        ends = [[] for _ in mus]
        for (i, j), m in zip(((i, j) for i in range(len(mus)) for j in range(i + 1, len(mus))), e):
            if m:
                letter = "abcdefghijklmnop"[sum(len(v) for v in ends) // 2]
                ends[i].append((letter, m, True))
                ends[j].append((letter, m, False))
        terms, what = [], []
        for mu, v in zip(mus, ends):
            idx = np.zeros([len(_multi(m)) for _, m, _ in v], dtype=np.int64)
            w = np.ones(idx.shape)
            for pos in np.ndindex(*idx.shape):
                ks = [_multi(m)[p] for p, (_, m, _) in zip(pos, v)]
                idx[pos] = self.at[tuple(sum(k[d] for k in ks) for d in range(3))]
                for k, (_, m, first) in zip(ks, v):
                    if first:
                        w[pos] *= math.factorial(m) / math.prod(math.factorial(q) for q in k)
            terms.append("z" + "".join(x[0] for x in v))
            what.append((mu, torch.tensor(idx, device=_dev()), torch.tensor(w, device=_dev())))
        return ",".join(terms) + "->z", what

    def sites(self, r, zi, zj, on, c=None, xi=None, s=None):
        """Site energies, basis rows and the radial functions' parts of dense neighbourhoods r [n, K, 3]."""
        c, xi, s = self.c if c is None else c, self.xi if xi is None else xi, self.s if s is None else s
        d = torch.sqrt((r * r).sum(-1))
        u = r / d[..., None]
        t = (2.0 * d - self.r_min - self.r_cut) / (self.r_cut - self.r_min)
        q = [torch.ones_like(t), t]
        for _ in range(2, self.n_q):
            q.append(2.0 * t * q[-1] - q[-2])
        q = torch.stack(q[:self.n_q], -1) * (torch.where(on, self.r_cut - d, torch.zeros_like(d)) ** 2)[..., None]
        f = torch.zeros(*d.shape, self.n_mu, dtype=F64, device=r.device)
        for a in range(self.kinds):
            for b in range(self.kinds):
                both = ((zi[:, None] == a) & (zj == b)).to(F64)[..., None]
                f = f + both * (q @ c[:, :, a, b].T)
        mono = {(0, 0, 0): torch.ones_like(d)}
        for k in self.multi[1:]:
            ax = next(i for i in range(3) if k[i])
            mono[k] = mono[tuple(v - (i == ax) for i, v in enumerate(k))] * u[..., ax]
        mom = f.transpose(1, 2) @ torch.stack([mono[k] for k in self.multi], -1)         # [n, mu, multi-index]
        g = []
        for eq, what in self.plans:
            g.append(torch.einsum(eq, *[mom[:, mu][:, idx.reshape(-1)].view(-1, *idx.shape) * w for mu, idx, w in what]))
        rows = torch.stack([functools.reduce(lambda p, k: p * g[k], b[1:], g[b[0]]) for b in self.bases], -1)
        return s[zi.long()] + rows @ xi, rows, (q, f)


@functools.lru_cache(maxsize=None)
def _model(name):
    return _Model(name)


class _Lattice:
    """Candidate neighbours of a displaced lattice: every lattice offset that the displacements can bring inside."""

    def __init__(self, case, axes, cell, reach):
        dev, base = _dev(), _sites(case["lattice"]).cpu().numpy()
        self.n = torch.tensor([case["n1"], case["n2"], case["n3"]], device=dev)
        self.cell = torch.tensor(cell, dtype=F64, device=dev)
        self.per = len(base)
        lim = [int(reach / h) + 2 for h in 1.0 / np.linalg.norm(np.linalg.inv(axes), axis=0)]
        box = np.stack(np.meshgrid(*[np.arange(-k, k + 1) for k in lim], indexing="ij"), -1).reshape(-1, 3)
        self.off = []
        for b in range(self.per):
            rows = [(o, t) for t in range(self.per) for o in box[np.linalg.norm((box + base[t] - base[b]) @ axes, axis=1) < reach]
                    if t != b or any(o)]
            self.off.append((torch.tensor(np.array([o for o, _ in rows]), device=dev),
                             torch.tensor([t for _, t in rows], device=dev)))

    def rows(self, x, lo, hi):
        """(centres, j, r) of the atoms of unit cells lo..hi, one block per basis atom."""
        cells = torch.arange(lo, hi, device=x.device)
        g = torch.stack([cells // (self.n[1] * self.n[2]), cells // self.n[2] % self.n[1], cells % self.n[2]], -1)
        for b, (o, t) in enumerate(self.off):
            to = g[:, None, :] + o[None]
            img = torch.div(to, self.n, rounding_mode="floor")
            k = to - img * self.n
            j = ((k[..., 0] * self.n[1] + k[..., 1]) * self.n[2] + k[..., 2]) * self.per + t[None]
            i = cells * self.per + b
            yield i, j, x[j] + img.to(F64) @ self.cell - x[i][:, None, :]


def _blocks(case, model, axes, cell, x, slack=0.0):
    """Dense neighbourhoods (i, j, r, inside) of a crystal, a bounded number of atoms at a time."""
    lat = _Lattice(case, axes, cell, model.r_cut + 13.0 * case["sigma"] + slack)
    cells = int(lat.n.prod())
    step = max(1, int(1.2e9 / (8.0 * len(lat.off[0][1]) * len(model.multi))))
    for lo in range(0, cells, step):
        for i, j, r in lat.rows(x, lo, min(cells, lo + step)):
            on = (r * r).sum(-1) < model.r_cut ** 2
            order = torch.argsort((~on).to(torch.int8), dim=1, stable=True)[:, :int(on.sum(1).max())]
            on, j = on.gather(1, order), j.gather(1, order)
            r = r.gather(1, order[..., None].expand(-1, -1, 3))
            far = torch.tensor([0.6, 0.7, 0.8], dtype=F64, device=r.device) * model.r_cut
            yield i, j, torch.where(on[..., None], r, far), on


def _evaluate(model, blocks, n, z, dtheta=False, cfg=None, n_cfg=1):
    """Site energies, forces, virials and dE/dtheta (per configuration) summed over neighbourhood blocks."""
    dev = z.device
    e, f = torch.zeros(n, dtype=F64, device=dev), torch.zeros(n, 3, dtype=F64, device=dev)
    w = torch.zeros(n_cfg, 6, dtype=F64, device=dev)
    k2, c = model.kinds ** 2, model.c
    g_c = torch.zeros(n_cfg * k2, c.shape[0] * c.shape[1], dtype=F64, device=dev)
    g_xi = torch.zeros(n_cfg, model.xi.numel(), dtype=F64, device=dev)
    cfg = torch.zeros(n, dtype=torch.long, device=dev) if cfg is None else cfg
    for i, j, r, on in blocks:
        r = r.detach().requires_grad_()
        es, rows, (q, fr) = model.sites(r, z[i], z[j], on)
        g, gf = torch.autograd.grad(es.sum(), (r, fr))
        g = torch.where(on[..., None], g, torch.zeros_like(g))
        e[i] = es.detach()
        f.index_add_(0, i, g.sum(1))
        f.index_add_(0, j.reshape(-1), -g.reshape(-1, 3))
        rd = r.detach()
        pair = torch.stack([g[..., a] * rd[..., b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], -1)
        w.index_add_(0, cfg[i], -pair.sum(1))
        if dtheta:
            g_xi.index_add_(0, cfg[i], rows.detach())
            slot = (cfg[i] * k2 + z[i].long() * model.kinds)[:, None] + z[j].long()
            part = (gf[..., :, None] * q.detach()[..., None, :]).reshape(-1, c.shape[0] * c.shape[1])
            g_c.index_add_(0, slot.reshape(-1), part)
    out = {"forces": f, "e_atom": e, "virial": w,
           "e": torch.zeros(n_cfg, dtype=F64, device=dev).index_add_(0, cfg, e)}
    if dtheta:
        g_s = torch.zeros(n_cfg * model.kinds, dtype=F64, device=dev)
        g_s.index_add_(0, cfg * model.kinds + z.long(), torch.ones(n, dtype=F64, device=dev))
        g_c = g_c.view(n_cfg, k2, -1).transpose(1, 2).reshape(n_cfg, -1)
        out["dtheta"] = torch.cat([g_s.view(n_cfg, -1), g_c, g_xi], 1)
    return out


def _set_blocks(model, off, cells, x):
    """Neighbourhood blocks of many small cells, by brute force over images."""
    dev, held, count = x.device, [], 0

    def dense(held):
        i, j, r = (torch.cat(v) for v in zip(*held))
        own, row, num = torch.unique(i, return_inverse=True, return_counts=True)
        first = torch.cumsum(num, 0) - num
        col = torch.arange(i.numel(), device=dev) - first[row]
        kk = int(num.max())
        jj = torch.zeros(own.numel(), kk, dtype=torch.long, device=dev)
        far = torch.tensor([0.6, 0.7, 0.8], dtype=F64, device=dev) * model.r_cut
        rr = far.expand(own.numel(), kk, 3).clone()
        on = torch.zeros(own.numel(), kk, dtype=torch.bool, device=dev)
        jj[row, col], rr[row, col], on[row, col] = j, r, True
        return own, jj, rr, on

    for k in range(len(cells)):
        h = cells[k]
        lim = [int(model.r_cut * v + 1.5) + 1 for v in np.linalg.norm(np.linalg.inv(h), axis=0)]
        box = np.stack(np.meshgrid(*[np.arange(-v, v + 1) for v in lim], indexing="ij"), -1).reshape(-1, 3)
        shift = torch.tensor(box @ h, dtype=F64, device=dev)
        p = x[off[k]:off[k + 1]]
        r = p[None, :, None, :] + shift[None, None] - p[:, None, None, :]
        d2 = (r * r).sum(-1)
        i, j, m = torch.nonzero((d2 < model.r_cut ** 2) & (d2 > 0.0), as_tuple=True)
        if i.numel():
            held.append((i + int(off[k]), j + int(off[k]), r[i, j, m]))
            count += p.shape[0]
        if held and (count >= 8000 or k + 1 == len(cells)):
            yield dense(held)
            held, count = [], 0


def _exact_force_match(case, seed, model, axes, cell, x, z):
    n = x.shape[0]
    d = _evaluate(model, _blocks(case, model, axes, cell, x), n, z)
    target = 0.5 * torch.randn(n, 3, generator=_gen(seed, 4), dtype=F64, device=_dev())
    diff = d["forces"] - target
    v = 2.0 * diff / diff.numel()
    c, xi = model.c.clone().requires_grad_(), model.xi.clone().requires_grad_()
    g_c, g_xi = torch.zeros_like(c), torch.zeros_like(xi)
    for i, j, r, on in _blocks(case, model, axes, cell, x):
        for part in torch.split(torch.arange(i.numel(), device=_dev()), 500):
            rp = r[part].detach().requires_grad_()
            es, _, _ = model.sites(rp, z[i[part]], z[j[part]], on[part], c, xi)
            g, = torch.autograd.grad(es.sum(), rp, create_graph=True)
            along = torch.where(on[part][..., None], v[j[part]] - v[i[part]][:, None, :], torch.zeros_like(rp))
            a, b = torch.autograd.grad(-(g * along).sum(), (c, xi))
            g_c += a
            g_xi += b
    grad = torch.cat([torch.zeros_like(model.s), g_c.detach().reshape(-1), g_xi.detach()])
    return {"energy": d["e"][0], "loss": (diff ** 2).mean(), "forces": d["forces"], "theta_grad": grad}


def _exact_md(case, seed, model, axes, cell, x, z):
    n, dt = x.shape[0], case["dt"]
    m = torch.tensor(MASSES[:model.kinds], dtype=F64, device=_dev())[z.long()][:, None] * MVV2E
    v = torch.randn(n, 3, generator=_gen(seed, 3), dtype=F64, device=_dev()) * torch.sqrt(300.0 * KB / m)
    v = v - (m * v).sum(0) / m.sum()
    start = _wrapped(x, cell) - x                          # the program's positions are the wrapped ones
    force = lambda y: _evaluate(model, _blocks(case, model, axes, cell, y, 0.5), n, z)  # noqa: E731
    f, e = force(x)["forces"], []
    for _ in range(case["steps"]):
        v = v + 0.5 * dt * f / m
        x = x + dt * v
        d = force(x)
        f = d["forces"]
        v = v + 0.5 * dt * f / m
        e.append(torch.stack([d["e"][0], (0.5 * m * v * v).sum()]))
    return {"x": x + start, "v": v, "forces": f, "energies": torch.stack(e, 1)}


def exact(case, seed):
    kind = case["kind"]
    model = _model(case["pot"])
    if kind == "batch":
        off, cells, x = _training_set(case, seed)
        x = torch.tensor(x, dtype=F64, device=_dev())
        z = _species(x.shape[0], model.kinds, _gen(seed, 2))
        cfg = torch.repeat_interleave(torch.arange(case["n_cfg"], device=_dev()),
                                      torch.tensor(np.diff(off), device=_dev()))
        d = _evaluate(model, _set_blocks(model, off, cells, x), x.shape[0], z, case["dtheta"], cfg, case["n_cfg"])
        alone = d["e_atom"] == 0.0                         # atoms without neighbours
        d["e_atom"] = torch.where(alone, model.s[z.long()], d["e_atom"])
        d["e"] = torch.zeros_like(d["e"]).index_add_(0, cfg, d["e_atom"])
        return d
    x, axes, cell = _crystal(case, seed)
    z = _species(x.shape[0], model.kinds, _gen(seed, 2))
    if kind == "force_match":
        return _exact_force_match(case, seed, model, axes, cell, x, z)
    if kind == "md":
        return _exact_md(case, seed, model, axes, cell, x, z)
    if kind == "grade":
        a = _json(case["pot"] + "-active")
        a_inv = torch.tensor(a["a_inv"], dtype=F64, device=_dev()).view(a["m"], a["m"])
        gamma = torch.empty(x.shape[0], dtype=F64, device=_dev())
        with torch.no_grad():
            for i, j, r, on in _blocks(case, model, axes, cell, x):
                _, rows, _ = model.sites(r, z[i], z[j], on)
                gamma[i] = (rows @ a_inv).abs().max(1).values
        return {"gamma": gamma, "flags": None, "gamma_max": float(gamma.max()), "status": None}
    return _evaluate(model, _blocks(case, model, axes, cell, x), x.shape[0], z, case["dtheta"])
