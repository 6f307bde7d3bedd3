"""Performance cases: the calls a lattice-QCD program makes through the public entry points.

A case is a dict of plain values whose "kind" names the entry point:

  schur       Handle.apply / apply_dagger on even-site fields (FP64 preconditioned operator)
  dirac       Handle.apply / apply_dagger on full 5D fields (FP64 Dirac operator)
  normal      Handle.apply_normal, S^dag S in FP64 (residual checks, Lanczos, Chebyshev filters)
  solve       Handle.cg_solve / cg_solve_batched, S^dag S x = b for several masses
  propagator  Handle.cg_solve on the full lattice, D x = b (valence propagators)
  serve       Server.submit / poll, several requests on one resident gauge field
  flow        Flow.set_gauge / run / get_gauge, gradient flow with measurements
  gauge       Handle.gauge_force, Wilson gauge action and force
  md          Handle.md_trajectory, Omelyan step with two-flavour pseudofermion terms

Solves run to 1e-11, ten times below the usual 1e-10, so that a solution is determined to better
than 1e-9 by its system alone at every mass used here.  `exact` restates the definitions in plain
FP64 torch.
"""
import math

import numpy as np
import torch

import paper_1811_08095_gb300 as odwf

M0 = 1.3          # domain-wall height of every configuration of this repository
LMIN, LMAX = 0.05, 6.2
TOL = 1e-11
BETA = 6.2
LAMBDA = 0.1931833275037836  # minimum-norm second-order integrator
DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one operator application on the 4^4 x 8 test lattice (launch latency)
        dict(name="schur_4x4x4x4_ns8", kind="schur", lx=4, ly=4, lz=4, lt=4, ns=8, mq=0.01, dagger=False, tbc=True),
        # a full Dirac operator on a ragged lattice with periodic time (spectrum and symmetry checks)
        dict(name="dirac_dag_6x10x4x14_ns16", kind="dirac", lx=6, ly=10, lz=4, lt=14, ns=16, mq=0.1, dagger=True,
             tbc=False),
        # the normal operator on the 16^3 x 32 x 16 lattice of the default benchmark workload
        dict(name="normal_16x16x16x32_ns16", kind="normal", lx=16, ly=16, lz=16, lt=32, ns=16, mq=0.04, tbc=True),
        # a single mixed-precision solve on the 4^4 x 8 lattice: iteration latency
        dict(name="solve_f16_4x4x4x4_ns8", kind="solve", lx=4, ly=4, lz=4, lt=4, ns=8, masses="0.04", prec="f16",
             links="f32", tbc=True),
        # one right-hand side in BF16 storage (the 64^4 workload's storage) on a middle lattice
        dict(name="solve_bf16_12x12x12x24_ns16", kind="solve", lx=12, ly=12, lz=12, lt=24, ns=16, masses="0.04",
             prec="bf16", links="f32", tbc=True),
        # the default benchmark workload: three masses in one batch on 16^3 x 32 x 16
        dict(name="solve_f16_16x16x16x32_ns16_3mass", kind="solve", lx=16, ly=16, lz=16, lt=32, ns=16,
             masses="0.002,0.04,0.5", prec="f16", links="f32", tbc=True),
        # plain FP64 CG (reference solves, measurements that ask for no reduced storage)
        dict(name="solve_f64_8x8x8x16_ns8", kind="solve", lx=8, ly=8, lz=8, lt=16, ns=8, masses="0.1", prec="f64",
             links="f32", tbc=True),
        # one column of a valence propagator: D x = b through the Schur system
        dict(name="propagator_f16_8x8x8x16_ns16", kind="propagator", lx=8, ly=8, lz=8, lt=16, ns=16, mq=0.04,
             prec="f16", tbc=True),
        # a burst of served requests with different masses on one resident field
        dict(name="serve_f16_8x8x8x8_ns8", kind="serve", lx=8, ly=8, lz=8, lt=8, ns=8, masses="0.01,0.05,0.2,0.5",
             nrhs=2, tbc=True),
        # gradient flow of one configuration with clover observables
        dict(name="flow_24x24x24x48", kind="flow", lx=24, ly=24, lz=24, lt=48, steps=5, every=5),
        # the inner time scale of the molecular dynamics: one gauge action and force
        dict(name="gauge_16x16x16x32", kind="gauge", lx=16, ly=16, lz=16, lt=32),
        # one molecular-dynamics step with a mass-preconditioned pair of terms
        dict(name="md_8x8x8x16_ns16", kind="md", lx=8, ly=8, lz=8, lt=16, ns=16, masses="0.1,0.5,2.6", inner=2,
             prec="f16"),
    ]


def _sites(c):
    return c["lx"] * c["ly"] * c["lz"] * c["lt"]


def _extents(rng, lo, hi, even=True):
    """Four extents with a volume spread over its logarithm between lo and hi sites."""
    while True:
        target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = target ** 0.25
        d = [max(2, int(round(side * rng.uniform(0.6, 1.6)))) for _ in range(4)]
        if even:
            d = [max(2, 2 * int(round(v / 2))) for v in d]
        if lo <= math.prod(d) <= hi:
            return dict(lx=d[0], ly=d[1], lz=d[2], lt=d[3])


def draw(rng):
    kind = rng.choice(["schur", "dirac", "normal", "solve", "solve", "solve", "propagator", "serve", "flow",
                       "gauge", "md"])
    mass = lambda lo, hi: round(math.exp(rng.uniform(math.log(lo), math.log(hi))), 5)  # noqa: E731
    if kind in ("schur", "dirac", "normal"):
        c = dict(kind=kind, **_extents(rng, 256, 131072), ns=rng.choice([4, 8, 16, 16, 32]), mq=mass(0.002, 0.5),
                 tbc=rng.random() < 0.7)
        if c["ns"] == 32 and _sites(c) > 65536:
            c["ns"] = 16
        if kind != "normal":
            c["dagger"] = rng.random() < 0.5
        return c
    if kind == "solve":
        prec = rng.choice(["f16", "f16", "f16", "bf16", "f32", "f64"])
        hi = 8192 if prec == "f64" else 65536
        n = rng.choice([1, 1, 2, 3]) if prec != "f64" else 1
        return dict(kind=kind, **_extents(rng, 256, hi), ns=rng.choice([8, 16]),
                    masses=",".join(str(mass(0.02, 0.5)) for _ in range(n)), prec=prec,
                    links=rng.choice(["f32", "f32", "f16"]) if prec in ("f16", "bf16") else "f32",
                    tbc=rng.random() < 0.7)
    if kind == "propagator":
        return dict(kind=kind, **_extents(rng, 256, 16384), ns=rng.choice([8, 16]), mq=mass(0.02, 0.5),
                    prec=rng.choice(["f16", "bf16"]), tbc=rng.random() < 0.7)
    if kind == "serve":
        return dict(kind=kind, **_extents(rng, 256, 8192), ns=rng.choice([8, 16]),
                    masses=",".join(str(mass(0.01, 0.5)) for _ in range(rng.choice([2, 3, 4]))),
                    nrhs=rng.choice([1, 2]), tbc=True)
    if kind == "flow":
        return dict(kind=kind, **_extents(rng, 625, 1048576, even=False), steps=rng.choice([2, 4, 6]), every=2)
    if kind == "gauge":
        return dict(kind=kind, **_extents(rng, 256, 262144))
    return dict(kind=kind, **_extents(rng, 256, 8192), ns=rng.choice([8, 16]), inner=rng.choice([1, 2]),
                masses="%s,%s" % (mass(0.05, 0.5), 2 * M0), prec="f16")


# ------------------------------------------------------------------ inputs
def _dims(c):
    return (c["lx"], c["ly"], c["lz"], c["lt"])


def _masses(c):
    return [float(m) for m in c["masses"].split(",")]


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _gaussian(shape, gen):
    return torch.view_as_complex(torch.randn(*shape, 2, dtype=torch.float64, device=DEV, generator=gen))


def _gauge_field(c, seed, eps=0.25):
    """Rough SU(3) links near the unit field: Gram-Schmidt of 1 + eps * noise, third row from the cross product."""
    lx, ly, lz, lt = _dims(c)
    a = eps * _gaussian((4, lt, lz, ly, lx, 2, 3), _gen(seed, 1))
    a[..., 0, 0] += 1.0
    a[..., 1, 1] += 1.0
    r0 = a[..., 0, :]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=-1, keepdim=True)
    r1 = a[..., 1, :]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    return torch.stack([r0, r1, torch.linalg.cross(r0, r1).conj()], dim=-2).contiguous()


def _momenta(c, seed):
    """Traceless anti-Hermitian Gaussian momenta with <p_a^2> = 1 for each of the eight generators."""
    lx, ly, lz, lt = _dims(c)
    a = _gaussian((4, lt, lz, ly, lx, 3, 3), _gen(seed, 3))
    return _ta(a) / math.sqrt(2.0)


def _even_field(c, seed, k=0):
    return _gaussian((c["ns"], _sites(c) // 2, 4, 3), _gen(seed, 10 + k))


def _full_field(c, seed):
    lx, ly, lz, lt = _dims(c)
    return _gaussian((c["ns"], lt, lz, ly, lx, 4, 3), _gen(seed, 10))


def _omega(ns):
    return odwf.odwf_zolotarev_omega(ns, LMIN, LMAX)[0]


def prepare(case, seed):
    c, k = dict(case), case["kind"]
    s = {"case": c}
    if k == "flow":
        s["U"] = _gauge_field(c, seed)
        s["out"] = torch.empty_like(s["U"])
        s["flow"] = odwf.Flow(_dims(c))
        return s
    U = _gauge_field(c, seed)
    if k == "gauge":
        s["U"], s["force"] = U, torch.empty_like(U)
        s["h"] = odwf.Handle(_dims(c), 8, M0, 0.1, _omega(8))
        return s
    if k == "serve":
        s["server"] = odwf.Server(4 << 30)
        torch.cuda.synchronize()
        s["server"].register_gauge(0, _dims(c), U, t_antiperiodic=c["tbc"])
        s["omega"] = _omega(c["ns"])
        s["b"] = [[_even_field(c, seed, 10 * i + j) for j in range(c["nrhs"])] for i in range(len(_masses(c)))]
        s["x"] = [[torch.empty_like(b) for b in bs] for bs in s["b"]]
        torch.cuda.synchronize()
        return s
    mq = c["mq"] if "mq" in c else _masses(c)[0]
    s["h"] = odwf.Handle(_dims(c), c["ns"], M0, mq, _omega(c["ns"]), t_antiperiodic=c.get("tbc", True))
    if k == "md":
        ms = _masses(c)
        s["U"], s["P"] = U, _momenta(c, seed)
        s["terms"] = [(_even_field(c, seed, i), ms[i], ms[i + 1]) for i in range(len(ms) - 1)]
        return s
    s["h"].set_gauge(U)
    if k == "solve":
        s["b"] = [_even_field(c, seed, i) for i in range(len(_masses(c)))]
    elif k in ("dirac", "propagator"):
        s["b"] = [_full_field(c, seed)]
    else:
        s["b"] = [_even_field(c, seed)]
    s["x"] = [torch.empty_like(b) for b in s["b"]]
    return s


def run(s):
    c = s["case"]
    k = c["kind"]
    if k in ("schur", "dirac"):
        mode = odwf.ODWF_MODE_SCHUR_EVEN if k == "schur" else odwf.ODWF_MODE_FULL
        op = s["h"].apply_dagger if c["dagger"] else s["h"].apply
        return op(s["x"][0], s["b"][0], mode)
    if k == "normal":
        return s["h"].apply_normal(s["x"][0], s["b"][0])
    if k == "solve":
        ms = _masses(c)
        if len(ms) == 1:
            s["h"].cg_solve(s["x"][0], s["b"][0], tol=TOL, prec=c["prec"], link_prec=c["links"], mq=ms[0])
        else:
            s["h"].cg_solve_batched(s["x"], s["b"], ms, tol=TOL, prec=c["prec"], link_prec=c["links"])
        return s["x"]
    if k == "propagator":
        s["h"].cg_solve(s["x"][0], s["b"][0], tol=TOL, prec=c["prec"], system=odwf.ODWF_SYS_FULL_DIRAC)
        return s["x"]
    if k == "serve":
        tickets = [s["server"].submit(0, c["ns"], M0, m, s["omega"], s["b"][i], s["x"][i], tol=TOL)
                   for i, m in enumerate(_masses(c))]
        for t in tickets:
            while s["server"].poll(t, 1000)[1]["status"] == 7:  # ODWF_PENDING
                pass
        return s["x"]
    if k == "flow":
        s["flow"].set_gauge(s["U"])
        obs = s["flow"].run(0.01, c["steps"], measure_every=c["every"])
        s["flow"].get_gauge(s["out"])
        return {"U": s["out"], "obs": [[o[n] for n in ("e_plaq", "e_clover", "plaq_min", "plaq_mean", "q_clover")] for o in obs]}
    if k == "gauge":
        return {"action": np.float64(s["h"].gauge_force(s["U"], BETA, s["force"])), "force": s["force"]}
    U, P = s["U"].clone(), s["P"].clone()  # the caller keeps the start for a rejected step
    h0, h1, _ = s["h"].md_trajectory(U, P, s["terms"], BETA, 0.05, 1, n_inner=c["inner"], tol=TOL, prec=c["prec"])
    return {"H": np.array([h0, h1]), "U": U, "P": P}


# ------------------------------------------------------------------ work that the path cannot do without
HOP_FLOPS = 1320 + 200  # Wilson hop on one 5D site, plus the site-local fifth-dimension operators


def _iterations(mq, tol=TOL):
    """CG iterations of S^dag S x = b: ln(2 / tol) / 2 times the square root of the condition number,
    fitted to 404, 392 and 138 iterations at m_q = 0.002, 0.04 and 0.5 (16^3 x 32 x 16, tol 1e-10)."""
    return math.log(2.0 / tol) * 17.0 / (1.0 + 3.9 * mq)


def _solve_work(c, masses, nrhs=1, storage=None):
    """Per iteration: p, r, x and the three intermediate fields read and written once, links once."""
    n5 = _sites(c) // 2 * c["ns"]
    spinor = {"f16": 52, "bf16": 52, "f32": 96, "f64": 192}[storage or c["prec"]]
    acc = 192 if (storage or c["prec"]) == "f64" else 96
    link = 144 if (storage or c["prec"]) == "f64" else 48
    it = sum(_iterations(m) for m in masses) * nrhs
    top = max(_iterations(m) for m in masses)
    return {"bytes": it * n5 * (2 * acc * 2 + 2 * spinor * 4) + top * _sites(c) * 4 * link, "flops": it * 4 * n5 * HOP_FLOPS}


def work(case):
    c, k = case, case["kind"]
    v = _sites(c)
    links = v * 4 * 144
    if k == "flow":
        # per step three stages: links read and written as 48-bit pairs (two rows), stage force carried
        return {"bytes": v * (2 * 576 + c["steps"] * 3 * (2 * 384 + 256)), "flops": v * c["steps"] * 3 * 4 * 3000.0}
    if k == "gauge":
        return {"bytes": 2 * links, "flops": v * 4 * 13 * 198.0}
    n5 = v // 2 * c["ns"]
    if k in ("schur", "normal"):
        hops = 2 if k == "schur" else 4
        return {"bytes": links + 2 * n5 * 192, "flops": hops * n5 * HOP_FLOPS}
    if k == "dirac":
        return {"bytes": links + 4 * n5 * 192, "flops": 2 * n5 * HOP_FLOPS}
    if k == "solve":
        return _solve_work(c, _masses(c))
    if k == "propagator":
        return _solve_work(c, [c["mq"]])
    if k == "serve":
        return _solve_work(c, _masses(c), c["nrhs"], "f16")
    w = _solve_work(c, _masses(c)[:-1] * 3)  # Omelyan: forces at the start, the middle and the end
    forces = 3 * (len(_masses(c)) - 1) * 4.0 * v * 4 * (672 * c["ns"] + 432)
    gauge = (4 * c["inner"] + 2) * v * 4 * 13 * 198.0
    return {"bytes": w["bytes"] + 4 * links, "flops": w["flops"] + forces + gauge}


# ------------------------------------------------------------------ the definitions in plain FP64 torch
def _dag(a):
    return a.conj().transpose(-1, -2)


def _ta(a):
    """Traceless anti-Hermitian part."""
    b = 0.5 * (a - _dag(a))
    tr = torch.diagonal(b, dim1=-2, dim2=-1).sum(-1) / 3.0
    return b - tr[..., None, None] * torch.eye(3, dtype=b.dtype, device=b.device)


class _Operator:
    """The 5D operator on parity-split fields [site][colour][spin][s], dense along s."""

    # gamma_mu = [[0, G], [G^dag, 0]], G = -i sigma_k (k = 1..3), 1: (column, phase) of each row of G and G^dag
    G = [[(1, -1j), (0, -1j)], [(1, -1), (0, 1)], [(0, -1j), (1, 1j)], [(0, 1), (1, 1)]]
    GD = [[(1, 1j), (0, 1j)], [(1, 1), (0, -1)], [(0, 1j), (1, -1j)], [(0, 1), (1, 1)]]

    def __init__(self, c, U, mq, tbc):
        self.dims, self.ns = _dims(c), c["ns"]
        lx, ly, lz, lt = self.dims
        v = lx * ly * lz * lt
        lex = torch.arange(v, device=DEV)
        x, y, z, t = lex % lx, lex // lx % ly, lex // (lx * ly) % lz, lex // (lx * ly * lz)
        par = (x + y + z + t) % 2
        self.lex = [lex[par == p] for p in (0, 1)]
        self.nbr, self.sign, self.links = [{}, {}], [{}, {}], [{}, {}]
        ext, co = (lx, ly, lz, lt), [x, y, z, t]
        stride = (1, lx, lx * ly, lx * ly * lz)
        Uf = U.reshape(4, v, 3, 3)
        for mu in range(4):
            for d in (1, -1):
                nb = lex + ((co[mu] + d) % ext[mu] - co[mu]) * stride[mu]
                edge = co[mu] == (ext[mu] - 1 if d == 1 else 0)
                sg = torch.where(edge & tbc, -1.0, 1.0) if mu == 3 else torch.ones_like(lex, dtype=torch.float64)
                for p in (0, 1):
                    sel = self.lex[p]
                    self.nbr[p][mu, d] = nb[sel] // 2
                    u = Uf[mu][sel] if d == 1 else _dag(Uf[mu][nb[sel]])
                    self.links[p][mu, d] = (u * sg[sel].to(u.dtype)[:, None, None]).contiguous()
        w = torch.as_tensor(_omega(self.ns), device=DEV)
        r = mq / (2.0 * M0)
        eye = torch.eye(self.ns, dtype=torch.float64, device=DEV)
        up = torch.roll(eye, 1, 0)
        up[0] *= -r
        dn = torch.roll(eye, -1, 0)
        dn[-1] *= -r
        W = torch.diag(w)
        self.B = [W + W @ s for s in (up, dn)]
        self.M = [(4.0 - M0) * b + eye - s for b, s in zip(self.B, (up, dn))]
        self.Mi = [torch.linalg.inv(m) for m in self.M]

    def s_op(self, mats, a, dag=False):
        """One matrix along s per chirality."""
        m = [(x if dag else x.T).to(a.dtype) for x in mats]
        return torch.cat([a[:, :, :2] @ m[0], a[:, :, 2:] @ m[1]], dim=2)

    def hop(self, a, p, dag=False):
        """W a (or W^dag a) on the sites of parity p."""
        y = torch.zeros((len(self.lex[p]), 3, 4, self.ns), dtype=a.dtype, device=DEV)
        for (mu, d), nb in self.nbr[p].items():
            sg = -d if not dag else d
            n = a[nb]
            h = torch.stack([n[:, :, i] + (sg * ph) * n[:, :, 2 + j] for i, (j, ph) in enumerate(self.G[mu])], dim=2)
            h = (self.links[p][mu, d] @ h.reshape(len(nb), 3, 2 * self.ns)).reshape(h.shape)
            y[:, :, :2] += h
            for i, (j, ph) in enumerate(self.GD[mu]):
                y[:, :, 2 + i] += (sg * ph) * h[:, :, j]
        return y

    def H(self, a, p):
        return -0.5 * self.hop(self.s_op(self.B, a), p)

    def Hd(self, a, p):
        return -0.5 * self.s_op(self.B, self.hop(a, p, dag=True), dag=True)

    def S(self, a):
        return a - self.s_op(self.Mi, self.H(self.s_op(self.Mi, self.H(a, 1)), 0))

    def Sd(self, a):
        a1 = self.s_op(self.Mi, a, dag=True)
        return a - self.Hd(self.s_op(self.Mi, self.Hd(a1, 1), dag=True), 0)

    def cg(self, b, tol=1e-14):
        x, r = torch.zeros_like(b), b.clone()
        p, rr = r.clone(), (r.abs() ** 2).sum()
        stop = tol * tol * float(rr)
        for i in range(4000):
            q = self.S(p)
            alpha = rr / (q.abs() ** 2).sum()
            x += alpha * p
            r -= alpha * self.Sd(q)
            new = (r.abs() ** 2).sum()
            p = r + (new / rr) * p
            rr = new
            if i % 10 == 9 and float(rr) < stop:
                break
        return x

    # external layouts: SCHUR_EVEN [s][site][spin][colour]; FULL [s][t][z][y][x][spin][colour]
    @staticmethod
    def load(f):
        return f.permute(1, 3, 2, 0).contiguous()

    @staticmethod
    def store(f):
        return f.permute(3, 0, 2, 1).contiguous()

    def split(self, f):
        f = f.reshape(self.ns, -1, 4, 3)
        return [self.load(f[:, lex]) for lex in self.lex]

    def join(self, e, o):
        f = torch.empty((self.ns, len(self.lex[0]) * 2, 4, 3), dtype=e.dtype, device=DEV)
        f[:, self.lex[0]], f[:, self.lex[1]] = self.store(e), self.store(o)
        lx, ly, lz, lt = self.dims
        return f.reshape(self.ns, lt, lz, ly, lx, 4, 3)


def _shift(U, mu, d):
    """U(x + d mu) of a [t][z][y][x]... field."""
    return torch.roll(U, -d, 3 - mu)


def _plaquette(U, m, n):
    return U[m] @ _shift(U[n], m, 1) @ _dag(_shift(U[m], n, 1)) @ _dag(U[n])


def _staples(U, m):
    """Sum over the six staples, so that U_m S_m is the sum of the plaquette loops through the link."""
    S = torch.zeros_like(U[m])
    for n in range(4):
        if n != m:
            S += _shift(U[n], m, 1) @ _dag(_shift(U[m], n, 1)) @ _dag(U[n])
            S += _shift(_dag(_shift(U[n], m, 1)) @ _dag(U[m]) @ U[n], n, -1)
    return S


def _loop_force(U):
    return torch.stack([_ta(U[m] @ _staples(U, m)) for m in range(4)])


def _plaq_re(U):
    return torch.stack([torch.diagonal(_plaquette(U, m, n), dim1=-2, dim2=-1).sum(-1).real
                        for m in range(4) for n in range(m + 1, 4)])


def _gauge_action(U):
    return BETA * float((1.0 - _plaq_re(U) / 3.0).sum())


def _expm_times(X, U):
    y = U.clone()
    for k in range(18, 0, -1):
        y = U + X @ y / k
    return y


def _trace(a, b):
    return float(torch.einsum("...ab,...ba->...", a, b).real.sum())


def _clover(U):
    """Site average of the clover energy and the total clover charge."""
    F, e = {}, 0.0
    for m in range(4):
        for n in range(m + 1, 4):
            q = _plaquette(U, m, n)
            um, un = _shift(U[m], m, -1), _shift(U[n], n, -1)                # U_m(x - m), U_n(x - n)
            q = q + U[n] @ _dag(_shift(um, n, 1)) @ _dag(_shift(U[n], m, -1)) @ um
            q = q + _dag(um) @ _dag(_shift(un, m, -1)) @ _shift(um, n, -1) @ un
            q = q + _dag(un) @ _shift(U[m], n, -1) @ _shift(un, m, 1) @ _dag(U[m])
            F[m, n] = _ta(q) / 4.0  # i F
            e -= _trace(F[m, n], F[m, n])
    charge = -(_trace(F[0, 1], F[2, 3]) - _trace(F[0, 2], F[1, 3]) + _trace(F[0, 3], F[1, 2])) / (4.0 * math.pi ** 2)
    return e / U[0, ..., 0, 0].numel(), charge


def _flow_obs(U):
    re = _plaq_re(U)
    n = U[0, ..., 0, 0].numel()
    e, charge = _clover(U)
    return [2.0 * float((3.0 - re).sum()) / n, e, float(re.min()) / 3.0, float(re.mean()) / 3.0, charge]


def _pf_terms(c, U, terms):
    """Action and force of the pseudofermion terms: S = phi^dag S2^dag (S1^dag S1)^-1 S2 phi.  With X the solution
    held fixed, dS = d(2 Re <X, S2 phi> - |S1 X|^2), differentiated by torch along U -> exp(eps T) U."""
    action, force = 0.0, torch.zeros_like(U)
    for phi, m1, m2 in terms:
        f = _Operator.load(phi)
        psi = _Operator(c, U, m2, True).S(f)
        one = _Operator(c, U, m1, True)
        X = one.cg(psi)
        action += float((one.S(X).abs() ** 2).sum())
        V = U.clone().requires_grad_(True)
        a, b = _Operator(c, V, m1, True), _Operator(c, V, m2, True)
        g = 2.0 * (X.conj() * b.S(f)).sum().real - (a.S(X).abs() ** 2).sum()
        (grad,) = torch.autograd.grad(g, V)
        # dg = Re sum conj(grad) dU with dU = T U: tr(T Pi) for Pi = ta(U grad^dag)
        force += _ta(U @ _dag(grad))
    return action, force


def _exact_md(c, s):
    U, P, h, inner = s["U"].clone(), s["P"].clone(), 0.05, c["inner"]

    def kick_gauge(e):
        return -BETA / 3.0 * _loop_force(U) * e

    def energy(pf):
        return pf - float(torch.einsum("...ab,...ba->...", P, P).real.sum()) + _gauge_action(U)

    a0, F = _pf_terms(c, U, s["terms"])
    H = [energy(a0)]
    P = P + 0.5 * LAMBDA * h * F
    for half in (0, 1):
        d = 0.5 * h / inner
        for _ in range(inner):
            P = P + kick_gauge(0.5 * LAMBDA * d)
            U = _expm_times(0.5 * d * P, U)
            P = P + kick_gauge(0.5 * (1.0 - 2.0 * LAMBDA) * d)
            U = _expm_times(0.5 * d * P, U)
            P = P + kick_gauge(0.5 * LAMBDA * d)
        a, F = _pf_terms(c, U, s["terms"])
        P = P + 0.5 * h * (LAMBDA if half else 1.0 - 2.0 * LAMBDA) * F
    H.append(energy(a))
    return {"H": np.array(H), "U": U, "P": P}


def exact(case, seed):
    c, k = dict(case), case["kind"]
    v = _sites(c)
    if k == "flow":
        if v * c["steps"] > 4000000:
            return None
        U, obs = _gauge_field(c, seed), []
        for i in range(c["steps"]):
            if i % c["every"] == 0:
                obs.append(_flow_obs(U))
            z0 = -0.01 * _loop_force(U)
            U = _expm_times(z0 / 4.0, U)
            z1 = -0.01 * _loop_force(U)
            U = _expm_times(8.0 / 9.0 * z1 - 17.0 / 36.0 * z0, U)
            U = _expm_times(-0.75 * 0.01 * _loop_force(U) - 8.0 / 9.0 * z1 + 17.0 / 36.0 * z0, U)
        if c["steps"] % c["every"] == 0:
            obs.append(_flow_obs(U))
        return {"U": U, "obs": obs}
    U = _gauge_field(c, seed)
    if k == "gauge":
        return {"action": np.float64(_gauge_action(U)), "force": -BETA / 3.0 * _loop_force(U)}
    if k == "md":
        if v * c["ns"] > 150000:
            return None
        ms = _masses(c)
        return _exact_md(c, {"U": U, "P": _momenta(c, seed),
                             "terms": [(_even_field(c, seed, i), ms[i], ms[i + 1]) for i in range(len(ms) - 1)]})
    if k in ("solve", "propagator", "serve") and v * c["ns"] > 700000:
        return None
    if k == "solve":
        return [_Operator.store(_Operator(c, U, m, c["tbc"]).cg(_Operator.load(_even_field(c, seed, i))))
                for i, m in enumerate(_masses(c))]
    if k == "serve":
        ops = [_Operator(c, U, m, c["tbc"]) for m in _masses(c)]
        return [[_Operator.store(op.cg(_Operator.load(_even_field(c, seed, 10 * i + j)))) for j in range(c["nrhs"])]
                for i, op in enumerate(ops)]
    op = _Operator(c, U, c["mq"], c["tbc"])
    if k == "propagator":
        e, o = op.split(_full_field(c, seed))
        be = op.s_op(op.Mi, e - op.H(op.s_op(op.Mi, o), 0))
        xe = op.cg(op.Sd(be))
        return [op.join(xe, op.s_op(op.Mi, o - op.H(xe, 1)))]
    if k == "dirac":
        e, o = op.split(_full_field(c, seed))
        if c["dagger"]:
            return op.join(op.s_op(op.M, e, dag=True) + op.Hd(o, 0), op.s_op(op.M, o, dag=True) + op.Hd(e, 1))
        return op.join(op.s_op(op.M, e) + op.H(o, 0), op.s_op(op.M, o) + op.H(e, 1))
    a = op.load(_even_field(c, seed))
    if k == "normal":
        return op.store(op.Sd(op.S(a)))
    return op.store(op.Sd(a) if c["dagger"] else op.S(a))
