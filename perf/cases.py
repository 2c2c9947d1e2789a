"""Performance cases of the library's public entry points (paper_0710_3612_gb300.mg).

``listed()`` are the calls a user of the solver makes, at the sizes of the
repository's workloads (32^2 .. 1024^2 lattices, 1 .. 64 right-hand sides, 8 or
12 vectors per chirality); ``draw(rng)`` gives more of the same ranges.  Every
case has a ``kind``:

* ``A``         the fused fine operator A = D^dagger D (outer CG: FP64; smoother: FP32);
* ``coarse``    the Galerkin coarse operator on one coarse level;
* ``transfer``  restriction and prolongation between the first two levels;
* ``vcycle``    one V-cycle, the preconditioner;
* ``coarsest``  the dense coarsest-level solve;
* ``setup``     the adaptive set-up of a hierarchy on a new gauge field;
* ``remass``    moving a hierarchy to another mass;
* ``solve``     MG-CG on one or many right-hand sides to a true FP64 residual.

``exact`` recomputes each result in complex128 with plain torch operations (the
method's own formulas: explicit stencil blocks, block Gram-Schmidt, Galerkin
products, dense coarsest factorisation, conjugate gradients).
"""
import math

import torch

from paper_0710_3612_gb300 import mg

DEV = "cuda:0"
C128, C64 = torch.complex128, torch.complex64
PREC = {"f64": mg.PREC_F64, "f32": mg.PREC_F32, "bf16": mg.PREC_BF16}
SOLVER = {"mixed": mg.SOLVER_MGCG_MIXED, "fp64": mg.SOLVER_MGCG_FP64}


# --------------------------------------------------------------------------- cases
def listed():
    return [
        # one residual or search-direction product of a single 128^2 solve: launch latency
        dict(name="A f64 128x128 x1", kind="A", Lx=128, Lt=128, beta=6.0, mass=-2.0, nrhs=1, prec="f64"),
        # A p of the batched FP64 outer iteration, 64 sources on 256^2
        dict(name="A f64 256x256 x64", kind="A", Lx=256, Lt=256, beta=10.0, mass=-2.0, nrhs=64, prec="f64"),
        # a lattice that no tile divides, a handful of sources
        dict(name="A f64 210x90 x12", kind="A", Lx=210, Lt=90, beta=6.0, mass=0.0, nrhs=12, prec="f64"),
        # the smoother's operator on the largest lattice, 16 sources
        dict(name="A f32 1024x1024 x16", kind="A", Lx=1024, Lt=1024, beta=10.0, mass=-2.0, nrhs=16, prec="f32"),
        # level 2 of the batched V-cycle: 64 sources against every coarse block
        dict(name="coarse bf16 256x256 x64", kind="coarse", Lx=256, Lt=256, Nv=8, beta=10.0, mass=-2.0, nrhs=64,
             prec="bf16"),
        # both transfers of the batched V-cycle's finest level
        dict(name="transfer f32 256x256 x64", kind="transfer", Lx=256, Lt=256, Nv=8, beta=10.0, mass=-2.0, nrhs=64,
             prec="f32"),
        # the preconditioner of a single mixed solve on a ragged lattice
        dict(name="vcycle f32 144x96", kind="vcycle", Lx=144, Lt=96, Nv=8, beta=6.0, mass=-2.0, prec="f32"),
        # the coarsest level of the 128^2 workload: 4096 unknowns, refined in FP64
        dict(name="coarsest 128x128", kind="coarsest", Lx=128, Lt=128, Nv=8, beta=6.0, mass=-2.0),
        # a new 128^2 configuration: relaxation, vectors, Galerkin operators, inverse
        dict(name="setup 128x128", kind="setup", Lx=128, Lt=128, Nv=8, beta=6.0, mass=-2.0),
        # the mass sweep on one configuration
        dict(name="remass 128x128", kind="remass", Lx=128, Lt=128, Nv=8, beta=6.0, mass=-2.0, to=-0.05),
        # one source near the critical mass, plain FP64-residual mixed MG-CG
        dict(name="solve mixed 128x128 x1", kind="solve", Lx=128, Lt=128, Nv=8, beta=6.0, mass=-2.0, nrhs=1,
             solver="mixed", tol=1e-12),
        # 64 sources of one configuration in one Krylov loop
        dict(name="solve mixed 256x256 x64", kind="solve", Lx=256, Lt=256, Nv=8, beta=10.0, mass=-2.0, nrhs=64,
             solver="mixed", tol=1e-12),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _fits(c):
    """A drawn case costs no more than the largest listed one of its kind."""
    V, r = c["Lx"] * c["Lt"], c.get("nrhs", 1)
    most = {"A": 1 << 24, "coarse": 1 << 22, "transfer": 1 << 22, "vcycle": 1 << 17, "coarsest": 1 << 17,
            "setup": 1 << 17, "remass": 1 << 17, "solve": 1 << 19 if c.get("solver") == "fp64" else 1 << 22}
    return V * r <= most[c["kind"]] and (c["kind"] == "A" or _unknowns(c) <= 4096)


def draw(rng):
    while True:
        kind = rng.choice(["A", "A", "A", "coarse", "coarse", "transfer", "transfer", "vcycle", "coarsest", "setup",
                           "remass", "solve", "solve"])
        if kind == "A":
            ext = [2 * round(_log_uniform(rng, 16, 1024) / 2) for _ in range(2)]
        else:
            ext = [8 * max(4, round(_log_uniform(rng, 32, 256) / 8)) for _ in range(2)]
        beta = rng.choice([3.0, 6.0, 10.0])
        c = dict(kind=kind, Lx=ext[0], Lt=ext[1], beta=beta, mass=rng.choice([-2.0, -1.95, -1.9, 0.0, 0.05]))
        if kind != "A":
            c["Nv"] = rng.choice([4, 8, 8, 8, 12])
        if kind in ("A", "coarse", "transfer", "solve"):
            c["nrhs"] = max(1, min(64, round(_log_uniform(rng, 1, 64))))
        if kind in ("A", "transfer", "vcycle"):
            c["prec"] = rng.choice(["f64", "f32"])
        if kind == "coarse":
            c["prec"] = rng.choice(["f64", "f32", "bf16", "bf16"])
        if kind == "remass":
            c["to"] = rng.choice([-0.05, 0.0, 0.1])
        if kind == "solve":
            c["solver"], c["tol"] = rng.choice(["mixed", "mixed", "mixed", "fp64"]), 1e-12
        if _fits(c):
            return c


# ------------------------------------------------------------------------- inputs
def _blocking(c):
    """4 x 4 blocks, then 2 x 2 down to at most 4096 coarsest unknowns."""
    if c["kind"] == "A":
        return [], []
    lx, lt, n = c["Lx"] // 4, c["Lt"] // 4, 2 * c["Nv"]
    blocks = [(4, 4)]
    while len(blocks) < 4 and lx % 2 == 0 and lt % 2 == 0 and min(lx, lt) >= 8 and (len(blocks) < 2 or lx * lt * n > 4096):
        lx, lt = lx // 2, lt // 2
        blocks.append((2, 2))
    return blocks, [c["Nv"]] * len(blocks)


def _shapes(c):
    """(Lt, Lx, dof) of every level."""
    out = [(c["Lt"], c["Lx"], 2)]
    for (bx, bt), nv in zip(*_blocking(c)):
        out.append((out[-1][0] // bt, out[-1][1] // bx, 2 * nv))
    return out


def _unknowns(c):
    return math.prod(_shapes(c)[-1])


def _gen(seed, k):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + k)
    return g


def _gauss(shape, seed, k, dtype=C128):
    """Complex Gaussian entries, E|z|^2 = 1."""
    g = _gen(seed, k)
    re = torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)
    im = torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)
    return (torch.complex(re, im) * math.sqrt(0.5)).to(dtype)


def _gauge(c, seed):
    """Quenched U(1) links [2][Lt][Lx] at coupling beta: in two dimensions the
    plaquette angles are independent (Gaussian of variance 1 / beta here), so the
    t links are their running sum along x; then a random gauge rotation."""
    Lx, Lt = c["Lx"], c["Lt"]
    g = _gen(seed, 1)
    plaq = torch.randn((Lt, Lx), generator=g, device=DEV, dtype=torch.float64) / math.sqrt(c["beta"])
    plaq -= plaq.mean(dim=1, keepdim=True)                 # no net flux through a row
    th_t = torch.cumsum(plaq, dim=1) - plaq
    om = 2 * math.pi * torch.rand((Lt, Lx), generator=g, device=DEV, dtype=torch.float64)
    th = torch.stack([torch.roll(om, -1, 1) - om, th_t + torch.roll(om, -1, 0) - om])
    return torch.polar(torch.ones_like(th), th).contiguous()


def _noise(c, seed):
    """The set-up's random starts (per level: Nv relaxation starts, power start, smoother start)."""
    sh = _shapes(c)
    total = sum((nv + 2) * math.prod(s) for s, nv in zip(sh[:-1], _blocking(c)[1]))
    return _gauss((total,), seed, 2) if total else None


def _vectors(c, seed):
    """The vectors a case works on, in its precision."""
    sh, k = _shapes(c), c["kind"]
    dt = C128 if c.get("prec", "f64") == "f64" else C64
    if k == "A":
        return {"x": _gauss((c["nrhs"],) + sh[0], seed, 3, dt)}
    if k == "coarse":
        return {"x": _gauss((c["nrhs"],) + sh[1], seed, 3, dt)}
    if k == "transfer":
        return {"f": _gauss((c["nrhs"],) + sh[0], seed, 3, dt), "c": _gauss((c["nrhs"],) + sh[1], seed, 4, dt)}
    if k == "vcycle":
        return {"x": _gauss(sh[0], seed, 3, dt)}
    if k in ("coarsest", "remass"):
        return {"x": _gauss(sh[-1], seed, 3)}
    if k == "solve":
        return {"x": _gauss((c["nrhs"],) + sh[0], seed, 3)}
    return {}


def prepare(case, seed):
    U, noise = _gauge(case, seed), _noise(case, seed)
    blocks, Nv = _blocking(case)
    st = {"case": case, "U": U, "noise": noise, "blocks": blocks, "Nv": Nv, **_vectors(case, seed)}
    if case["kind"] != "setup":
        more = {"max_rhs": case["nrhs"]} if case["kind"] == "solve" else {}
        st["mg"] = mg.Multigrid(U, case["mass"], blocks, Nv, noise, **more)
    if case["kind"] == "solve":                              # the source b = D^dagger chi
        st["b"] = torch.empty_like(st["x"])
        mg.mg_apply_D(st["mg"].h, st["x"], st["b"], case["nrhs"], True, mg.PREC_F64)
    elif case["kind"] == "transfer":
        st["fout"], st["cout"] = torch.empty_like(st["f"]), torch.empty_like(st["c"])
    elif "x" in st:
        st["y"] = torch.empty_like(st["x"])
    return st


def run(st):
    c = st["case"]
    k, h = c["kind"], st["mg"].h if "mg" in st else None
    if k == "A":
        mg.mg_apply_A(h, st["x"], st["y"], c["nrhs"], PREC[c["prec"]])
        return st["y"]
    if k == "coarse":
        mg.mg_apply_coarse(h, 2, st["x"], st["y"], c["nrhs"], PREC[c["prec"]])
        return st["y"]
    if k == "transfer":
        mg.mg_restrict(h, 1, st["f"], st["cout"], c["nrhs"], PREC[c["prec"]])
        mg.mg_prolong(h, 1, st["c"], st["fout"], c["nrhs"], PREC[c["prec"]])
        return st["cout"], st["fout"]
    if k == "vcycle":
        mg.mg_vcycle(h, st["x"], st["y"], PREC[c["prec"]])
        return st["y"]
    if k == "coarsest":
        mg.mg_coarsest_solve(h, st["x"], st["y"])
        return st["y"]
    if k == "setup":
        with mg.Multigrid(st["U"], c["mass"], st["blocks"], st["Nv"], st["noise"]) as s:
            return _hierarchy(s, c, vectors=True)
    if k == "remass":
        st["mg"].set_mass(c["to"])
        mg.mg_coarsest_solve(h, st["x"], st["y"])
        out = _hierarchy(st["mg"], c, vectors=False)
        out["coarsest"] = st["y"]
        return out
    x, _ = st["mg"].solve(st["b"], tol=c["tol"], solver=SOLVER[c["solver"]])
    return x


def _hierarchy(s, c, vectors):
    """The parts of a hierarchy that a user reads back."""
    out, sh = {}, _shapes(c)
    for l in range(1, len(sh)):
        lt, lx, n = sh[l]
        out["op%d" % (l + 1)] = torch.empty((lt, lx, 9, n, n), dtype=C128, device=DEV)
        mg.mg_get_coarse_op(s.h, l + 1, out["op%d" % (l + 1)])
        out["smoother%d" % l] = list(mg.mg_get_smoother(s.h, l))
        if vectors:
            out["vectors%d" % l] = torch.empty((n // 2,) + sh[l - 1], dtype=C128, device=DEV)
            mg.mg_get_null_vectors(s.h, l, out["vectors%d" % l])
    return out


# --------------------------------------------------------------------------- work
def work(case):
    """Bytes with every input read once and every output written once, and the
    multiply-adds of the formulas (2 flops each; a complex product 8)."""
    sh, k, r = _shapes(case), case["kind"], case.get("nrhs", 1)
    V = case["Lx"] * case["Lt"]
    rs = 8 if case.get("prec", "f64") == "f64" else 4       # bytes of a real number
    siz = [math.prod(s) for s in sh]
    blk = [s[0] * s[1] * 9 * s[2] ** 2 for s in sh]         # complex entries of a level's operator
    if k == "A":
        return {"bytes": 2 * rs * (4 * V * r + 2 * V), "flops": 2 * 56 * V * r}
    if k == "coarse":
        return {"bytes": blk[1] * {"f64": 16, "f32": 8, "bf16": 4}[case["prec"]] + 2 * siz[1] * r * 2 * rs,
                "flops": 8 * blk[1] * r}
    if k == "transfer":
        P = V * 2 * case["Nv"]
        return {"bytes": 2 * 2 * rs * (P + r * (siz[0] + siz[1])), "flops": 2 * 8 * P * r}
    N = siz[-1]
    P = [s * nv for s, nv in zip(siz, _blocking(case)[1])]
    cyc_b, cyc_f = 0, 0                                      # one V-cycle of the FP32 preconditioner
    for l in range(len(sh) - 1):
        op = 2 * V * 8 if l == 0 else blk[l] * 4
        cyc_b += 4 * op + 2 * 8 * P[l] + r * 8 * 10 * siz[l]
        cyc_f += r * (4 * (112 * V if l == 0 else 8 * blk[l]) + 2 * 8 * P[l])
    cyc_b, cyc_f = cyc_b + 4 * N * N, cyc_f + 8 * N * N * r
    if k == "vcycle":
        return {"bytes": cyc_b * (rs // 4), "flops": cyc_f}
    if k == "coarsest":
        return {"bytes": 4 * N * N + 32 * N, "flops": 8 * N * N}
    ops = sum(16 * b for b in blk[1:])
    gal = sum(8 * 9 * p * 2 * nv for p, nv in zip(P, _blocking(case)[1]))   # Galerkin products
    inv = 4 * N ** 3                                                        # Hermitian inverse
    if k == "remass":
        return {"bytes": 4 * ops, "flops": inv + 4 * ops / 16}
    if k == "setup":
        relax = sum((8 * nv + 34) * (112 * V if l == 0 else 8 * blk[l]) for l, nv in enumerate(_blocking(case)[1]))
        return {"bytes": 32 * V + sum(16 * (nv + 2) * s + 16 * p for nv, s, p in zip(_blocking(case)[1], siz, P)) + ops,
                "flops": relax + gal + inv}
    its = 10 if case["mass"] > -1.0 else 50 if case["mass"] > -1.97 else 150
    return {"bytes": its * (cyc_b + r * 16 * 12 * siz[0] + 32 * V), "flops": its * (cyc_f + r * (112 * V + 30 * siz[0]))}


# -------------------------------------------------------------------------- exact
DISP = [(dx, dt) for dt in (-1, 0, 1) for dx in (-1, 0, 1)]  # the order of the coarse operators' blocks


def _shift(x, dx, dt, dims):
    """x(j + (dx, dt)) on the periodic lattice; dims = (t axis, x axis)."""
    return torch.roll(x, (-dt, -dx), dims)


class _Exact:
    """The method in complex128: every level's operator as 9-point stencil blocks
    [Lt][Lx][9][n][n], P as per-site matrices [Lt][Lx][n][2 Nv]."""

    def __init__(self, c, seed, mass):
        self.c, self.U, self.noise = c, _gauge(c, seed), _noise(c, seed)
        self.blocks, self.Nv = _blocking(c)
        self.P = []
        self.ops = [self.fine(mass)]

    def fine(self, mass):
        """A = D^dagger D as stencil blocks."""
        Lt, Lx = self.c["Lt"], self.c["Lx"]
        ux, ut = self.U[0], self.U[1].clone()
        ut[Lt - 1] *= -1                                     # antiperiodic in t
        one = torch.eye(2, dtype=C128, device=DEV)
        s1 = torch.tensor([[0, 1], [1, 0]], dtype=C128, device=DEV)
        s2 = torch.tensor([[0, -1j], [1j, 0]], dtype=C128, device=DEV)

        def hops(sign):
            out = {(0, 0): ((4.0 + mass) * one).expand(Lt, Lx, 2, 2)}
            for (e, u, s) in (((1, 0), ux, s1), ((0, 1), ut, s2)):
                back = torch.roll(u, (e[1], e[0]), (0, 1)).conj()
                out[e] = -0.5 * u[..., None, None] * (one - sign * s)
                out[(-e[0], -e[1])] = -0.5 * back[..., None, None] * (one + sign * s)
            return out

        D, Dd = hops(1), hops(-1)
        A = torch.zeros((Lt, Lx, 9, 2, 2), dtype=C128, device=DEV)
        for e1, m1 in Dd.items():
            for e2, m2 in D.items():
                d = (e1[0] + e2[0], e1[1] + e2[1])
                if max(abs(d[0]), abs(d[1])) < 2:            # two hops along one axis vanish
                    A[:, :, DISP.index(d)] += m1 @ _shift(m2, e1[0], e1[1], (0, 1))
        return A

    @staticmethod
    def apply(A, x):
        """(A x)(j) = sum_d A[j][d] x(j + d) on [..., Lt, Lx, n]."""
        y = torch.zeros_like(x)
        for d, (dx, dt) in enumerate(DISP):
            xs = _shift(x, dx, dt, (-3, -2))
            if x.shape[-1] == 2:                             # 2 x 2 blocks: elementwise products
                for a in (0, 1):
                    y[..., a] += A[:, :, d, a, 0] * xs[..., 0] + A[:, :, d, a, 1] * xs[..., 1]
            else:
                y += torch.einsum("txab,...txb->...txa", A[:, :, d], xs)
        return y

    def level(self, l):
        """Relaxed, block-orthonormalised vectors of level l and its smoother data."""
        A, (Lt, Lx, n), nv, (bx, bt) = self.ops[l], _shapes(self.c)[l], self.Nv[l], self.blocks[l]
        pos = sum((v + 2) * math.prod(s) for s, v in zip(_shapes(self.c)[:l], self.Nv[:l]))
        z = self.noise[pos:pos + (nv + 2) * Lt * Lx * n].reshape(nv + 2, Lt, Lx, n)
        v = z[nv] / z[nv].norm()
        for _ in range(30):
            w = self.apply(A, v)
            lam = torch.sum(v.conj() * w).real.item()
            v = w / w.norm()
        e = z[:nv].clone()
        for _ in range(8):
            e = e - self.apply(A, e) / lam
        h = n // 2
        q = e.reshape(nv, Lt // bt, bt, Lx // bx, bx, 2, h).permute(1, 3, 5, 0, 2, 4, 6)
        q = q.reshape(Lt // bt, Lx // bx, 2, nv, bt * bx * h).clone()
        for k in range(nv):
            u = q[..., k, :]
            for _ in range(2):
                for j in range(k):
                    u = u - torch.sum(q[..., j, :].conj() * u, -1, keepdim=True) * q[..., j, :]
            q[..., k, :] = u / u.norm(dim=-1, keepdim=True)
        q = q.reshape(Lt // bt, Lx // bx, 2, nv, bt, bx, h).permute(3, 0, 4, 1, 5, 2, 6).reshape(nv, Lt, Lx, n)
        P = torch.zeros((Lt, Lx, n, 2 * nv), dtype=C128, device=DEV)
        for s in (0, 1):
            P[:, :, s * h:(s + 1) * h, s * nv:(s + 1) * nv] = q[..., s * h:(s + 1) * h].permute(1, 2, 3, 0)
        return P, q, lam

    def galerkin(self, A, P, bx, bt):
        Lt, Lx, n, m = P.shape
        out = torch.zeros((Lt // bt, Lx // bx, 9, m, m), dtype=C128, device=DEV)
        PH = P.conj().transpose(-1, -2)
        for d, (dx, dt) in enumerate(DISP):
            G = PH @ (A[:, :, d] @ _shift(P, dx, dt, (0, 1)))
            G = G.reshape(Lt // bt, bt, Lx // bx, bx, m, m)
            for ot in range(bt):
                for ox in range(bx):
                    out[:, :, ((ox + dx) // bx + 1) + 3 * ((ot + dt) // bt + 1)] += G[:, ot, :, ox]
        return out

    def build(self, levels):
        """Vectors and operators of the first `levels` coarsenings."""
        self.q, self.lam = [], []
        for l in range(levels):
            P, q, lam = self.level(l)
            self.P.append(P)
            self.q.append(q)
            self.lam.append(lam)
            self.ops.append(self.galerkin(self.ops[l], P, *self.blocks[l]))
        return self

    def at(self, mass):
        """The same vectors at another mass."""
        self.ops = [self.fine(mass)]
        for P, b in zip(self.P, self.blocks):
            self.ops.append(self.galerkin(self.ops[-1], P, *b))
        return self

    def smoother(self, l):
        sh, nv = _shapes(self.c), self.Nv[l]
        pos = sum((v + 2) * math.prod(s) for s, v in zip(sh[:l], self.Nv[:l])) + (nv + 1) * math.prod(sh[l])
        r, a = self.noise[pos:pos + math.prod(sh[l])].reshape(sh[l]), []
        for _ in range(2):
            q = self.apply(self.ops[l], r)
            a.append((torch.sum(q.conj() * r).real / torch.sum(q.conj() * q).real).item())
            r = r - 0.8 * a[-1] * q
        return 0.8 * (a[0] + a[1]), -0.64 * a[0] * a[1]

    def restrict(self, l, f):
        bx, bt = self.blocks[l]
        y = torch.einsum("txas,...txa->...txs", self.P[l].conj(), f)
        Lt, Lx, m = y.shape[-3:]
        return y.reshape(y.shape[:-3] + (Lt // bt, bt, Lx // bx, bx, m)).sum((-2, -4))

    def prolong(self, l, e):
        bx, bt = self.blocks[l]
        e = e.repeat_interleave(bt, dim=-3).repeat_interleave(bx, dim=-2)
        return torch.einsum("txas,...txs->...txa", self.P[l], e)

    def coarsest(self, b):
        A = self.ops[-1]
        Lt, Lx, _, n, _ = A.shape
        M = torch.zeros((Lt * Lx, n, Lt * Lx, n), dtype=C128, device=DEV)
        idx = torch.arange(Lt * Lx, device=DEV)
        for d, (dx, dt) in enumerate(DISP):
            nb = ((idx // Lx + dt) % Lt) * Lx + (idx % Lx + dx) % Lx
            M[idx, :, nb, :] += A[:, :, d].reshape(Lt * Lx, n, n)
        M = M.reshape(Lt * Lx * n, -1)
        x, v = torch.linalg.solve(M, b.reshape(-1)), b.reshape(-1)
        x = x + torch.linalg.solve(M, v - M @ x)
        return x.reshape(b.shape)

    def vcycle(self, b, l=0):
        if l == len(self.blocks):
            return self.coarsest(b)
        A, (c0, c1) = self.ops[l], self.smoother(l)
        x = c0 * b + c1 * self.apply(A, b)
        x = x + self.prolong(l, self.vcycle(self.restrict(l, b - self.apply(A, x)), l + 1))
        r = b - self.apply(A, x)
        return x + c0 * r + c1 * self.apply(A, r)

    def solve(self, b):
        """Conjugate gradients on A x = b for every right-hand side, restarted once from the true residual."""
        A = self.ops[0]
        x = torch.zeros_like(b)
        dot = lambda u, v: torch.sum((u.conj() * v).real, (-3, -2, -1), keepdim=True)  # noqa: E731
        for tol in (1e-10, 1e-6):
            r = b - self.apply(A, x)
            p, rr = r.clone(), dot(r, r)
            stop = rr * tol * tol
            for it in range(20000):
                q = self.apply(A, p)
                a = rr / dot(p, q).clamp_min(1e-300)
                x, r = x + a * p, r - a * q
                new = dot(r, r)
                if it % 25 == 0 and bool((new <= stop).all()):
                    break
                p, rr = r + (new / rr.clamp_min(1e-300)) * p, new
        return x


def exact(case, seed):
    k, v = case["kind"], {n: x.to(C128) for n, x in _vectors(case, seed).items()}
    h = _Exact(case, seed, case["mass"])
    if k == "A":
        if case["nrhs"] * case["Lx"] * case["Lt"] > 1 << 22:  # in parts, to stay small
            return torch.cat([h.apply(h.ops[0], x) for x in v["x"].split(4)])
        return h.apply(h.ops[0], v["x"])
    if k == "solve":
        D = lambda x: _dagger(h.U, case, x)  # noqa: E731
        return h.solve(D(v["x"]))
    n = len(h.blocks)
    if k == "coarse":
        return h.apply(h.build(1).ops[1], v["x"])
    if k == "transfer":
        h.build(1)
        return h.restrict(0, v["f"]), h.prolong(0, v["c"])
    h.build(n)
    if k == "vcycle":
        return h.vcycle(v["x"])
    if k == "coarsest":
        return h.coarsest(v["x"])
    if k == "remass":
        h.at(case["to"])
    out = {}
    for l in range(1, n + 1):
        out["op%d" % (l + 1)] = h.ops[l]
        out["smoother%d" % l] = [*h.smoother(l - 1), h.lam[l - 1], 1.0 / h.lam[l - 1]]
        if k == "setup":
            out["vectors%d" % l] = h.q[l - 1]
    if k == "remass":
        out["coarsest"] = h.coarsest(v["x"])
    return out


def _dagger(U, c, x):
    """D^dagger x by shifted products (Sec. 1 with the projectors exchanged)."""
    ux, ut = U[0], U[1].clone()
    ut[c["Lt"] - 1] *= -1
    y = (4.0 + c["mass"]) * x
    xf = ux * _shift(x, 1, 0, (-3, -2)).movedim(-1, 0)
    xb = _shift((ux.conj() * x.movedim(-1, 0)).movedim(0, -1), -1, 0, (-3, -2)).movedim(-1, 0)
    tf = ut * _shift(x, 0, 1, (-3, -2)).movedim(-1, 0)
    tb = _shift((ut.conj() * x.movedim(-1, 0)).movedim(0, -1), 0, -1, (-3, -2)).movedim(-1, 0)
    y[..., 0] -= 0.5 * ((xf[0] + xf[1]) + (xb[0] - xb[1]) + (tf[0] - 1j * tf[1]) + (tb[0] + 1j * tb[1]))
    y[..., 1] -= 0.5 * ((xf[1] + xf[0]) + (xb[1] - xb[0]) + (tf[1] + 1j * tf[0]) + (tb[1] - 1j * tb[0]))
    return y
