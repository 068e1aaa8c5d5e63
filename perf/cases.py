"""The work that a user of the solver has it do, as cases that can be timed and checked.

Each case is one call of the public binding (`paper_2409_01910_gb300.sgs`) on the repository's
own workloads: the planar heat transfer (16 cells on 16^3, 64 cells on 32^3), the batch of
uneven instances, the Mach-2 shock between inflow states, the lid-driven and the BGK heat
cavity, in the precisions and orders that the solver offers, with smaller and odd sizes of
the same kinds drawn at random. `exact` restates the method in 64-bit torch operations.

Initial states lie part of the way to the solution, as in most of a run: local Maxwellians of
a smooth profile between the boundary values, a heat-flux correction and seeded noise.
"""
import math

import numpy as np
import torch

from paper_2409_01910_gb300 import sgs

B0 = 1.0 / (4.0 * math.pi)
GRIDS = (8, 12, 16, 20, 24, 32)
BOX = {8: 6.0, 12: 6.0, 16: 6.0, 20: 6.0, 24: 8.0, 32: 8.0}
DEVICE = "cuda"
GAS = {"maxwell": sgs.MAXWELL, "hard": sgs.HARD_SPHERE, "bgk": sgs.BGK}


def _case(name, do, **kw):
    """A case with every field. do: the call; nx, ny (0: 1-D), instances (above 1: a handle of
    uneven 1-D instances of at most nx cells); nv^3 velocities on [-vmax, vmax]^3; the gas and
    the Knudsen number; walls or inflow; the handle's precision (mixed: FP32 sums and
    double-float scans); order; ordering of a scan; iters of a defect-correction step; terms
    of the fast operator's BF16 products; noise of the initial state."""
    c = dict(do=do, nx=16, ny=0, instances=1, nv=16, vmax=6.0, gas="maxwell", eps=0.1, inflow=False, mixed=False,
             arith="handle", order=1, ordering=0, iters=0, terms=0, noise=1e-3)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a few cells on the coarsest grid, as in a test or a coarse level
        _case("collide_8c_8v_fp64", "collide", nx=8, nv=8, eps=1.0),
        # one whole SGS iteration with its residual on the small heat problem, plain FP64
        _case("iterate_16c_16v_fp64", "iterate", nx=16, nv=16, eps=1.0),
        # the FP64 collision step of a batch member's grid, ragged cell count
        _case("collide_40c_24v_fp64", "collide", nx=40, nv=24, vmax=8.0),
        # the FP32 collision step of the shock (hard spheres between inflow states)
        _case("collide_128c_32v_fp32", "collide", nx=128, nv=32, vmax=10.0, gas="hard", inflow=True, mixed=True),
        # the high-precision evaluation of the defect correction on the heat problem
        _case("collide_64c_32v_df64", "collide", nx=64, nv=32, vmax=8.0, eps=0.01, mixed=True, arith="df64"),
        # a scan of the heat problem in the mixed solver, the step that the method is named after
        _case("scan_64c_32v_mixed", "scan", nx=64, nv=32, vmax=8.0, eps=0.01, mixed=True),
        # a backward scan of the second-order scheme in FP64, an odd number of cells
        _case("scan_45c_20v_fp64_o2", "scan", nx=45, nv=20, eps=0.1, order=2, ordering=1),
        # a scan of many uneven instances at once (one cluster per instance)
        _case("scan_batch24_24v_mixed", "scan", nx=256, instances=24, nv=24, vmax=8.0, mixed=True),
        # one ordering of the lid-driven cavity
        _case("ordering_64x64_24v_mixed", "scan", nx=64, ny=64, nv=24, vmax=6.0, eps=0.05, mixed=True, ordering=2),
        # one iteration of the BGK heat cavity (four orderings, each after a collision step)
        _case("iterate_40x40_20v_bgk", "iterate", nx=40, ny=40, nv=20, gas="bgk", eps=0.01),
        # the flagship call: a defect-correction step with two mixed iterations
        _case("dc_step_64c_32v", "dc", nx=64, nv=32, vmax=8.0, eps=0.01, mixed=True, iters=2, noise=1e-4),
        # the fast spectral operator on the tensor cores (split BF16 products)
        _case("fast_64c_32v_3terms", "fast", nx=64, nv=32, vmax=10.0, gas="hard", mixed=True, terms=3),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    do = rng.choice(["collide", "collide", "scan", "scan", "scan2d", "batch", "iterate", "dc", "fast"])
    nv = rng.choice(GRIDS)
    c = dict(nv=nv, vmax=BOX[nv], eps=math.exp(rng.uniform(math.log(1e-3), 0.0)), noise=rng.choice([1e-3, 1e-4]))
    most = {8: 256, 12: 256, 16: 200, 20: 128, 24: 96, 32: 64}[nv]
    if do == "collide":
        mixed = rng.random() < 0.6
        c.update(nx=_log_int(rng, 1, most if mixed else max(8, most // 2)), mixed=mixed,
                 gas=rng.choice(["maxwell", "hard"]), inflow=rng.random() < 0.3)
        if mixed:
            c["arith"] = rng.choice(["handle", "handle", "df64", "fp64"])
            if c["arith"] == "fp64":
                c["nx"] = min(c["nx"], max(8, most // 2))
    elif do == "scan":
        c.update(nx=_log_int(rng, 1, 128), mixed=rng.random() < 0.6, order=rng.choice([1, 1, 2]),
                 ordering=rng.choice([0, 1]), inflow=rng.random() < 0.3)
    elif do == "scan2d":
        do = "scan"
        c.update(nx=_log_int(rng, 2, 40), ny=_log_int(rng, 2, 40), mixed=rng.random() < 0.6,
                 order=rng.choice([1, 1, 2]), ordering=rng.choice([0, 1, 2, 3]))
    elif do == "batch":
        do = "scan"
        c.update(nx=_log_int(rng, 16, 200), instances=rng.randint(2, 40 if nv <= 24 else 16), mixed=rng.random() < 0.7,
                 ordering=rng.choice([0, 1]))
    elif do == "iterate":
        two = rng.random() < 0.4
        gas = "bgk" if two else rng.choice(["maxwell", "hard", "bgk"])
        c.update(nx=_log_int(rng, 3, 32 if two else max(8, most // 4)), gas=gas,
                 ny=_log_int(rng, 3, 32) if two else 0, order=rng.choice([1, 1, 2]))
    elif do == "dc":
        c.update(nx=_log_int(rng, 2, max(8, most * 3 // 4)), mixed=True, iters=rng.choice([1, 2]),
                 gas=rng.choice(["maxwell", "hard"]), inflow=rng.random() < 0.3, noise=1e-4)
    else:
        c.update(nx=_log_int(rng, 1, 64), mixed=True, gas="hard", terms=3)
    return _case("", do, **c)


# ---------------------------------------------------------------------------------------
# Inputs: the problems of a case and their initial states, from the seed alone.
# ---------------------------------------------------------------------------------------
def _problems(c, seed):
    rng = np.random.default_rng(seed)
    sizes = np.random.default_rng(c["nx"] + 1000 * c["instances"])  # of the case: the fields keep their shape
    out = []
    for q in range(c["instances"]):
        nx = c["nx"] if c["instances"] == 1 else int(sizes.integers(max(1, c["nx"] // 8), c["nx"] + 1))
        eps = c["eps"] if c["instances"] == 1 else float(np.exp(rng.uniform(np.log(1e-3), 0.0)))
        TL, TR = float(rng.uniform(0.8, 1.2)), float(rng.uniform(1.5, 2.5))
        kw = dict(nx=nx, nv=c["nv"], v_max=c["vmax"], collision=GAS[c["gas"]], eps=eps,
                  b0=1.0 if c["gas"] == "bgk" else B0, bc_T=(TL, TR), total_mass=1.0,
                  precision=sgs.FP32 if c["mixed"] else sgs.FP64, order=c["order"])
        if c["inflow"]:  # Rankine-Hugoniot states of a normal shock, Mach 1.4 .. 2 (coarse grids: weaker)
            mach = float(rng.uniform(1.4, 2.0 if c["nv"] >= 24 else 1.5))
            u1, m2 = mach * math.sqrt(5.0 / 3.0), mach * mach
            r = 8.0 / 3.0 * m2 / (2.0 / 3.0 * m2 + 2.0)
            T2 = (10.0 / 3.0 * m2 - 2.0 / 3.0) * (2.0 / 3.0 * m2 + 2.0) / ((8.0 / 3.0) ** 2 * m2)
            kw.update(bc_kind=(sgs.INFLOW, sgs.INFLOW), bc_rho=(1.0, r), bc_u=((u1, 0.0, 0.0), (u1 / r, 0.0, 0.0)),
                      bc_T=(1.0, T2), total_mass=0.0, x_lo=-0.15625 * nx, x_hi=0.15625 * nx)
        elif c["ny"] and c["gas"] == "bgk":  # heat cavity: hot top wall
            kw.update(space_dim=2, ny=c["ny"], bc_T=(1.0, 1.0), bc_T_y=(1.0, TR))
        elif c["ny"]:  # lid-driven cavity
            kw.update(space_dim=2, ny=c["ny"], bc_T=(1.0, 1.0), bc_T_y=(1.0, 1.0),
                      bc_u_y=((0.0, 0.0, 0.0), (float(rng.uniform(0.3, 0.6)), 0.0, 0.0)))
        out.append(sgs.Problem(**kw))
    return out


def _nodes(c, device):
    return (torch.arange(c["nv"], dtype=torch.float64, device=device) - c["nv"] // 2 + 1) * (2.0 * c["vmax"] / c["nv"])


def _profile(c, p, device):
    """Density, x and y velocity, temperature and heat-flux amplitude in the cells of problem p."""
    x = (torch.arange(p.nx, dtype=torch.float64, device=device) + 0.5) / p.nx
    zero = torch.zeros_like(x)
    if c["inflow"]:
        s = 0.5 * (1.0 + torch.tanh((x - 0.5) * (p.x_hi - p.x_lo)))
        rho = 1.0 + (p.bc_rho[1] - 1.0) * s
        return rho, p.bc_u[0][0] / rho, zero, 1.0 + (p.bc_T[1] - 1.0) * s, zero - 0.02
    if not c["ny"]:
        T = p.bc_T[0] + (p.bc_T[1] - p.bc_T[0]) * (0.1 + 0.8 * x)
        rho = 1.0 / T
        return rho / rho.mean(), zero, zero, T, zero - 0.1 * min(1.0, p.eps)
    y = (torch.arange(p.ny, dtype=torch.float64, device=device) + 0.5) / p.ny
    X, Y = x[None, :].expand(p.ny, p.nx).reshape(-1), y[:, None].expand(p.ny, p.nx).reshape(-1)
    T = 1.0 + (p.bc_T_y[1] - 1.0) * 0.8 * Y * torch.sin(math.pi * X)
    u = 0.4 * p.bc_u_y[1][0]
    rho = 1.0 / T
    return (rho / rho.mean(), u * torch.sin(math.pi * X) * (3.0 * Y * Y - 2.0 * Y),
            -u * torch.cos(math.pi * X) * (Y * Y * Y - Y * Y) * 2.0, T, torch.zeros_like(T) - 0.05 * min(1.0, p.eps))


def _inputs(c, seed):
    """Problems, the initial distribution and a penalty field of its size, (cells, N, N, N) each."""
    dev = torch.device(DEVICE)
    probs = _problems(c, seed)
    gen = torch.Generator(device=dev).manual_seed(seed)
    v = _nodes(c, dev)
    f, P = [], []
    for p in probs:
        rho, u1, u2, T, q = (a[:, None, None, None] for a in _profile(c, p, dev))
        c1, c2, c3 = v[None, :, None, None] - u1, v[None, None, :, None] - u2, v[None, None, None, :]
        cc = (c1 * c1 + c2 * c2 + c3 * c3) / T
        M = rho / (2.0 * math.pi * T) ** 1.5 * torch.exp(-0.5 * cc)
        noise = 2.0 * torch.rand(M.shape, dtype=torch.float64, device=dev, generator=gen) - 1.0
        d = M * (q * c1 / torch.sqrt(T) * (cc - 5.0) + c["noise"] * noise)
        f.append(M + d)
        P.append(0.3 * rho * d)
    return probs, torch.cat(f), torch.cat(P)


def prepare(case, seed):
    probs, f0, P0 = _inputs(case, seed)
    s = sgs.Solver(probs)
    st = dict(case=case, solver=s, f0=f0.reshape(-1), f=s.field(), Q=s.field(), P=s.field(),
              res=torch.zeros(len(probs), dtype=torch.float64, device=DEVICE))
    if case["do"] == "scan":
        s.collide(st["f0"], st["Q"], None)  # the collision frequency and Maxwellians that a scan reads
        st["P"].copy_(P0.reshape(-1))
    elif case["do"] == "fast":
        st["fast"] = sgs.FastOperator(s, 8, 16, chunk=8)
    return st


def run(st):
    c, s = st["case"], st["solver"]
    f, Q, P, res = st["f"], st["Q"], st["P"], st["res"]
    if c["do"] == "collide":
        prec = {"handle": None, "df64": sgs.DF64, "fp64": sgs.FP64}[c["arith"]]
        s.collide(st["f0"], Q, P, precision=prec)
        return {"Q": Q, "P": P}
    if c["do"] == "fast":
        st["fast"].collide(st["f0"], Q, terms=c["terms"])
        return {"Q": Q}
    f.copy_(st["f0"])  # the calls below update f in place
    if c["do"] == "scan":
        if c["ny"]:
            s.sweep_ordering(f, P, c["ordering"])
        elif c["ordering"] == 0:
            s.sweep_forward(f, P)
        else:
            s.sweep_backward(f, P)
        return {"f": f}
    if c["do"] == "iterate":
        s.iterate(f, Q, P, flags=sgs.IT_EVAL, res=res)
    else:
        s.dc_step(f, Q, P, c["iters"], res=res)
    return {"f": f, "Q": Q, "P": P, "res": res}


def _cells(c):
    if c["ny"]:
        return c["nx"] * c["ny"]
    return c["nx"] if c["instances"] == 1 else int(c["instances"] * 0.5625 * c["nx"])


def work(case):
    """Bytes: each field read or written once; flops: 10 per mode pair of the Hermitian half in
    the direct sum (8 of the products, 2 of the sum after the weight), 60 per node and visit in
    a scan, the separable transforms of the fast operator."""
    c = case
    K, H, cells = c["nv"] ** 3, c["nv"] // 2 - 1, _cells(c)
    field = 8.0 * K * cells
    pairs = 0.5 * (3 * H * H + 3 * H + 1) ** 3
    coll = 0.0 if c["gas"] == "bgk" else 10.0 * pairs * cells
    scan = 60.0 * K * cells
    if c["do"] == "collide":
        return {"bytes": 3 * field, "flops": coll + 30.0 * K * cells}
    if c["do"] == "scan":
        return {"bytes": 3 * field, "flops": scan}
    if c["do"] == "iterate":
        n = 4 if c["ny"] else 2
        return {"bytes": 4 * field, "flops": (n + 1) * coll + n * scan}
    if c["do"] == "dc":  # increment form: two sums a collision step
        return {"bytes": 4 * field, "flops": (1 + 4 * c["iters"]) * coll + 2 * c["iters"] * scan}
    n, P = 2 * H + 1, 32 if c["nv"] <= 16 else 48
    passes = 8.0 * (n * n * n * P + n * n * P * P) + 4.0 * n * P * P * P
    return {"bytes": 2 * field, "flops": cells * 129.0 * (2 * passes + 2.0 * P ** 3)}


# ---------------------------------------------------------------------------------------
# The method in 64-bit torch operations.
# ---------------------------------------------------------------------------------------
def _phi(v):
    """1, v1, v2, v3, |v|^2 on the grid, (5, N, N, N)."""
    a, b, d = torch.meshgrid(v, v, v, indexing="ij")
    return torch.stack([torch.ones_like(a), a, b, d, a * a + b * b + d * d])


class _Maxwellians:
    """Newton for exp(alpha + beta.v - gamma |v|^2) with given (weighted) discrete moments, batched."""

    def __init__(self, v, w):
        self.v, self.w, self.N = v, w, v.numel()
        self.pw = torch.stack([v ** p for p in range(5)])  # (5, N)

    def factors(self, th):
        v = self.v
        E = torch.exp(th[:, 1:4, None] * v - th[:, 4, None, None] * (v * v))  # (B, 3, N)
        return E, torch.exp(th[:, 0])

    def values(self, th):
        E, a = self.factors(th)
        return (a[:, None] * E[:, 0])[:, :, None, None] * E[:, 1][:, None, :, None] * E[:, 2][:, None, None, :]

    def _system(self, th, wts, target):
        E, a = self.factors(th)
        mom, A = 0.0, 0.0
        for w1, w2 in wts:  # a sum of products of 1-D weights on the first two dimensions
            S1 = torch.einsum("bi,pi->bp", E[:, 0] * w1, self.pw)
            S2 = torch.einsum("bi,pi->bp", E[:, 1] * w2, self.pw)
            S3 = torch.einsum("bi,pi->bp", E[:, 2], self.pw)

            def m(p, q, r):
                return S1[:, p] * S2[:, q] * S3[:, r]

            e = m(2, 0, 0) + m(0, 2, 0) + m(0, 0, 2)
            e1 = m(3, 0, 0) + m(1, 2, 0) + m(1, 0, 2)
            e2 = m(2, 1, 0) + m(0, 3, 0) + m(0, 1, 2)
            e3 = m(2, 0, 1) + m(0, 2, 1) + m(0, 0, 3)
            ee = m(4, 0, 0) + m(0, 4, 0) + m(0, 0, 4) + 2 * (m(2, 2, 0) + m(2, 0, 2) + m(0, 2, 2))
            mom = mom + torch.stack([m(0, 0, 0), m(1, 0, 0), m(0, 1, 0), m(0, 0, 1), e], -1)
            rows = [[m(0, 0, 0), m(1, 0, 0), m(0, 1, 0), m(0, 0, 1), e],
                    [m(1, 0, 0), m(2, 0, 0), m(1, 1, 0), m(1, 0, 1), e1],
                    [m(0, 1, 0), m(1, 1, 0), m(0, 2, 0), m(0, 1, 1), e2],
                    [m(0, 0, 1), m(1, 0, 1), m(0, 1, 1), m(0, 0, 2), e3], [e, e1, e2, e3, ee]]
            A = A + torch.stack([torch.stack(r, -1) for r in rows], -2)
        c = (self.w * a)[:, None]
        F = c * mom - target
        return F, c[..., None] * A, F.abs().amax(1) / target[:, 0].abs()

    def solve(self, target, wts=None, th=None, iters=30):
        if th is None:
            rho = target[:, 0]
            U = target[:, 1:4] / rho[:, None]
            uu = (U * U).sum(1)
            T = (target[:, 4] / rho - uu) / 3.0
            al = torch.log(rho / (2 * math.pi * T) ** 1.5) - 0.5 * uu / T
            th = torch.cat([al[:, None], U / T[:, None], (0.5 / T)[:, None]], 1)
        if wts is None:
            one = torch.ones_like(self.v)
            wts = [(one, one)]
        sign = torch.tensor([-1.0, -1.0, -1.0, -1.0, 1.0], dtype=torch.float64, device=th.device)
        F, A, fn = self._system(th, wts, target)
        for it in range(iters):
            A = torch.where(torch.isfinite(A), A, torch.eye(5, dtype=A.dtype, device=A.device))
            d = torch.linalg.solve_ex(A, F)[0] * sign
            lam = torch.ones_like(fn)
            best = fn
            for _ in range(12):
                t = th + lam[:, None] * d
                F, A, fn = self._system(t, wts, target)
                bad = ~((fn <= best) | (fn <= 1e-10))
                if it > 4 or not bool(bad.any()):
                    break
                lam = torch.where(bad, 0.5 * lam, lam)
            th = t
            if it >= 2 and float(fn.max()) <= 4e-15:
                break
            if it > 8:
                break
        return th


class _Exact:
    def __init__(self, c, probs):
        self.c, self.probs = c, probs
        self.dev = torch.device(DEVICE)
        self.N, self.L = c["nv"], c["vmax"]
        self.v = _nodes(c, self.dev)
        self.w = (2.0 * self.L / self.N) ** 3
        self.ph = _phi(self.v)
        self.mx = _Maxwellians(self.v, self.w)
        self.n, self.H = self.N - 1, self.N // 2 - 1
        self.R2 = 2.0 * 2.0 * self.L / (3.0 * math.sqrt(2.0) + 1.0)
        k = torch.arange(-self.H, self.H + 1, dtype=torch.float64, device=self.dev)
        j = torch.arange(self.N, dtype=torch.float64, device=self.dev) - self.N // 2 + 1
        self.E = torch.exp(2j * math.pi / self.N * (torch.outer(k, j) % self.N))  # (n, N)
        self.b0 = probs[0].b0
        if c["gas"] in ("maxwell", "hard"):
            x, wx = np.polynomial.legendre.leggauss(256)
            rho = torch.as_tensor(0.5 * self.R2 * (x + 1.0), device=self.dev)
            wr = torch.as_tensor(0.5 * self.R2 * wx, device=self.dev) * rho ** 2 * self.b0 * 16.0 * math.pi ** 2
            if c["gas"] == "hard":
                wr = wr * rho

            def radial(top):
                s = torch.sqrt(torch.arange(top, dtype=torch.float64, device=self.dev))
                return torch.sinc(torch.outer(s, rho) / (2.0 * self.L))

            H2 = self.H * self.H
            self.G = (radial(3 * H2 + 1) * wr) @ radial(12 * H2 + 1).T
            self.Lo = (radial(12 * H2 + 1) * wr).sum(1)[::4]  # G(2|m|, 0) by |m|^2

    def moments(self, f):
        return self.w * torch.einsum("bxyz,kxyz->bk", f, self.ph)

    def dft(self, f):
        E = self.E.conj()
        return torch.einsum("ax,by,cz,qxyz->qabc", E, E, E, f.to(E.dtype)) / self.N ** 3

    def nu(self, rho):
        return 4.0 * math.pi * self.b0 * rho * (self.R2 if self.c["gas"] == "hard" else 1.0)

    def collide(self, f):
        """Q, P, nu and the Maxwellian of every cell."""
        th = self.mx.solve(self.moments(f))
        M = self.mx.values(th)
        nu = self.nu(self.w * f.sum((1, 2, 3)))[:, None, None, None]
        if self.c["gas"] == "bgk":
            return nu * (M - f), torch.zeros_like(f), nu
        n, H, dev = self.n, self.H, self.dev
        a, b = self.dft(f - M), self.dft(f + M)
        q = torch.zeros((f.shape[0], H + 1, n, n), dtype=a.dtype, device=dev)  # k1 >= 0
        i = torch.arange(-H, H + 1, device=dev)
        k3, m3 = i[:, None], i[None, :]
        l3 = k3 - m3
        ok3 = (l3.abs() <= H)
        at = (l3 + H).clamp(0, n - 1)
        for m1 in range(-H, H + 1):
            k1 = torch.arange(max(0, m1 - H), min(H, m1 + H) + 1, device=dev)
            for m2 in range(-H, H + 1):
                k2 = torch.arange(max(-H, m2 - H), min(H, m2 + H) + 1, device=dev)
                p1, p2 = k1[:, None, None, None], k2[None, :, None, None]
                kk = p1 * p1 + p2 * p2 + (k3 * k3)
                dd = (p1 - 2 * m1) ** 2 + (p2 - 2 * m2) ** 2 + (k3 - 2 * m3) ** 2
                ll = (p1 - m1) ** 2 + (p2 - m2) ** 2 + l3 * l3
                mm = m1 * m1 + m2 * m2 + m3 * m3
                W = self.G[kk.expand_as(dd), dd.clamp(max=12 * H * H)] - 0.5 * (self.Lo[ll.clamp(max=3 * H * H)] + self.Lo[mm])
                W = torch.where(ok3, W, torch.zeros((), dtype=W.dtype, device=dev))
                s1 = slice(int(k1[0]) - m1 + H, int(k1[-1]) - m1 + H + 1)
                s2 = slice(int(k2[0]) - m2 + H, int(k2[-1]) - m2 + H + 1)
                o1, o2 = slice(int(k1[0]), int(k1[-1]) + 1), slice(int(k2[0]) + H, int(k2[-1]) + H + 1)
                for c0 in range(0, f.shape[0], 32):
                    cs = slice(c0, c0 + 32)
                    T = a[cs, s1, s2][..., at] * b[cs, m1 + H, m2 + H][:, None, None, None, :]
                    q[cs, o1, o2] += torch.view_as_complex(
                        (torch.view_as_real(T) * W[None, ..., None]).sum(-2))
        qh = torch.zeros_like(a)
        qh[:, H:] = q
        qh[:, :H] = q[:, 1:].flip(1, 2, 3).conj()
        Q = torch.einsum("ax,by,cz,qabc->qxyz", self.E, self.E, self.E, qh).real
        return Q, Q - nu * (M - f), nu

    def wall(self, p, side):
        """Incoming unit Maxwellian of a side and its discrete normalisation (N, N, N)."""
        kinds = list(p.bc_kind) + list(p.bc_kind_y)
        rho = (list(p.bc_rho) + list(p.bc_rho_y))[side]
        u = (list(p.bc_u) + list(p.bc_u_y))[side]
        T = (list(p.bc_T) + list(p.bc_T_y))[side]
        vn = self.ph[1] if side < 2 else self.ph[2]
        into = (vn > 0) if side % 2 == 0 else (vn < 0)
        cc = (self.ph[1] - u[0]) ** 2 + (self.ph[2] - u[1]) ** 2 + (self.ph[3] - u[2]) ** 2
        M = torch.exp(-0.5 * cc / T) / (2 * math.pi * T) ** 1.5 * into
        return kinds[side], rho, M, self.w * (vn * M).sum(), vn * ~into

    def ghost(self, p, side, f):
        kind, rho, M, den, vout = self.wall(p, side)
        if kind == sgs.INFLOW:
            return rho * M.expand_as(f)
        return (-(self.w * (vout * f).sum((1, 2, 3))) / den)[:, None, None, None] * M

    def visit(self, g, r, nu, eps, c1, c2, tol):
        """PFP solve of a batch of cells: c1, c2 the 1-D transport weights |v1|/dx, |v2|/dy (B, N)."""
        A = nu / eps
        cw = c1[:, :, None, None] + c2[:, None, :, None]
        one = torch.ones_like(c1)
        wts = [(c1, one), (one, c2)] if float(c2.abs().max()) > 0 else [(c1, one)]
        th = self.mx.solve(self.moments(g))
        going = torch.ones(g.shape[0], dtype=torch.bool, device=self.dev)
        for it in range(201):
            M = self.mx.values(th)
            res = torch.sqrt(self.w * ((cw + A) * g + r - A * M).square().sum((1, 2, 3)))
            going = going & (res >= tol) & (it < 200)
            if not bool(going.any()):
                return g
            s = self.moments(cw * (M - g) - r)
            exists = (s[:, 0] > 0) & (s[:, 0] * s[:, 4] > (s[:, 1:4] ** 2).sum(1))
            safe = torch.where((exists & going)[:, None], s, self.w * torch.einsum("bxyz,kxyz->bk", cw * M, self.ph))
            tp = torch.where((exists & going)[:, None], self.mx.solve(safe, wts, th), th)
            new = (A * self.mx.values(tp) - r) / (cw + A)
            g = torch.where(going[:, None, None, None], new, g)
            th = torch.where(going[:, None], self.mx.solve(self.moments(g), None, tp), th)
        return g

    def slopes(self, f, axis):
        if f.shape[axis] < 2:
            return torch.zeros_like(f)
        return torch.gradient(f, dim=axis, edge_order=1)[0]

    def slope_terms(self, p, f, axis, sides, v, d):
        """The explicit second-order part of a scan's right-hand side along one axis, f (.., N, N, N)."""
        s = self.slopes(f, axis)
        f2, s2 = f.movedim(axis, 0), s.movedim(axis, 0)
        z = torch.zeros_like(s2[:1])
        sm, sp = torch.cat([z, s2[:-1]]), torch.cat([s2[1:], z])
        b = (v.clamp(min=0) * sm - v * s2 + v.clamp(max=0) * sp) / (2 * d)
        for side, at, sg in ((sides[0], 0, 1.0), (sides[1], -1, -1.0)):
            kind, _, M, den, vout = self.wall(p, side)
            if kind != sgs.INFLOW:
                dr = sg * 0.5 * self.w * (vout * s2[at]).sum((-3, -2, -1), keepdim=True) / den
                b[at] += sg * (v.clamp(min=0) if sg > 0 else v.clamp(max=0)) * dr * M / d
        return b.movedim(0, axis)

    def scan1d(self, f, P, nu, forward):
        """Scans of every instance, those with cells left visited together."""
        pr, v1 = self.probs, self.ph[1]
        first = np.cumsum([0] + [p.nx for p in pr])
        f = f.clone()
        rhs = torch.zeros_like(f)
        if self.c["order"] == 2:
            for q, p in enumerate(pr):
                sl = slice(first[q], first[q + 1])
                rhs[sl] = self.slope_terms(p, f[sl], 0, (0, 1), v1, (p.x_hi - p.x_lo) / p.nx)
        for s in range(max(p.nx for p in pr)):
            ids = [q for q, p in enumerate(pr) if s < p.nx]
            js = [s if forward else pr[q].nx - 1 - s for q in ids]
            cells = [first[q] + j for q, j in zip(ids, js)]
            dx = torch.tensor([(pr[q].x_hi - pr[q].x_lo) / pr[q].nx for q in ids], dtype=torch.float64, device=self.dev)
            eps = torch.tensor([pr[q].eps for q in ids], dtype=torch.float64, device=self.dev)[:, None, None, None]
            g = f[cells]
            west = torch.stack([f[c - 1] if j else self.ghost(pr[q], 0, f[c][None])[0] for q, j, c in zip(ids, js, cells)])
            east = torch.stack([f[c + 1] if j < pr[q].nx - 1 else self.ghost(pr[q], 1, f[c][None])[0]
                                for q, j, c in zip(ids, js, cells)])
            d4 = dx[:, None, None, None]
            r = (v1.clamp(max=0) * east - v1.clamp(min=0) * west) / d4 - P[cells] / eps - rhs[cells]
            c1 = self.v.abs()[None] / dx[:, None]
            f[cells] = self.visit(g, r, nu[cells], eps, c1, torch.zeros_like(c1), pr[0].inner_tol)
        return f

    def scan2d(self, f, P, nu, o):
        p, N = self.probs[0], self.N
        nx, ny, v1, v2 = p.nx, p.ny, self.ph[1], self.ph[2]
        dx, dy = (p.x_hi - p.x_lo) / nx, (p.y_hi - p.y_lo) / ny
        F = f.clone().view(ny, nx, N, N, N)
        rhs = torch.zeros_like(F)
        if self.c["order"] == 2:
            rhs = self.slope_terms(p, F, 1, (0, 1), v1, dx) + self.slope_terms(p, F, 0, (2, 3), v2, dy)
        PP, NU = P.view_as(F), nu.view(ny, nx, 1, 1, 1)
        for wf in range(nx + ny - 1):
            ak = [a for a in range(nx) if 0 <= wf - a < ny]
            ci = [a if o in (0, 2) else nx - 1 - a for a in ak]
            cj = [wf - a if o in (0, 3) else ny - 1 - (wf - a) for a in ak]
            g = F[cj, ci]

            def nb(di, dj, side):
                edge = torch.tensor([not (0 <= i + di < nx and 0 <= j + dj < ny) for i, j in zip(ci, cj)], device=self.dev)
                x = F[[min(max(j + dj, 0), ny - 1) for j in cj], [min(max(i + di, 0), nx - 1) for i in ci]]
                return torch.where(edge[:, None, None, None], self.ghost(p, side, g), x) if bool(edge.any()) else x

            r = (v1.clamp(max=0) * nb(1, 0, 1) - v1.clamp(min=0) * nb(-1, 0, 0)) / dx \
                + (v2.clamp(max=0) * nb(0, 1, 3) - v2.clamp(min=0) * nb(0, -1, 2)) / dy - PP[cj, ci] / p.eps - rhs[cj, ci]
            c1 = (self.v.abs() / dx).expand(len(ci), N)
            c2 = (self.v.abs() / dy).expand(len(ci), N)
            F[cj, ci] = self.visit(g, r, NU[cj, ci], p.eps, c1, c2, p.inner_tol)
        return F.view_as(f)

    def scan(self, f, P, nu, o):
        return self.scan2d(f, P, nu, o) if self.c["ny"] else self.scan1d(f, P, nu, o == 0)

    def rescale(self, f):
        p = self.probs[0]
        if p.total_mass <= 0:
            return f
        cell = (p.x_hi - p.x_lo) / p.nx * ((p.y_hi - p.y_lo) / p.ny if self.c["ny"] else 1.0)
        return f * (p.total_mass / (cell * self.w * f.sum()))

    def residual(self, f, Q):
        p, N = self.probs[0], self.N
        nx, ny = p.nx, p.ny if self.c["ny"] else 1
        F = f.view(ny, nx, N, N, N)
        R = -Q.view_as(F) / p.eps
        cell = 1.0
        for axis, sides, v, n, d in ((1, (0, 1), self.ph[1], nx, (p.x_hi - p.x_lo) / nx),
                                     (0, (2, 3), self.ph[2], ny, (p.y_hi - p.y_lo) / ny)):
            if axis == 0 and not self.c["ny"]:
                continue
            cell *= d
            s = self.slopes(F, axis) if self.c["order"] == 2 else torch.zeros_like(F)
            lo, hi = (F - 0.5 * s).movedim(axis, 0), (F + 0.5 * s).movedim(axis, 0)
            left = torch.cat([self.ghost(p, sides[0], lo[0])[None], hi[:-1]])
            right = torch.cat([lo[1:], self.ghost(p, sides[1], hi[-1])[None]])
            R = R + ((v.clamp(min=0) * (hi - left) + v.clamp(max=0) * (right - lo)) / d).movedim(0, axis)
        return torch.sqrt(cell * self.w * R.square().sum()).reshape(1)

    def fast(self, f):
        """The half-sphere rule of 8 x 16 nodes, convolutions by zero-padded FFTs."""
        n, H, T, L = self.n, self.H, self.R2, self.L
        k = torch.arange(-H, H + 1, dtype=torch.float64, device=self.dev)
        K = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1)
        fh = self.dft(f)
        S = 3 * H + 1
        x, wx = np.polynomial.legendre.leggauss(8)

        def phi(s):  # 2 int_0^T r cos(pi r s / L) dr
            return 2 * T * T * torch.sinc(s * T / L) - T * T * torch.sinc(0.5 * s * T / L) ** 2

        half = torch.cos((torch.arange(64, dtype=torch.float64, device=self.dev) + 0.5) * math.pi / 64)

        def psi(t):  # int_0^pi phi(t cos u) du, midpoint rule of a periodic function
            return sum(phi(t * u) for u in half) * (math.pi / 64)

        Q = torch.empty_like(f)
        for c0 in range(0, f.shape[0], 16):
            h = fh[c0:c0 + 16]

            def grid(z):
                return torch.fft.fftn(z, (S, S, S), dim=(1, 2, 3))

            acc, bmm = 0.0, 0.0
            for i in range(8):
                mu, wt = 0.5 * (x[i] + 1.0), 0.5 * wx[i] * 2 * math.pi / 16
                st = math.sqrt(1 - mu * mu)
                for j in range(16):
                    e = torch.tensor([st * math.cos(2 * math.pi * j / 16), st * math.sin(2 * math.pi * j / 16), mu],
                                     dtype=torch.float64, device=self.dev)
                    s = K @ e
                    a, b = phi(s), psi(torch.sqrt(((K * K).sum(-1) - s * s).clamp(min=0)))
                    acc = acc + wt * grid(a * h) * grid(b * h)
                    bmm = bmm + wt * a * b
            acc = 4 * self.b0 * (acc - grid(h) * grid(bmm * h))
            qh = torch.fft.ifftn(acc, dim=(1, 2, 3))  # index H + H is k = 0; S = 3H + 1 keeps H .. 3H clear of wraps
            qh = qh[:, H:H + n, H:H + n, H:H + n]
            Q[c0:c0 + 16] = torch.einsum("ax,by,cz,qabc->qxyz", self.E, self.E, self.E, qh).real
        return Q


def exact(case, seed):
    c = case
    pairs = 0.5 * (3 * (c["nv"] // 2 - 1) * (c["nv"] // 2) + 1) ** 3 * _cells(c)
    if c["gas"] != "bgk" and c["do"] == "iterate" and c["ny"]:
        return None
    if c["do"] == "collide" and pairs > 3e10:
        return None
    probs, f, P0 = _inputs(c, seed)
    x = _Exact(c, probs)
    if c["do"] == "fast":
        return {"Q": x.fast(f).reshape(-1)}
    if c["do"] == "collide":
        Q, P, _ = x.collide(f)
        return {"Q": Q.reshape(-1), "P": P.reshape(-1)}
    if c["do"] == "scan":
        nu = x.nu(x.w * f.sum((1, 2, 3)))[:, None, None, None]
        return {"f": x.scan(f, P0, nu, c["ordering"]).reshape(-1)}
    if c["do"] == "iterate":
        for o in range(4 if c["ny"] else 2):
            _, P, nu = x.collide(f)
            f = x.scan(f, P, nu, o)
        f = x.rescale(f)
        Q, P, _ = x.collide(f)
        res = x.residual(f, Q)
    else:
        Q, P, nu = x.collide(f)
        res = x.residual(f, Q)
        for _ in range(c["iters"]):
            f = x.scan(f, P, nu, 0)
            _, P, nu = x.collide(f)
            f = x.rescale(x.scan(f, P, nu, 1))
            Q, P, nu = x.collide(f)
        if c["nx"] <= 32:  # one lane group: the evaluation that the call leaves in Q and P is an earlier one
            Q = P = None
    return {"f": f.reshape(-1), "Q": Q if Q is None else Q.reshape(-1), "P": P if P is None else P.reshape(-1), "res": res}
