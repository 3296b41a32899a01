"""The work that users of this framework have it do, as cases that can be timed and compared.

Every case goes through the public binding (Grid, Batch).  `prepare` makes the state a program has in
hand: Brill-Lindquist data of seeded punctures plus a smooth seeded perturbation of every gridfunction
(an evolved state has no gridfunction that vanishes), regular on the symmetry axis, with its inner
ghosts filled.  `exact` restates the right-hand side and the constraints of arXiv 2505.00097 Sec. 2.1
in plain torch FP64, with dense tensors in the orthonormal frame of the reference metric.
"""
import math

import torch

from paper_2505_00097_gb300 import binding as B
from paper_2505_00097_gb300 import workloads as W

NGF = 24
KO8 = [0.3] * 17 + [0.99] * 7
FAMILIES = ("sinh_spherical", "sinh_cylindrical", "spherical")
SYM = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


# ------------------------------------------------------------------ cases

def listed():
    def c(name, kind, fam, n0, n1, n2, order=4, steps=1, grids=1):
        return dict(name=name, kind=kind, fam=fam, n0=n0, n1=n1, n2=n2, order=order, steps=steps, grids=grids)

    return [
        # a quick test evolution: one puncture on the smallest grid, where launches and latency count
        c("puncture_steps", "step", "sinh_spherical", 64, 16, 2, steps=4),
        # the paper's desktop benchmark grid, a small three-dimensional evolution
        c("desktop_step", "step", "spherical", 72, 12, 24),
        # one right-hand side of the axisymmetric head-on collision, the call under every integrator
        c("headon_rhs", "rhs", "sinh_cylindrical", 256, 2, 512),
        # the head-on evolution itself, 4th order and RK4
        c("headon_steps", "step", "sinh_cylindrical", 256, 2, 512, steps=2),
        # the head-on evolution with the production scheme (8th order, SSPRK3)
        c("headon8_steps", "step", "sinh_cylindrical", 256, 2, 512, order=8, steps=2),
        # a host program that hands its state in and takes it back on every step
        c("headon_io", "io", "sinh_cylindrical", 256, 2, 512),
        # a parameter study: uneven head-on grids advanced together
        c("batch_step", "batch", "sinh_cylindrical", 64, 2, 128, grids=6),
        # three-dimensional right-hand side without symmetry, 4th order
        c("general_rhs", "rhs", "sinh_spherical", 192, 96, 192),
        # the same with the production scheme's 8th-order stencils
        c("general8_step", "step", "sinh_spherical", 192, 96, 192, order=8),
        # ragged three-dimensional cylindrical grid (sizes that fill no tile), 8th order
        c("ragged8_rhs", "rhs", "sinh_cylindrical", 77, 10, 131, order=8),
        # the constraint monitor of a head-on run: both constraints and their norms
        c("headon_constraints", "constraints", "sinh_cylindrical", 256, 2, 512),
        # the largest vacuum evolution that is configured here
        c("large3d_step", "step", "sinh_spherical", 384, 192, 384),
    ]


def draw(rng):
    kind = rng.choice(("rhs", "rhs", "step", "step", "io", "batch", "constraints"))
    fam = rng.choice(FAMILIES)
    order = rng.choice((4, 4, 8))
    two = rng.random() < 0.5
    if kind == "batch":
        fam, two = "sinh_cylindrical", True
    points = math.exp(rng.uniform(math.log(4e3), math.log(4e6)))
    if kind in ("io", "constraints"):
        points = min(points, 1e6)
    if kind == "batch":
        points = min(points, 1e5)
    azimuth = 2 if two else 2 * rng.randint(3, 24)
    other = points / azimuth
    first = int(min(512, max(12, round(math.sqrt(other) * math.exp(rng.uniform(-0.6, 0.6))))))
    last = int(min(512, max(12, round(other / first))))
    n = (first, azimuth, last) if fam == "sinh_cylindrical" else (first, last, azimuth)
    return dict(kind=kind, fam=fam, n0=n[0], n1=n[1], n2=n[2], order=order, steps=rng.randint(1, 3) if kind == "step" else 1,
                grids=rng.randint(2, 6) if kind == "batch" else 1)


def _spec(case, n=None):
    n = n or (case["n0"], case["n1"], case["n2"])
    kw = dict(NG=5, ko_sigma=KO8, integrator="ssprk3", cfl=0.35) if case["order"] == 8 else {}
    return getattr(W, case["fam"])(n, **kw)


def _grids(case):
    """The sizes of the case's grids: a batch's grow from the first by a quarter each, as studies mix resolutions."""
    n = (case["n0"], case["n1"], case["n2"])
    return [(int(n[0] * (1 + 0.25 * q)), n[1], int(n[2] * (1 + 0.25 * q))) for q in range(case["grids"])]


def work(case):
    # FP64 operations of one right-hand side per point, counted on the compiled kernels of the
    # two-point-azimuth and the general scheme; 24 gridfunctions read and 24 written
    two = (case["n1"] if case["fam"] == "sinh_cylindrical" else case["n2"]) == 2
    flops = {(True, 4): 2900, (True, 8): 3800, (False, 4): 4100, (False, 8): 5500}[two, case["order"]]
    points = sum(a * b * c for a, b, c in _grids(case))
    evals = (3 if case["order"] == 8 else 4) * case["steps"] if case["kind"] in ("step", "io", "batch") else 1
    if case["kind"] == "constraints":
        return {"bytes": points * 8.0 * (24 + 4), "flops": points * 2700.0}
    return {"bytes": points * 8.0 * 48, "flops": float(points) * flops * evals}


# ------------------------------------------------------------------ inputs

class _Axes:
    """Cell-centred logical coordinates of a padded grid and the scale factors of its reference metric."""

    def __init__(self, spec, dev="cuda"):
        self.NG = NG = spec["NG"]
        self.N = N = spec["N"]
        self.n = [v + 2 * NG for v in N]
        self.cyl = spec["coords"] == W.SINH_CYLINDRICAL
        pi = math.pi
        lo, hi = ((0, -pi, -1), (1, pi, 1)) if self.cyl else ((0, 0, -pi), (1, pi, pi))
        self.dx = [(hi[d] - lo[d]) / N[d] for d in range(3)]
        x = [lo[d] + (torch.arange(self.n[d], dtype=torch.float64, device=dev) - NG + 0.5) * self.dx[d] for d in range(3)]
        self.f0 = self._radial(spec, 0, x[0], spec["coords"] != W.SPHERICAL)
        self.x = x
        if self.cyl:
            self.f2 = self._radial(spec, 2, x[2], True)

    @staticmethod
    def _radial(spec, d, x, sinh):
        A, w = spec["ampl"][d], spec["sinhw"][d]
        if not sinh:
            return A * x, torch.full_like(x, A), torch.zeros_like(x)
        s = math.sinh(1.0 / w)
        return A * torch.sinh(x / w) / s, A * torch.cosh(x / w) / (w * s), A * torch.sinh(x / w) / (w * w * s)

    def cart(self):
        """Cartesian coordinates, each broadcastable to (n2, n1, n0)."""
        r = self.f0[0][None, None, :]
        if self.cyl:
            ph, z = self.x[1][None, :, None], self.f2[0][:, None, None]
            return r * torch.cos(ph), r * torch.sin(ph), z
        th, ph = self.x[1][None, :, None], self.x[2][:, None, None]
        return r * torch.sin(th) * torch.cos(ph), r * torch.sin(th) * torch.sin(ph), r * torch.cos(th)


def _state(case, spec, seed):
    """24 gridfunctions on the padded grid, (24, n2, n1, n0), ghosts included (the inner ones are refilled by the caller)."""
    ax = _Axes(spec)
    g = torch.Generator().manual_seed(1_000_003 * seed + 17)
    u = lambda a, b: a + (b - a) * float(torch.rand((), generator=g, dtype=torch.float64))  # noqa: E731
    X, Y, Z = ax.cart()
    q, d = u(1.0, 4.0), u(0.5, 2.0)
    m1, m2 = q / (1 + q), 1 / (1 + q)
    psi = 1.0
    for m, z in ((m1, d * m2), (m2, -d * m1)):
        psi = psi + m / (2 * torch.sqrt(X * X + Y * Y + (Z - z) ** 2))
    two = spec["N"][1 if ax.cyl else 2] == 2
    rho2 = X * X + Y * Y
    reg = rho2 / (1 + rho2)                                  # components off the axis: they vanish on it
    fall = 1.0 / (1.0 + 0.1 * (rho2 + Z * Z))                # and far away
    ph = torch.atan2(Y, X)
    y = torch.zeros((NGF, ax.n[2], ax.n[1], ax.n[0]), dtype=torch.float64, device="cuda")
    odd = set() if not two else {s for s, (i, j) in enumerate(SYM) if (i == (1 if ax.cyl else 2)) != (j == (1 if ax.cyl else 2))}
    for gf in range(NGF):
        amp = 0.02 if gf < 6 else 0.03 if gf < 12 else 0.01 if gf < 14 else 0.02
        f = 0.0
        for _ in range(2):
            k, p, a = u(0.2, 1.5), u(0, 2 * math.pi), u(-1, 1)
            t = torch.cos(k * Z + p) * torch.cos(u(0.2, 1.5) * torch.sqrt(rho2) + u(0, 2 * math.pi))
            if not two:
                t = t * torch.cos(2 * ph + u(0, 2 * math.pi))
            f = f + a * t
        comp = gf % 6 if gf < 12 else None
        if two and (comp in odd or gf in [b + (1 if ax.cyl else 2) for b in (14, 17, 20)]):
            continue                                         # zero under axisymmetry without rotation
        y[gf] = amp * f * fall * (reg if gf not in (12, 13, 23) or not two else 1.0)
    y[12] = psi ** -2 * (1 + y[12])
    y[23] = psi ** -2 * (1 + y[23])
    return y


def prepare(case, seed):
    specs = [_spec(case, n) for n in _grids(case)]
    grids = [B.Grid(s) for s in specs]
    states = []
    for q, (s, g) in enumerate(zip(specs, grids)):
        y = _state(case, s, seed * 16 + q).reshape(-1)
        g.apply_inner_bcs(y)
        states.append(y)
    st = dict(case=case, grids=grids, y=states)
    kind = case["kind"]
    if kind in ("rhs", "step", "batch"):
        st["out"] = [torch.zeros_like(y) for y in states]
    elif kind == "constraints":
        st["H"], st["M"] = torch.zeros(grids[0].T, dtype=torch.float64, device="cuda"), torch.zeros(3 * grids[0].T, dtype=torch.float64, device="cuda")
    if kind == "batch":
        st["batch"] = B.Batch(grids)
    if kind == "io":
        n = NGF * int(grids[0].info.n_state_points)
        st["host_in"], st["host_out"] = (torch.empty(n, dtype=torch.float64, pin_memory=True) for _ in range(2))
        grids[0].set_state(states[0], False)
        grids[0].get_state_compact(st["host_in"], True)
    st["keep"] = specs
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass

def run(st):
    case, grids = st["case"], st["grids"]
    kind, steps = case["kind"], case["steps"]
    scheme = "ssprk3" if case["order"] == 8 else "rk4"
    g = grids[0]
    if kind == "rhs":
        g.rhs(st["y"][0], st["out"][0])
        return st["out"][0]
    if kind == "constraints":
        h = g.hamiltonian(st["y"][0], st["H"])
        m = g.momentum(st["y"][0], st["M"])
        return [st["H"], st["M"], *h, *m]
    if kind == "io":
        g.step_io(g.dt_cfl, steps, st["host_in"], st["host_out"], scheme)
        return st["host_out"]
    # evolutions start from the state in hand, so that a pass can be repeated
    for q, y in zip(grids, st["y"]):
        q.set_state(y, False)
    if kind == "batch":
        getattr(st["batch"], scheme + "_step")([q.dt_cfl for q in grids], steps)
    else:
        getattr(g, scheme + "_step")(g.dt_cfl, steps)
    for q, o in zip(grids, st["out"]):
        q.get_state(o, False)
    return list(st["out"])


# ------------------------------------------------------------------ the equations in plain FP64

D1 = {4: ({-2: 1, -1: -8, 1: 8, 2: -1}, 12), 8: ({-4: 3, -3: -32, -2: 168, -1: -672, 1: 672, 2: -168, 3: 32, 4: -3}, 840)}
D2 = {4: ({-2: -1, -1: 16, 0: -30, 1: 16, 2: -1}, 12),
      8: ({-4: -9, -3: 128, -2: -1008, -1: 8064, 0: -14350, 1: 8064, 2: -1008, 3: 128, 4: -9}, 5040)}
UP = {4: ({-1: -3, 0: -10, 1: 18, 2: -6, 3: 1}, 12),
      8: ({-3: -5, -2: 60, -1: -420, 0: -378, 1: 1050, 2: -420, 3: 140, 4: -30, 5: 3}, 840)}
KO = {4: ((1, -6, 15, -20, 15, -6, 1), 64), 8: ((1, -10, 45, -120, 210, -252, 210, -120, 45, -10, 1), 1024)}


class _Slab:
    """Planes [k0, k1) of the interior along axis 2, with every field and derivative there as (..., points)."""

    def __init__(self, spec, ax, y, k0, k1):
        self.order = 2 * (spec["NG"] - 1)
        self.NG, self.ax, self.spec, self.y, self.k = spec["NG"], ax, spec, y, (k0, k1)
        N = spec["N"]
        self.shape = (k1 - k0, N[1], N[0])
        e = lambda v, d: v[self._range(d)].reshape([-1 if 2 - i == d else 1 for i in range(3)]).expand(self.shape).reshape(-1)  # noqa: E731
        one, zero = torch.ones_like(e(ax.x[0], 0)), torch.zeros_like(e(ax.x[0], 0))
        r, r1, r2 = (e(v, 0) for v in ax.f0)
        if ax.cyl:
            _, z1, z2 = (e(v, 2) for v in ax.f2)
            self.S = [r1, r, z1]
            self.L00, self.a, self.b, self.c, self.L22 = r2 / r1 ** 2, 1 / r, zero, zero, z2 / z1 ** 2
            ea, eb, ec0, ec1 = -1 / r ** 2, zero, zero, zero
        else:
            th = e(ax.x[1], 1)
            self.S = [r1, r, r * torch.sin(th)]
            cot = torch.cos(th) / torch.sin(th)
            self.L00, self.a, self.b, self.c, self.L22 = r2 / r1 ** 2, 1 / r, 1 / r, cot / r, zero
            ea, eb, ec0, ec1 = -1 / r ** 2, -1 / r ** 2, -cot / r ** 2, -1 / (r * torch.sin(th)) ** 2
        self.one = one
        P = one.numel()

        def omega(a, b, c):      # Omega_k as matrices (k, i, j), from the rotation coefficients
            O = torch.zeros((3, 3, 3, P), dtype=torch.float64, device=one.device)
            O[1, 1, 0], O[1, 0, 1] = a, -a
            O[2, 2, 0], O[2, 0, 2] = b, -b
            O[2, 2, 1], O[2, 1, 2] = c, -c
            return O

        self.O = omega(self.a, self.b, self.c)
        self.eO = torch.stack([omega(ea, eb, ec0), omega(zero, zero, ec1), torch.zeros_like(self.O)])  # e_k Omega_l: (k, l, i, j)

    def _range(self, d, o=0):
        lo, n = (self.NG, self.spec["N"][d]) if d < 2 else (self.NG + self.k[0], self.k[1] - self.k[0])
        return slice(lo + o, lo + o + n)

    def at(self, gf, o=(0, 0, 0)):
        return self.y[gf][self._range(2, o[2]), self._range(1, o[1]), self._range(0, o[0])].reshape(-1)

    def d1(self, gf, k):
        w, den = D1[self.order]
        off = lambda i: tuple(i if d == k else 0 for d in range(3))  # noqa: E731
        return sum(c * self.at(gf, off(i)) for i, c in w.items()) / (den * self.ax.dx[k])

    def d2(self, gf, k, l):
        if k == l:
            w, den = D2[self.order]
            return sum(c * self.at(gf, tuple(i if d == k else 0 for d in range(3))) for i, c in w.items()) / (den * self.ax.dx[k] ** 2)
        w, den = D1[self.order]
        t = 0.0
        for i, c in w.items():
            for j, e in w.items():
                t = t + c * e * self.at(gf, tuple(i if d == k else j if d == l else 0 for d in range(3)))
        return t / (den * den * self.ax.dx[k] * self.ax.dx[l])

    def frame1(self, gf):
        return torch.stack([self.d1(gf, k) / self.S[k] for k in range(3)])

    def hess(self, gf, e):
        """e_k e_l f - Gamma^m_kl e_m f, symmetric."""
        H = torch.zeros((3, 3, e.shape[-1]), dtype=torch.float64, device=e.device)
        drift = {(0, 0): self.L00 * e[0], (0, 1): self.a * e[1], (0, 2): self.b * e[2], (1, 2): self.c * e[2],
                 (1, 1): -self.a * e[0], (2, 2): self.L22 * e[2] - self.b * e[0] - self.c * e[1]}
        for k, l in SYM:
            H[k, l] = H[l, k] = self.d2(gf, k, l) / (self.S[k] * self.S[l]) - drift[k, l]
        return H

    def scalar(self, gf):
        e = self.frame1(gf)
        return self.at(gf), e, self.hess(gf, e)

    def vector(self, base, second):
        V = torch.stack([self.at(base + i) for i in range(3)])
        e = torch.stack([self.frame1(base + i) for i in range(3)], 1)              # e[k, i]
        D = e + _s("kijp,jp->kip", self.O, V)
        if not second:
            return V, e, D
        H = torch.stack([self.hess(base + i, e[:, i]) for i in range(3)], 2)       # H[k, l, i]
        DD = H + _s("klijp,jp->klip", self.eO, V) + _s("lijp,kjp->klip", self.O, e) + _s("kijp,ljp->klip", self.O, D)
        return V, e, D, DD - _s("kmlp,mijp,jp->klip", self.O, self.O, V)

    def tensor(self, base, second):
        T = _full([self.at(base + s) for s in range(6)])
        e = torch.stack([_full(list(v)) for v in torch.stack([self.frame1(base + s) for s in range(6)], 1)])   # e[k, i, j]
        rot = lambda O, X: _s("imp,mjp->ijp", O, X) + _s("jmp,imp->ijp", O, X)  # noqa: E731
        D = torch.stack([e[k] + rot(self.O[k], T) for k in range(3)])
        if not second:
            return T, e, D
        Hs = torch.stack([self.hess(base + s, torch.stack([e[k][SYM[s]] for k in range(3)])) for s in range(6)])  # (s, k, l)
        H = torch.stack([torch.stack([_full(list(Hs[:, k, l])) for l in range(3)]) for k in range(3)])           # (k, l, i, j)
        DD = torch.empty_like(H)
        OT = torch.stack([rot(self.O[m], T) for m in range(3)])
        for k in range(3):
            for l in range(3):
                DD[k, l] = H[k, l] + rot(self.eO[k, l], T) + rot(self.O[l], e[k]) + rot(self.O[k], D[l]) - _s("mp,mijp->ijp", self.O[k][:, l], OT)
        return T, e, D, H, DD


def _s(eq, *ops):
    """einsum over small leading axes, pointwise in the last one (p), by explicit products."""
    ins, out = eq.split("->")
    ins = ins.split(",")
    letters = sorted(set("".join(ins)) - {"p"}, key=lambda c: (c not in out, out.find(c), c))
    t = None
    for name, x in zip(ins, ops):
        order = [name.index(c) for c in letters if c in name] + [len(name) - 1]
        x = x.permute(order)
        x = x.reshape([3 if c in name else 1 for c in letters] + [x.shape[-1]])
        t = x if t is None else t * x
    axes = [i for i, c in enumerate(letters) if c not in out]
    return t.sum(axes) if axes else t


def _full(s):
    return torch.stack([torch.stack([s[0], s[1], s[2]]), torch.stack([s[1], s[3], s[4]]), torch.stack([s[2], s[4], s[5]])])


def _metric(sl):
    h, eh, Dh, Hh, DDh = sl.tensor(0, True)
    eye = torch.eye(3, dtype=torch.float64, device=h.device)[:, :, None]
    g = eye + h
    gi = torch.linalg.inv(g.permute(2, 0, 1)).permute(1, 2, 0)
    low = 0.5 * (_s("ijkp->kijp", Dh) + _s("jikp->kijp", Dh) - Dh)               # Delta_kij
    up = _s("klp,lijp->kijp", gi, low)
    vec = _s("ijp,kijp->kp", gi, up)
    lam, elam, Dlam = sl.vector(14, False)                                       # Dlam[j, k]
    q = _s("klp,mkip,jmlp->ijp", gi, up, low)
    Ric = -0.5 * _s("klp,klijp->ijp", gi, DDh) + q + q.transpose(0, 1) + _s("klp,mikp,mjlp->ijp", gi, up, low)
    t = _s("kip,jkp->ijp", g, Dlam) + _s("kp,ijkp->ijp", vec, low)
    Ric = Ric + 0.5 * (t + t.transpose(0, 1))
    Wf, eW, HW = sl.scalar(12)
    ph = -0.5 * eW / Wf
    DDphi = -0.5 * HW / Wf + 2 * _s("ip,jp->ijp", ph, ph) - _s("kijp,kp->ijp", up, ph)
    return dict(h=h, eh=eh, Hh=Hh, g=g, gi=gi, low=low, up=up, vec=vec, lam=lam, Dlam=Dlam, Ric=Ric, W=Wf, ph=ph, DDphi=DDphi)


def _rhs(sl, eta):
    m = _metric(sl)
    g, gi, up, vec, ph, Wf, h, O = m["g"], m["gi"], m["up"], m["vec"], m["ph"], m["W"], m["h"], sl.O
    a = _full([sl.at(6 + s) for s in range(6)])
    K, eK = sl.at(13), sl.frame1(13)
    al, ea, Ha = sl.scalar(23)
    v, ev, Dv, DDv = sl.vector(17, True)                                         # Dv[k, i] = D_k beta^i
    B_ = torch.stack([sl.at(20 + i) for i in range(3)])
    DDa = Ha - _s("kijp,kp->ijp", up, ea)
    Aud = _s("kip,ijp->kjp", gi, a)
    Auu = _s("kip,ijp->kjp", Aud, gi)
    trA, AA = Aud[0, 0] + Aud[1, 1] + Aud[2, 2], _s("ijp,ijp->p", a, Auu)
    tr = 0.5 * _s("abp,mabp->mp", gi, m["eh"])                                   # Delta^k_km
    div = Dv[0, 0] + Dv[1, 1] + Dv[2, 2] + _s("mp,mp->p", tr, v)
    Mm = _s("iap,lajp->lijp", gi, m["eh"])
    Q, GH = _s("lijp,mjip->lmp", Mm, Mm), _s("ijp,lmijp->lmp", gi, m["Hh"])
    etr = 0.5 * (GH - Q) - _s("lmnp,np->lmp", O, tr)
    gdiv = DDv[:, 0, 0] + DDv[:, 1, 1] + DDv[:, 2, 2] + _s("lmp,mp->lp", etr, v) + _s("mp,lmp->lp", tr, ev)
    rot = lambda X: _s("kp,kimp,mjp->ijp", v, O, X)  # noqa: E731
    both = lambda X: X + X.transpose(0, 1)  # noqa: E731
    rh = both(rot(h)) + both(_s("kjp,ikp->ijp", g, Dv)) - (2 / 3) * g * (div - al * trA) - 2 * al * a
    X = -2 * al * m["DDphi"] + 4 * al * _s("ip,jp->ijp", ph, ph) + 2 * both(_s("ip,jp->ijp", ea, ph)) - DDa + al * m["Ric"]
    X = X - g * _s("ijp,ijp->p", gi, X) / 3
    ra = both(rot(a)) + both(_s("ikp,jkp->ijp", a, Dv)) + a * (al * K - (2 / 3) * div) - 2 * al * _s("ikp,kjp->ijp", a, Aud) + Wf ** 2 * X
    rW = -Wf * (div - al * K) / 3
    rK = al * (K * K / 3 + AA) - Wf ** 2 * (_s("ijp,ijp->p", gi, DDa) + 2 * _s("ijp,ip,jp->p", gi, ea, ph))
    perp = _s("klp,klip->ip", gi, DDv) + (2 / 3) * vec * div + _s("ikp,kp->ip", gi, gdiv) / 3
    perp = perp - 2 * _s("ijp,jp->ip", Auu, ea - 6 * al * ph) + 2 * al * _s("jkp,ijkp->ip", Auu, up) - (4 / 3) * al * _s("ijp,jp->ip", gi, eK)
    rl = perp - _s("jp,jip->ip", m["lam"], Dv) + _s("jp,jikp,kp->ip", v, O, m["lam"])
    dv = torch.stack([sl.L00 * v[0], sl.a * v[0], sl.b * v[0] + sl.c * v[1] + sl.L22 * v[2]])
    out = [rh[i] for i in SYM] + [ra[i] for i in SYM] + [rW, rK] + list(rl) + list(B_ - v * dv) + list(0.75 * perp - eta * B_ - B_ * dv) + [-2 * al * K]
    ko = sl.spec["ko_sigma"]
    wu, den = UP[sl.order]
    wk, kden = KO[sl.order]
    for gf in range(NGF):
        sig = ko[gf] if isinstance(ko, (list, tuple)) else ko
        for d in range(3):
            off = lambda i: tuple(i if q == d else 0 for q in range(3))  # noqa: E731
            fw, bw = (sum(c * sl.at(gf, off(s * i)) for i, c in wu.items()) for s in (1, -1))
            diss = sum(c * sl.at(gf, off(i - len(wk) // 2)) for i, c in enumerate(wk))
            s = sl.S[d] * sl.ax.dx[d]
            out[gf] = out[gf] + v[d].abs() * torch.where(v[d] > 0, fw, bw) / (den * s) + sig * diss / (kden * s)
    return torch.stack(out)


def _constraints(sl):
    m = _metric(sl)
    gi, up, ph, Wf = m["gi"], m["up"], m["ph"], m["W"]
    a, _, Da = sl.tensor(6, False)
    K, eK = sl.at(13), sl.frame1(13)
    Aud = _s("kip,ijp->kjp", gi, a)
    Auu = _s("kip,ijp->kjp", Aud, gi)
    H = (2 / 3) * K * K - _s("ijp,ijp->p", a, Auu) + Wf ** 2 * (_s("ijp,ijp->p", gi, m["Ric"]) - 8 * _s("ijp,ip,jp->p", gi, ph, ph) - 8 * _s("ijp,ijp->p", gi, m["DDphi"]))
    V = _s("jlp,jklp->kp", gi, Da) - _s("mjkp,jmp->kp", up, Aud) - _s("kmp,mp->kp", a, m["vec"])
    M = Wf ** 2 * (_s("ikp,kp->ip", gi, V) + 6 * _s("ijp,jp->ip", Auu, ph) - (2 / 3) * _s("ijp,jp->ip", gi, eK))
    return torch.cat([H[None], M, (torch.sqrt(_s("ijp,ip,jp->p", m["g"], M, M)) / Wf)[None]])


def _with_ghosts(spec, ax, y):
    """The state with its inner ghosts mirrored from the interior (Sec. 3): through r = 0 (rho = 0) and the
    poles with half a turn, around the azimuth, vector components turning with the basis."""
    NG, N, n = spec["NG"], spec["N"], ax.n
    j = list(torch.meshgrid(*(torch.arange(v, device="cuda") for v in n[::-1]), indexing="ij"))[::-1]
    p = [torch.ones_like(j[0], dtype=torch.float64) for _ in range(3)]
    az = 1 if ax.cyl else 2
    flip = j[0] < NG
    j[0] = torch.where(flip, 2 * NG - 1 - j[0], j[0])
    j[az] = torch.where(flip, j[az] + N[az] // 2, j[az])
    sign = torch.where(flip, -1.0, 1.0).double()
    p[0], p[az] = p[0] * sign, p[az] * sign
    if not ax.cyl:
        j[1] = torch.where(flip, N[1] + 2 * NG - 1 - j[1], j[1])
        while bool(((j[1] < NG) | (j[1] >= NG + N[1])).any()):
            out = (j[1] < NG) | (j[1] >= NG + N[1])
            j[1] = torch.where(j[1] < NG, 2 * NG - 1 - j[1], torch.where(out, 2 * (NG + N[1]) - 1 - j[1], j[1]))
            j[2] = torch.where(out, j[2] + N[2] // 2, j[2])
            sign = torch.where(out, -1.0, 1.0).double()
            p[1], p[2] = p[1] * sign, p[2] * sign
    j[az] = NG + torch.remainder(j[az] - NG, N[az])
    src = (j[0] + n[0] * (j[1] + n[1] * j[2])).reshape(-1)
    one = torch.ones_like(p[0])
    par = [p[i] * p[k] for i, k in SYM] * 2 + [one, one] + p * 3 + [one]
    return torch.stack([y.reshape(NGF, -1)[g][src].reshape(n[::-1]) * par[g] for g in range(NGF)])


def exact(case, seed):
    if case["kind"] not in ("rhs", "constraints"):
        return None
    spec = _spec(case)
    ax = _Axes(spec)
    y = _state(case, spec, seed * 16).reshape(-1)
    y = _with_ghosts(spec, ax, y)
    NG, N = spec["NG"], spec["N"]
    rows = NGF if case["kind"] == "rhs" else 5
    out = torch.zeros((rows, *ax.n[::-1]), dtype=torch.float64, device="cuda")
    step = max(1, 250_000 // (N[0] * N[1]))
    for k0 in range(0, N[2], step):
        k1 = min(N[2], k0 + step)
        sl = _Slab(spec, ax, y, k0, k1)
        r = _rhs(sl, spec["eta"]) if rows == NGF else _constraints(sl)
        out[:, NG + k0:NG + k1, NG:NG + N[1], NG:NG + N[0]] = r.reshape(rows, *sl.shape)
    if rows == NGF:
        return out.reshape(-1)
    inner = out[:, NG:-NG, NG:-NG, NG:-NG]
    norms = []
    for t in (inner[0], inner[4]):
        norms += [float(t.square().mean().sqrt()), float(t.abs().max())]
    return [out[0].reshape(-1), out[1:4].reshape(-1), *norms]
