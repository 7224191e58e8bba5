"""Measured cases of the shifted-HSS Helmholtz solver: what a user of the library has it do.

Every case goes through the Python binding of the C ABI (``paper_2506_18694_gb300.hh``):

* ``solve``         one FGMRES solve to the workloads' tolerance of 1e-8 (``Problem.solve``);
* ``precondition``  one application of the shifted-HSS preconditioner, that is ceil(k) HSS steps
                    with a V(2,2) cycle each (``Problem.precondition``): what every outer iteration
                    of a solve spends its time on, for one problem or for a batch (``nb`` > 1);
* ``vcycle``        one multigrid cycle on A_L x = b from 0 (``Problem.vcycle``), with scaled Jacobi
                    or with the paper's W-cycle and GMRES(5) smoother (``smoother``);
* ``jacobi``        one scaled-Jacobi sweep (``Problem.jacobi``);
* ``pack``          FGMRES solves on different grids that share their launches (``Pack``).

Right sides are load vectors b = M f of Gaussian sources at seeded centres with complex normal
amplitudes, plus a little noise.  ``exact`` restates the method in 64-bit torch from the weak
forms (tensor products of the 1D Q1 rows) and shares no code with the library.
"""
import math

import torch

from paper_2506_18694_gb300 import hh

C64, C128 = torch.complex64, torch.complex128
LEVELS = 4


# ---------------------------------------------------------------- cases
def listed():
    S2, S3 = "SSSS", "SSSSDS"
    return [
        # the smallest configuration: plain FP64 method, 1089 unknowns, launches and latency
        dict(name="solve_2d_n32_k10_c128", kind="solve", dim=2, n=32, k=10.0, bc=S2, prec="c128"),
        # a small 3D request of the serving workload (n a multiple of 8, u = 0 on z = 0)
        dict(name="solve_3d_n40_k20_c64", kind="solve", dim=3, n=40, k=20.0, bc=S3, prec="c64"),
        # the headline 2D configuration: one outer iteration's preconditioner
        dict(name="precondition_2d_n512_k80_c64", kind="precondition", dim=2, n=512, k=80.0, bc=S2, prec="c64", nb=1),
        # a large ragged 2D request of the serving workload, k not a whole number
        dict(name="precondition_2d_n856_k93_c64", kind="precondition", dim=2, n=856, k=93.4, bc=S2, prec="c64", nb=1),
        # the 3D configuration: one outer iteration's preconditioner
        dict(name="precondition_3d_n128_k40_c64", kind="precondition", dim=3, n=128, k=40.0, bc=S3, prec="c64", nb=1),
        # the headline configuration's plain FP64 comparison
        dict(name="precondition_2d_n512_k80_c128", kind="precondition", dim=2, n=512, k=80.0, bc=S2, prec="c128",
             nb=1),
        # the batched configuration: 64 problems, k in {20, 40, 80}
        dict(name="precondition_2d_batch64_n256", kind="precondition", dim=2, n=256, k=80.0, bc=S2, prec="c64",
             nb=64),
        # the 2D roofline grid (larger than L2): one V-cycle
        dict(name="vcycle_2d_n4096_c64", kind="vcycle", dim=2, n=4096, k=80.0, bc=S2, prec="c64", smoother="jacobi"),
        # the 3D roofline grid (larger than L2): one V-cycle, and its dominant kernel alone
        dict(name="vcycle_3d_n256_c64", kind="vcycle", dim=3, n=256, k=40.0, bc=S3, prec="c64", smoother="jacobi"),
        dict(name="jacobi_3d_n256_c64", kind="jacobi", dim=3, n=256, k=40.0, bc=S3, prec="c64"),
        # the paper's multigrid (W-cycle, GMRES(5) with Jacobi), the server's fallback for stalled requests
        dict(name="wcycle_gmres5_2d_n256_c64", kind="vcycle", dim=2, n=256, k=20.0, bc=S2, prec="c64",
             smoother="gmres5"),
        # uneven grids solved together (the packed-launch workload)
        dict(name="pack8_2d_n64_256", kind="pack", dim=2, ns="64,96,128,160,192,224,256,96", ks="20,20,40,20,20,40,20,40",
             bc=S2, prec="c64"),
    ]


def _mult8(v, lo, hi):
    return min(max(int(round(v / 8.0)) * 8, lo), hi)


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _k(rng, n, top):
    """Wavenumber at 10 or more points per wavelength, as the serving workload draws it."""
    top = min(top, 2.0 * math.pi * n / 10.0)
    return round(rng.uniform(min(10.0, top), top), 2)


def _bc(rng, dim):
    if rng.random() < 0.6:
        return "SSSS" if dim == 2 else "SSSSDS"
    sides = [rng.choice("SSD") for _ in range(2 * dim)]
    sides[rng.randrange(2 * dim)] = "S"  # (a radiation side is left)
    return "".join(sides)


def draw(rng):
    kind = rng.choice(["solve2", "solve3", "pre2", "pre2", "pre2", "pre3", "pre3", "batch", "batch", "v2", "v2", "v3",
                       "v3", "j2", "j3", "gmres", "pack"])
    prec = rng.choice(["c64", "c64", "c128"])
    if kind == "solve2":
        n = _mult8(_log(rng, 16, 64), 16, 64)
        return dict(kind="solve", dim=2, n=n, k=_k(rng, n, 16.0), bc="SSSS", prec=prec)
    if kind == "solve3":
        n = _mult8(_log(rng, 16, 40), 16, 40)
        return dict(kind="solve", dim=3, n=n, k=_k(rng, n, 20.0), bc="SSSSDS", prec="c64")
    if kind == "pre2":
        n = _mult8(_log(rng, 64, 512 if prec == "c128" else 1024), 64, 1024)
        return dict(kind="precondition", dim=2, n=n, k=_k(rng, n, 80.0 if prec == "c128" else 160.0), bc=_bc(rng, 2),
                    prec=prec, nb=1)
    if kind == "pre3":
        n = _mult8(_log(rng, 32, 128), 32, 128)
        return dict(kind="precondition", dim=3, n=n, k=_k(rng, n, 40.0), bc=_bc(rng, 3), prec="c64", nb=1)
    if kind == "batch":
        n = _mult8(_log(rng, 64, 256), 64, 256)
        return dict(kind="precondition", dim=2, n=n, k=_k(rng, n, 80.0), bc=_bc(rng, 2), prec="c64",
                    nb=int(round(_log(rng, 4, 64))))
    if kind == "v2":
        n = _mult8(_log(rng, 512, 4096), 512, 4096)
        return dict(kind="vcycle", dim=2, n=n, k=_k(rng, n, 160.0), bc=_bc(rng, 2), prec="c64", smoother="jacobi")
    if kind == "v3":
        n = _mult8(_log(rng, 64, 256), 64, 256)
        return dict(kind="vcycle", dim=3, n=n, k=_k(rng, n, 80.0), bc=_bc(rng, 3), prec="c64", smoother="jacobi")
    if kind == "j2":
        n = _mult8(_log(rng, 256, 4096), 256, 4096)
        return dict(kind="jacobi", dim=2, n=n, k=_k(rng, n, 160.0), bc=_bc(rng, 2), prec=prec)
    if kind == "j3":
        n = _mult8(_log(rng, 64, 256), 64, 256)
        return dict(kind="jacobi", dim=3, n=n, k=_k(rng, n, 80.0), bc=_bc(rng, 3), prec=prec)
    if kind == "gmres":
        n = _mult8(_log(rng, 64, 256), 64, 256)
        return dict(kind="vcycle", dim=2, n=n, k=_k(rng, n, 40.0), bc="SSSS", prec="c64", smoother="gmres5")
    m = rng.randint(3, 8)
    ns = [rng.choice([64, 96, 128, 160, 192]) for _ in range(m)]
    return dict(kind="pack", dim=2, ns=",".join(map(str, ns)), ks=",".join(str(rng.choice([20, 40])) for _ in ns),
                bc="SSSS", prec="c64")


# ---------------------------------------------------------------- inputs
def _ks(case):
    """Wavenumbers of the case's problems: a batch draws from {k / 4, k / 2, k} in turn."""
    nb = case.get("nb", 1)
    return [case["k"]] if nb == 1 else [case["k"] / (4, 2, 1, 1)[i % 4] for i in range(nb)]


def _dhat(case, k):
    """delta_hat = k, as the configurations have it; 2 with the paper's multigrid."""
    return 2.0 if case.get("smoother") == "gmres5" else k


def _gauss(dim, n, nb, gen):
    """(nb, [z,] y, x) nodal sources: a Gaussian (sigma 0.05) at a random centre with a complex
    normal amplitude, and noise of 1e-3."""
    dev = "cuda"
    x = torch.arange(n + 1, dtype=torch.float64, device=dev) / n
    out = torch.randn((nb,) + (n + 1,) * dim, dtype=C128, device=dev, generator=gen)
    out *= 1e-3
    cen = torch.rand((nb, dim), dtype=torch.float64, device=dev, generator=gen)
    amp = torch.randn((nb,), dtype=C128, device=dev, generator=gen)
    e = torch.exp(-(x[None, None, :] - cen[:, :, None]) ** 2 / (2 * 0.05 ** 2))  # (nb, dim, n + 1)
    g = torch.einsum("ba,bc->bac", e[:, 1], e[:, 0])
    if dim == 3:
        g = torch.einsum("bz,bac->bzac", e[:, 2], g)
    out += amp.view((nb,) + (1,) * dim) * g
    return out


def _inputs(case, seed, n=None):
    """Right side b = M f, scaled to a 2-norm of 1 per problem as the Krylov vectors have it, as
    (nb, [z,] y, x) complex128 (zeros at Dirichlet nodes), and the generator for what follows."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n = case["n"] if n is None else n
    nb = case.get("nb", 1)
    ref = _Level(case["dim"], n, case["bc"])
    b = ref.apply(_gauss(case["dim"], n, nb, gen), 0.0, 1.0, 0.0)
    b /= torch.linalg.vector_norm(b.reshape(nb, -1), dim=1).view((nb,) + (1,) * case["dim"])
    return b, gen


def _jacobi_inputs(case, seed):
    b, gen = _inputs(case, seed)
    x = _gauss(case["dim"], case["n"], 1, gen) * _Level(case["dim"], case["n"], case["bc"]).mask
    return b, x


def _tags(case):
    return [hh.DIRICHLET if c == "D" else hh.SOMMERFELD for c in case["bc"]]


def _options(case, **kw):
    prec = hh.HH_C128 if case["prec"] == "c128" else hh.HH_C64
    if case.get("smoother") == "gmres5":
        kw.update(cycle_gamma=2, nu_pre=5, nu_post=5, nu_coarse=5, smoother=hh.HH_SMOOTH_GMRES)
    return hh.default_options(precision=prec, levels=LEVELS, **kw)


def prepare(case, seed):
    kind, dim = case["kind"], case["dim"]
    dt = C128 if case["prec"] == "c128" else C64
    if kind == "pack":
        problems, rhs = [], []
        for i, (n, k) in enumerate(zip(case["ns"].split(","), case["ks"].split(","))):
            n, k = int(n), float(k)
            b, _ = _inputs(case, 1000 * int(seed) + i, n)
            problems.append(hh.Problem(dim, n, k, 0.0, k, _tags(case), _options(case)))
            rhs.append(b.reshape(-1).contiguous())
        return dict(kind=kind, pack=hh.Pack(capacity=len(problems)), problems=problems, rhs=rhs)
    ks = _ks(case)
    dh = [_dhat(case, k) for k in ks]
    one = len(ks) == 1
    # single kernels and cycles need no Krylov basis to speak of; solves take the workloads' length
    restart = 1 if kind in ("vcycle", "jacobi") else (60 if dim == 3 else 30)
    p = hh.Problem(dim, case["n"], ks[0] if one else ks, 0.0, dh[0] if one else dh, _tags(case),
                   _options(case, restart=restart))
    if kind == "jacobi":
        b, x = _jacobi_inputs(case, seed)
        return dict(kind=kind, p=p, b=b.reshape(-1).to(dt), x=x.reshape(-1).to(dt))
    b, _ = _inputs(case, seed)
    b = b.reshape(-1).contiguous()
    if kind == "vcycle":
        return dict(kind=kind, p=p, b=b.to(dt))
    p.prepare()
    return dict(kind=kind, p=p, b=b)


def run(state):
    kind = state["kind"]
    if kind == "jacobi":
        return state["p"].jacobi(0, state["b"], state["x"])
    if kind == "vcycle":
        return state["p"].vcycle(state["b"])
    if kind == "precondition":
        return state["p"].precondition(state["b"])
    if kind == "solve":
        u, info = state["p"].solve(state["b"], tol=1e-8)
        return dict(u=u, outer_its=info.outer_its)
    pack, us, its = state["pack"], {}, {}
    slot = {pack.add(p, b, tol=1e-8): i for i, (p, b) in enumerate(zip(state["problems"], state["rhs"]))}
    while slot:
        for s in pack.run():
            u, info = pack.take(s)
            i = slot.pop(s)
            us[i], its[i] = u, info.outer_its
    return dict(u=[us[i] for i in range(len(us))], outer_its=[its[i] for i in range(len(its))])


def work(case):
    """Bytes: each input vector read once and each output written once.  Operations: those of the
    method (stencil applications and updates of the sweeps, residuals and HSS right sides)."""
    dim, kind = case["dim"], case["kind"]
    e = 16 if case["prec"] == "c128" else 8
    per = 40.0 if dim == 2 else 70.0  # one stencil application with its update, per node

    def cycle(n):
        nodes = [((n >> l) + 1) ** dim for l in range(LEVELS)]
        if case.get("smoother") == "gmres5":  # 5 applications and their orthogonalisation per step
            visits = [2 ** l for l in range(LEVELS)]
            return sum(v * m * (2 * (5 * per + 300.0) + per) for v, m in zip(visits, nodes))
        return per * (sum(nodes[:-1]) * 4 + nodes[-1] * 7)  # 1 + 1 + 2 stencils; 7 after the first sweep

    def hss(n, k):
        return math.ceil(k) * (cycle(n) + per * (n + 1) ** dim)

    if kind == "pack":
        pairs = [(int(n), float(k)) for n, k in zip(case["ns"].split(","), case["ks"].split(","))]
        # (the outer counts grow with k: at least about k iterations at delta_hat = k)
        return dict(bytes=sum(32.0 * (n + 1) ** 2 for n, _ in pairs), flops=sum(k * hss(n, k) for n, k in pairs))
    n = case["n"]
    N = (n + 1) ** dim
    if kind == "jacobi":
        return dict(bytes=3.0 * e * N, flops=per * N)
    if kind == "vcycle":
        return dict(bytes=2.0 * e * N, flops=cycle(n))
    if kind == "precondition":
        return dict(bytes=32.0 * N * case["nb"], flops=sum(hss(n, k) for k in _ks(case)))
    return dict(bytes=32.0 * N, flops=case["k"] * hss(n, case["k"]))


# ---------------------------------------------------------------- the same in 64 bits
class _Level:
    """One grid level: Q1 operators c_K K + c_M M + c_G M_Gamma as tensor products of 1D rows."""

    def __init__(self, dim, n, bc, dev="cuda"):
        self.dim, self.n, self.h, self.bc = dim, n, 1.0 / n, bc
        cnt = torch.full((n + 1,), 2.0, dtype=torch.float64, device=dev)
        cnt[0] = cnt[-1] = 1.0
        self.kc, self.mc = cnt / self.h, cnt * self.h / 3.0
        self.ko, self.mo = -1.0 / self.h, self.h / 6.0
        self.gc, free = [], []
        for a in range(dim):
            g, f = torch.zeros_like(cnt), torch.ones_like(cnt)
            for side, at in ((0, 0), (1, n)):
                if bc[2 * a + side] == "S":
                    g[at] = 1.0
                else:
                    f[at] = 0.0
            self.gc.append(g)
            free.append(f)
        self.mask = self._outer(free)

    def _shape(self, v, a):
        return v.reshape((-1,) + tuple(self.n + 1 if d == a else 1 for d in reversed(range(self.dim))))

    def _outer(self, vs):
        out = self._shape(vs[0], 0)
        for a in range(1, self.dim):
            out = out * self._shape(vs[a], a)
        return out

    def _row(self, v, a, centre, off):
        """(T v) along axis a with the 1D row (off, centre_i, off); off and centre may be per problem."""
        ax = v.dim() - 1 - a
        out = self._shape(centre, a) * v
        m = self.n
        s = torch.zeros_like(v)
        s.narrow(ax, 0, m).add_(v.narrow(ax, 1, m))
        s.narrow(ax, 1, m).add_(v.narrow(ax, 0, m))
        if torch.is_tensor(off):
            off = off.reshape((-1,) + (1,) * self.dim)
        out += off * s
        return out

    def _stiff(self, v, a, cK, cG):
        if not torch.is_tensor(cG):
            return self._row(v, a, cK * self.kc + cG * self.gc[a], cK * self.ko)
        return self._row(v, a, cK * self.kc[None] + cG[:, None] * self.gc[a][None], cK * self.ko)

    def apply(self, v, cK, cM, cG):
        """op v; cK real, cM and cG numbers or one per problem."""
        v = v * self.mask
        if torch.is_tensor(cM):
            cM = cM.reshape((-1,) + (1,) * self.dim)
        m, s = self._row(v, 0, self.mc, self.mo), self._stiff(v, 0, cK, cG)
        for a in range(1, self.dim):
            s = self._row(s, a, self.mc, self.mo) + self._stiff(m, a, cK, cG)
            m = self._row(m, a, self.mc, self.mo)
        return (s + cM * m) * self.mask

    def diag(self, cK, cM, cG):
        nb = cM.numel()
        m = self._shape(self.mc, 0)
        s = self._shape(cK * self.kc[None] + cG[:, None] * self.gc[0][None], 0)
        for a in range(1, self.dim):
            mc = self._shape(self.mc, a)
            s = s * mc + m * self._shape(cK * self.kc[None] + cG[:, None] * self.gc[a][None], a)
            m = m * mc
        return s + cM.reshape((nb,) + (1,) * self.dim) * m

    def dense(self, cK, cM, cG, a):
        """1D matrices of axis a on its free nodes: c_K K + c_G G, M."""
        k = torch.diag((cK * self.kc + cG * self.gc[a]).to(C128))
        m = torch.diag(self.mc.to(C128))
        i = torch.arange(self.n, device=k.device)
        for t, o in ((k, cK * self.ko), (m, self.mo)):
            t[i, i + 1] = t[i + 1, i] = o
        lo = 1 if self.bc[2 * a] == "D" else 0
        hi = self.n if self.bc[2 * a + 1] == "D" else self.n + 1
        return k[lo:hi, lo:hi], m[lo:hi, lo:hi], lo, hi


class _Method:
    """Multigrid cycles and HSS steps for problems k, delta_hat (tensors, one entry per problem)."""

    def __init__(self, case, ks, dhs):
        dim = case["dim"]
        self.lv = [_Level(dim, case["n"] >> l, case["bc"]) for l in range(LEVELS)]
        self.ks = torch.tensor(ks, dtype=torch.float64, device="cuda")
        dh = torch.tensor(dhs, dtype=torch.float64, device="cuda")
        k = self.ks
        self.AL = (1.0, torch.complex(dh * dh - k * k, -2 * dh * k * k), torch.complex(dh, -k * k))
        self.AR = (-1.0, torch.complex(k * k - dh * dh, -2 * dh * k * k), torch.complex(-dh, -k * k))
        omega = 0.6 if dim == 2 else 0.5
        self.wd = [omega / l.diag(*self.AL) for l in self.lv]
        self.gm = case.get("smoother") == "gmres5"

    def A(self, l, x):
        return self.lv[l].apply(x, *self.AL)

    def sweeps(self, l, b, x, nu):
        if self.gm:
            return self.gmres(l, b, x, nu)
        for _ in range(nu):
            r = b * self.lv[l].mask if x is None else b - self.A(l, x)
            x = (0 if x is None else x) + self.wd[l] * r * self.lv[l].mask
        return x

    def gmres(self, l, b, x, its):
        r = b if x is None else b - self.A(l, x)
        r = self.wd[l] * r * self.lv[l].mask
        beta = torch.linalg.vector_norm(r)
        V, H = [r / beta], torch.zeros((its + 1, its), dtype=C128, device=r.device)
        for j in range(its):
            w = self.wd[l] * self.A(l, V[j])
            B = torch.stack([v.reshape(-1) for v in V])
            wf = w.reshape(-1)
            for _ in range(2):
                c = B.conj() @ wf
                H[: j + 1, j] += c
                wf = wf - c @ B
            h = torch.linalg.vector_norm(wf)
            H[j + 1, j] = h
            V.append((wf / h).reshape(r.shape))
        rhs = torch.zeros((its + 1, 1), dtype=C128, device=r.device)
        rhs[0] = beta
        y = torch.linalg.lstsq(H, rhs).solution[:, 0]
        d = sum(y[j] * V[j] for j in range(its))
        return d if x is None else x + d

    def restrict(self, l, r):
        for a in range(r.dim() - 1):
            ax = r.dim() - 1 - a
            m = r.shape[ax] // 2
            idx = torch.arange(0, 2 * m + 1, 2, device=r.device)
            odd = r.index_select(ax, idx[:-1] + 1)
            c = r.index_select(ax, idx).clone()
            c.narrow(ax, 0, m).add_(odd, alpha=0.5)
            c.narrow(ax, 1, m).add_(odd, alpha=0.5)
            r = c
        return r * self.lv[l + 1].mask

    def prolong(self, l, e):
        e = e * self.lv[l + 1].mask
        for a in range(e.dim() - 1):
            ax = e.dim() - 1 - a
            m = e.shape[ax] - 1
            shape = list(e.shape)
            shape[ax] = 2 * m + 1
            f = torch.zeros(shape, dtype=e.dtype, device=e.device)
            at = torch.arange(0, 2 * m + 1, 2, device=e.device)
            f.index_copy_(ax, at, e)
            f.index_copy_(ax, at[:-1] + 1, 0.5 * (e.narrow(ax, 0, m) + e.narrow(ax, 1, m)))
            e = f
        return e * self.lv[l].mask

    def cycle(self, l, b):
        if l == LEVELS - 1:
            return self.sweeps(l, b, None, 5 if self.gm else 8)
        nu = 5 if self.gm else 2
        x = self.sweeps(l, b, None, nu)
        rc = self.restrict(l, (b - self.A(l, x)) * self.lv[l].mask)
        e = self.cycle(l + 1, rc)
        if self.gm:  # W-cycle: one more cycle on what the first leaves
            e = e + self.cycle(l + 1, rc - self.A(l + 1, e))
        return self.sweeps(l, b, x + self.prolong(l, e), nu)

    def hss(self, r):
        nb = self.ks.numel()
        shape = (nb,) + (1,) * (r.dim() - 1)
        c1 = ((self.ks - 1) / (self.ks + 1)).reshape(shape)
        c2 = (2 * self.ks / (self.ks + 1)).reshape(shape)
        steps = torch.ceil(self.ks - 1e-9 * self.ks).to(torch.int64)
        u = torch.zeros_like(r)
        for it in range(int(steps.max())):
            new = self.cycle(0, c1 * self.lv[0].apply(u, *self.AR) + c2 * r)
            u = torch.where((steps > it).reshape(shape), new, u)
        return u * self.lv[0].mask


def _direct(case, n, k, b):
    """u with B u = b by block elimination along the slowest axis (B = K - k^2 M - i k M_Gamma)."""
    lv = _Level(case["dim"], n, case["bc"])
    cK, cM, cG = 1.0, complex(-k * k), complex(0.0, -k)
    S, M, lo, hi = lv.dense(cK, cM, cG, 0)
    cut = [(lo, hi)]
    for a in range(1, case["dim"]):
        Sa, Ma, lo, hi = lv.dense(cK, cM, cG, a)
        cut.append((lo, hi))
        if a < case["dim"] - 1:
            S, M = torch.kron(Ma, S) + torch.kron(Sa, M), torch.kron(Ma, M)
    X = S + cM * M
    f = b[0]
    for ax, (lo, hi) in enumerate(reversed(cut)):
        f = f.narrow(ax, lo, hi - lo)
    m = f.shape[0]
    f = f.reshape(m, -1)
    O = Ma[0, 1] * X + Sa[0, 1] * M
    G, y = [], []
    for j in range(m):
        D = Ma[j, j] * X + Sa[j, j] * M
        r = f[j]
        if j:
            D = D - O @ G[-1]
            r = r - O @ y[-1]
        sol = torch.linalg.solve(D, torch.cat([O, r[:, None]], 1))
        G.append(sol[:, :-1])
        y.append(sol[:, -1])
    u = torch.zeros_like(b[0])
    v = u
    for ax, (lo, hi) in enumerate(reversed(cut)):
        v = v.narrow(ax, lo, hi - lo)
    x = [None] * m
    for j in reversed(range(m)):
        x[j] = y[j] if j == m - 1 else y[j] - G[j] @ x[j + 1]
    v.copy_(torch.stack(x).reshape(v.shape))
    return u.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "pack":
        us = []
        for i, (n, k) in enumerate(zip(case["ns"].split(","), case["ks"].split(","))):
            b, _ = _inputs(case, 1000 * int(seed) + i, int(n))
            us.append(_direct(case, int(n), float(k), b))
        return dict(u=us, outer_its=[None] * len(us))
    if kind == "solve":
        b, _ = _inputs(case, seed)
        return dict(u=_direct(case, case["n"], case["k"], b), outer_its=None)
    lo = (lambda v: v) if case["prec"] == "c128" else (lambda v: v.to(C64).to(C128))
    ks = _ks(case)
    m = _Method(case, ks, [_dhat(case, k) for k in ks])
    if kind == "jacobi":
        b, x = _jacobi_inputs(case, seed)
        return m.sweeps(0, lo(b), lo(x), 1).reshape(-1)
    b, _ = _inputs(case, seed)
    if kind == "vcycle":
        return m.cycle(0, lo(b)).reshape(-1)
    return m.hss(b).reshape(-1)
