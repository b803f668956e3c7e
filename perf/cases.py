"""The solves whose speed this library is measured by.

A case is one pass of a program that uses the library through ``RomContext``: draw the
pass's random ordinate sets (plain DOM: the set is already there), solve, read the flux.
The context, with its grid, kernel and options, is what such a program keeps between
passes.  The sweeps run in FP32, so the flux is kept as FP32 once it is read.

``exact`` is the same source iteration in 64 bits in plain torch, written from the cell
equations, with none of the library's code.
"""
import math

import numpy as np
import torch

from paper_2407_12527_gb300 import KERNEL_FLAG_NORMALIZE, RomContext

FACES = ("xl", "xr", "yb", "yt")
DEVICE = "cuda"


def _case(name, **kw):
    """Defaults of every field: a 2D isotropic ROM solve with the library's own options.

    m: ordinates per quadrant (octant in 3D) and sample, 0 = uneven, drawn per sample from
    {2, 4, 8, 16}; quad: a DOM set in their place; fixed: sweeps run, 0 = to ``tol``, where
    ``sweeps`` says about how many that takes; precision: the dense operator's product."""
    c = dict(dim=2, I=32, J=32, K=1, medium="box", kernel="iso", g=0.0, samples=1, m=4, quad="",
             n1=0, n2=0, scheme="dd", tol=1e-6, fixed=0, sweeps=0, tile_g=0, precision=0,
             inflow=False)
    c.update(kw)
    if c["fixed"]:
        c["sweeps"] = c["fixed"]
    c["name"] = name
    return c


def listed():
    return [
        # plain DOM on a small grid: the shortest solve, all latency and launches
        _case("dom_32", I=32, J=32, quad="product_gl", n1=4, n2=8, sweeps=10),
        # Example 2.1 with the 16 random sets of 36 ordinates of the ray-effect study
        _case("example_100", I=100, J=100, samples=16, m=9, sweeps=10),
        # the same problem with the linear kernel, a batch of the error tables' samples
        _case("example_linear_100", I=100, J=100, kernel="linear", g=0.9, samples=256, m=4,
              sweeps=10),
        # the benchmark's default: point source, 64 samples of 16, measured work-item shape
        _case("point_source_256", I=256, J=256, medium="gauss", samples=64, m=4, tile_g=-1,
              sweeps=25),
        # plain DOM on the same problem: one sample, 256 ordinates
        _case("point_source_dom_256", I=256, J=256, medium="gauss", quad="uniform", n1=8,
              sweeps=25),
        # heterogeneous blocks, 256 samples of uneven size, measured work-item shape
        _case("checkerboard_448", I=448, J=448, medium="checker", samples=256, m=0, tile_g=-1,
              sweeps=26),
        # ragged heterogeneous grid lit through its faces, positive (step) scheme
        _case("inflow_step_211x173", I=211, J=173, medium="random", samples=24, m=8,
              scheme="step", inflow=True, fixed=20),
        # several problems in one batch, each with its own grid and samples of uneven size
        _case("mixed_grids", I=200, J=160, medium="grids", samples=48, m=0, fixed=15),
        # Henyey-Greenstein (rows normalised), dense operator on the tensor cores
        _case("hg_disc_512", I=512, J=512, medium="disc", kernel="hg", g=0.8, samples=32, m=32,
              precision=1, sweeps=16),
        # the same kernel on a smaller ragged grid with the FP32 product
        _case("hg_fp32_150x130", I=150, J=130, medium="disc", kernel="hg", g=0.8, samples=8, m=12,
              fixed=12),
        # 3D lognormal medium, 64 samples of 48 ordinates
        _case("lognormal_128", dim=3, I=128, J=128, K=128, medium="lognormal", samples=64, m=6,
              sweeps=11),
        # a small ragged 3D grid
        _case("cube_45x38x52", dim=3, I=45, J=38, K=52, medium="lognormal", samples=8, m=4,
              fixed=10),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["rom", "rom", "rom", "rom", "dom", "grids", "dense", "cube"])
        if kind in ("rom", "grids", "dom"):
            I, J = size(24, 512), size(24, 512)
            kw = dict(I=I, J=J, fixed=rng.randint(6, 30), samples=size(1, 256),
                      m=rng.choice([0, 2, 3, 4, 6, 9, 16]),
                      medium=rng.choice(["box", "gauss", "checker", "random"]),
                      scheme=rng.choice(["dd", "dd", "dd", "step"]), tile_g=rng.choice([0, -1]),
                      inflow=rng.random() < 0.2)
            if rng.random() < 0.25:
                kw.update(kernel="linear", g=round(rng.uniform(0.2, 0.95), 2))
            if kind == "dom":
                kw.update(samples=1, m=4, quad=rng.choice(["uniform", "gauss"]),
                          n1=rng.randint(2, 16))
            if kind == "grids":
                kw.update(medium="grids", inflow=False, samples=max(3, kw["samples"]))
        elif kind == "dense":
            kw = dict(I=size(32, 512), J=size(32, 512), medium="disc", kernel="hg",
                      g=round(rng.uniform(0.2, 0.6), 2), samples=size(2, 32),
                      m=rng.choice([6, 8, 12, 16, 24, 32]), precision=rng.choice([0, 1]),
                      fixed=rng.randint(6, 20))
        else:
            kw = dict(dim=3, I=size(20, 128), J=size(20, 128), K=size(20, 128),
                      medium="lognormal", samples=size(1, 64), m=rng.choice([1, 2, 4, 6]),
                      fixed=rng.randint(4, 12))
        c = _case("", **kw)
        del c["name"]
        if 2e6 < _updates(c) < 3e10 and work(c)["flops"] < 3e11:
            return c


# ------------------------------------------------------------------ inputs

def _partition(m):
    nz = max(d for d in range(1, int(math.sqrt(m)) + 1) if m % d == 0)
    return nz, m // nz


def _partitions(c, seed):
    """(n_zeta, n_theta) of each sample."""
    if c["m"]:
        ms = [c["m"]] * c["samples"]
    else:  # uneven: a shuffled, even share of each size, so that the work is the same
        ms = [(2, 4, 8, 16)[k % 4] for k in range(c["samples"])]
        np.random.default_rng(seed + 31).shuffle(ms)
    return [_partition(m) for m in ms]


def _ordinate_count(c):
    """Ordinates of all samples."""
    if c["quad"] == "uniform":
        return 4 * c["n1"] ** 2
    if c["quad"] == "gauss":
        return 2 * c["n1"] * (c["n1"] + 1)
    if c["quad"] == "product_gl":
        return c["n1"] * c["n2"]
    return (8 if c["dim"] == 3 else 4) * sum(a * b for a, b in _partitions(c, 0))


def _extent(c):
    """(x_L, x_R, y_B, y_T, ...): cells of the first problem's width along every axis."""
    if c["medium"] == "gauss":
        return (-1.0, 1.0, -1.0, 1.0)
    if c["medium"] == "checker":
        return (0.0, 7.0, 0.0, 7.0)
    return (0.0, 1.0) * c["dim"]


def _grids(c, seed):
    """[(I, J, bounds, sigma_t, sigma_s, q, samples)]: the grids of a batch of problems."""
    rng = np.random.default_rng(seed)
    S, out = c["samples"], []
    share = [S // 3, S // 3, S - 2 * (S // 3)]
    for p, (I, J) in enumerate([(c["I"], c["J"]), (max(8, c["I"] // 2), max(8, c["J"] * 3 // 4)),
                                (max(8, c["I"] // 3 + 1), max(8, c["J"] // 2 + 1))]):
        st, ss, q = _blotches(I, J, rng)
        out.append((I, J, (0.0, 1.0 + 0.5 * p, 0.0, 1.0), st, ss, q, share[p]))
    return out


def _blotches(I, J, rng):
    """A heterogeneous medium [J, I]: independent sigma_T, sigma_S and q per cell."""
    st = rng.uniform(0.5, 4.0, size=(J, I))
    return st, st * rng.uniform(0.0, 0.9, size=(J, I)), rng.uniform(0.0, 2.0, size=(J, I))


def _medium(c, seed):
    """(sigma_t, sigma_s, q), FP64, [J, I] or [K, J, I]."""
    rng = np.random.default_rng(seed)
    I, J, K = c["I"], c["J"], c["K"]
    if c["medium"] == "lognormal":
        noise = torch.from_numpy(rng.standard_normal((K, J, I)))
        f = torch.fft.rfftn(noise)
        for axis, n in enumerate((K, J, I)):  # covariance exp(-r^2 / (2 * 8^2)) cells
            d = torch.minimum(torch.arange(n), n - torch.arange(n)).double()
            k = torch.fft.rfft(torch.exp(-d * d / 64)) if axis == 2 else torch.fft.fft(
                torch.exp(-d * d / 64))
            f = f * k.reshape([-1 if a == axis else 1 for a in range(3)])
        G = torch.fft.irfftn(f, s=(K, J, I), dim=(0, 1, 2)).numpy()
        G = (G - G.mean()) / G.std()
        st = np.exp(-0.125 + 0.5 * G)
        q = np.zeros((K, J, I))
        lo = [n // 2 - max(1, n // 32) for n in (K, J, I)]
        hi = [n // 2 + max(1, n // 32) for n in (K, J, I)]
        q[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] = rng.uniform(0.8, 1.2)
        return st, 0.8 * st, q
    if c["medium"] == "random":
        return _blotches(I, J, rng)
    xl, xr, yb, yt = _extent(c)[:4]
    X, Y = np.meshgrid(xl + (np.arange(I) + 0.5) * (xr - xl) / I,
                       yb + (np.arange(J) + 0.5) * (yt - yb) / J, indexing="xy")
    one = np.ones((J, I))
    amp = rng.uniform(0.8, 1.2)
    if c["medium"] == "box":
        return one, 0.5 * one, np.where((abs(X - 0.5) < 0.1) & (abs(Y - 0.5) < 0.1), 2.0 * amp, 0.0)
    if c["medium"] == "gauss":
        s = max(0.02, 1.0 / min(I, J))
        return one, 0.9 * one, amp * np.exp(-(X * X + Y * Y) / (2 * s * s))
    if c["medium"] == "disc":
        return one, 0.95 * one, np.where((X - 0.5) ** 2 + (Y - 0.5) ** 2 <= 0.05 ** 2, amp, 0.0)
    bi, bj = np.floor(X).astype(int), np.floor(Y).astype(int)  # checker: 7 x 7 blocks
    centre = (bi == 3) & (bj == 3)
    absorber = ((bi + bj) % 2 == 0) & ~centre
    return np.where(absorber, 10.0, 1.0), np.where(absorber, 0.0, 0.9), np.where(centre, amp, 0.0)


def _inflow(c, seed):
    """Isotropic incoming flux per face cell, x_L, x_R, y_B, y_T."""
    rng = np.random.default_rng(seed + 7)
    return [rng.uniform(0.0, 1.0, size=n) for n in (c["J"], c["J"], c["I"], c["I"])]


class _State:
    pass


def prepare(case, seed):
    c = case
    s = _State()
    s.case = c
    s.seed = 1000 + seed
    s.stream = torch.cuda.Stream()
    ctx = s.ctx = RomContext(torch.cuda.current_device())
    ctx.set_stream(s.stream.cuda_stream)
    if c["medium"] == "grids":
        grids = _grids(c, seed)
        ctx.set_grids([g[:6] for g in grids], [g[6] for g in grids])
    elif c["dim"] == 3:
        ctx.set_grid3(c["I"], c["J"], c["K"], _extent(c), *_medium(c, seed))
    else:
        ctx.set_grid(c["I"], c["J"], _extent(c), *_medium(c, seed))
    if c["inflow"]:
        for face, v in zip(FACES, _inflow(c, seed)):
            ctx.set_inflow_isotropic(face, v)
    if c["kernel"] != "iso":
        # Henyey-Greenstein with normalised rows: few ordinates resolve its peak so badly that
        # the raw operator can make the source iteration diverge
        ctx.set_kernel(c["kernel"], c["g"], KERNEL_FLAG_NORMALIZE if c["kernel"] == "hg" else 0)
    ctx.set_options(scheme=c["scheme"], tol=c["tol"], fixed_iters=c["fixed"], tile_g=c["tile_g"],
                    dense_precision=c["precision"])
    if c["quad"]:
        ctx.set_quadrature(c["quad"], c["n1"], c["n2"])
    else:
        parts = _partitions(c, seed)
        s.nz, s.nt = [a for a, _ in parts], [b for _, b in parts]
    if c["medium"] != "grids":
        shape = (c["K"], c["J"], c["I"]) if c["dim"] == 3 else (c["J"], c["I"])
        s.flux = torch.empty(shape, dtype=torch.float64, device="cuda")
    return s


def run(state):
    ctx, c = state.ctx, state.case
    if not c["quad"]:
        if c["dim"] == 3:
            ctx.set_ordinates_seed_xyz(state.seed, state.nz, state.nt)
        else:
            ctx.set_ordinates_seed(state.seed, state.nz, state.nt)
    ctx.solve()
    if c["medium"] == "grids":
        return [ctx.grid_average(p).astype(np.float32) for p in range(3)]
    ctx.scalar_flux_device(state.flux)
    with torch.cuda.stream(state.stream):
        return state.flux.float()


# -------------------------------------------------------------------- work

def _cells(c):
    if c["medium"] == "grids":
        return sum(g[0] * g[1] * g[6] for g in _grids(c, 0)) / c["samples"]
    return c["I"] * c["J"] * c["K"]


def _updates(c):
    return float(_cells(c)) * _ordinate_count(c) * c["sweeps"]


def work(case):
    """Flops of the cell updates of every sweep (diamond difference: the source and the two or
    three incoming fluxes, the division, the outgoing fluxes, the moment), of the dense
    operator's product where there is one; bytes of the coefficients in and the flux out."""
    c = case
    uniform = c["medium"] in ("box", "gauss", "disc")
    per = (8 if uniform else 11) if c["dim"] == 2 else 14
    if c["kernel"] == "linear":
        per += 6
    if c["kernel"] == "hg":
        per += 2 * 4 * c["m"]
    return {"bytes": _cells(c) * (3 if c["medium"] == "grids" else 1) * (3 * 4 + 8),
            "flops": _updates(c) * per}


# ------------------------------------------------------------------- exact

def _u01(seed, n):
    """SplitMix64 output n of `seed` as a number in [0, 1): its top 53 bits."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (n + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _first_quadrant(c, seed, first, count):
    """(|c|, |s|, |zeta|, w, sample) of samples first .. first + count - 1, the ordinates of
    the first quadrant (octant): every set is symmetric under the reflections."""
    if c["quad"]:
        n = c["n1"]
        if c["quad"] == "uniform":
            i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
            zeta, theta = (2 * n - 2 * i - 1) / (2.0 * n), (2 * j + 1) * np.pi / (4 * n)
            w = np.full(n * n, 1.0 / (4 * n * n))
        else:
            x, wx = np.polynomial.legendre.leggauss(2 * (n if c["quad"] == "gauss" else c["n1"]))
            x, wx = x[x > 0][::-1], wx[x > 0][::-1]
            per = [i + 1 for i in range(n)] if c["quad"] == "gauss" else [c["n2"] // 4] * n
            zeta = np.concatenate([[x[i]] * k for i, k in enumerate(per)])
            theta = np.concatenate([(2 * np.arange(k) + 1) * np.pi / (4 * k) for k in per])
            w = np.concatenate([[wx[i] / (4 * k)] * k for i, k in enumerate(per)])
        zeta, theta = zeta.reshape(-1), theta.reshape(-1)
        sid = np.zeros(zeta.size, dtype=np.int64)
    else:
        z_, t_, w_, s_ = [], [], [], []
        for k, (nz, nt) in list(enumerate(_partitions(c, seed)))[first:first + count]:
            cell = np.arange(nz * nt, dtype=np.uint64)
            ctr = (np.uint64(k) << np.uint64(32)) | (cell << np.uint64(1))
            i, j = (cell // np.uint64(nt)).astype(float), (cell % np.uint64(nt)).astype(float)
            z_.append((nz - 1 - i + _u01(1000 + seed, ctr)) / nz)
            t_.append((j + _u01(1000 + seed, ctr | np.uint64(1))) * np.pi / (2 * nt))
            w_.append(np.full(nz * nt, 1.0 / ((8 if c["dim"] == 3 else 4) * nz * nt)))
            s_.append(np.full(nz * nt, k - first))
        zeta, theta, w, sid = (np.concatenate(v) for v in (z_, t_, w_, s_))
    rho = np.sqrt(1 - zeta * zeta)
    return [torch.from_numpy(np.ascontiguousarray(v)).to(DEVICE) for v in
            (rho * np.cos(theta), rho * np.sin(theta), zeta, w, sid)]


class _Exact:
    """Source iteration of one grid's samples in 64 bits.  Cells (k, j) of one step t are those
    with i + j + k = t: the arrays are padded along i, so that a step is one strided view."""

    def __init__(self, c, seed, I, J, K, bounds, st, ss, q, first, count):
        self.c, self.I, self.J, self.K, self.S = c, I, J, K, count
        self.dim3 = c["dim"] == 3
        n = [I, J, K][:c["dim"]]
        f = 2.0 if c["scheme"] == "dd" else 1.0
        mu = _first_quadrant(c, seed, first, count)
        self.mu, self.w, self.sid = mu[:3], mu[3], mu[4]
        self.n = self.w.numel()
        self.coef = [f * m / ((bounds[2 * d + 1] - bounds[2 * d]) / n[d])
                     for d, m in enumerate(mu[:c["dim"]])]
        signs = [(x, y, z) for z in ((1, -1) if self.dim3 else (1,)) for y in (1, -1)
                 for x in (1, -1)]
        # the quadrants at once in 2D, one octant at a time in 3D
        self.groups = [[s] for s in signs] if self.dim3 else [signs]
        self.even = bool((torch.bincount(self.sid) == self.n // count).all())
        self.T0 = J - 1 + K - 1
        as64 = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(DEVICE).reshape(K, J, I)  # noqa: E731
        # what the library is given: FP64 coefficients, kept in FP32
        self.st, self.ss, self.q = (as64(v).float().double() for v in (st, ss, q))
        self.uniform = bool((self.st == self.st.flatten()[0]).all())
        self.face = [torch.from_numpy(v).to(DEVICE).float().double() for v in _inflow(c, seed)] if c["inflow"] else None

    def flip(self, v, sign):
        dims = [d for d, s in zip((-1, -2, -3), sign) if s < 0]
        return v.flip(dims) if dims else v

    def skewed(self, v, t):
        """Cells of step t of v [..., K, J, I + 2 T0]."""
        st = list(v.stride())
        st[-3], st[-2] = st[-3] - 1, st[-2] - 1
        return v.as_strided(v.shape[:-1], st[:-1], self.T0 + t)

    def pad(self, v):
        return torch.nn.functional.pad(v, (self.T0, self.T0))

    def sweep(self, src, mom):
        """src: the source moments [S, K, J, I], or (mom = 0) by sign every ordinate's source
        [n, K, J, I].  Returns the flux moments, and (mom = 0) psi by sign."""
        c, I, J, K, S, n = self.c, self.I, self.J, self.K, self.S, self.n
        step = c["scheme"] == "step"
        co = [v.reshape(1, n, 1, 1) for v in self.coef]
        total = None
        psis = {}
        for signs in self.groups:
            Q = len(signs)
            if mom:
                srcs = [torch.stack([self.pad(self.flip(v, s)) for s in signs]) for v in src]
            else:
                per = torch.stack([self.pad(self.flip(src[s], s)) for s in signs])
                out = torch.zeros_like(per)
            acc = [torch.zeros((Q, S, K, J, I + 2 * self.T0), dtype=torch.float64, device=DEVICE)
                   for _ in range(mom or 1)]
            sx = torch.tensor([float(s[0]) for s in signs], device=DEVICE).double().reshape(Q, 1, 1, 1)
            sy = torch.tensor([float(s[1]) for s in signs], device=DEVICE).double().reshape(Q, 1, 1, 1)
            ww = self.w.reshape(1, n, 1, 1)
            wm = [ww]
            if mom == 3:
                cx, cy = sx * self.mu[0].reshape(1, n, 1, 1), sy * self.mu[1].reshape(1, n, 1, 1)
                wm = [ww, ww * cx, ww * cy]
            if self.uniform:
                r = 1.0 / (self.st.flatten()[0] + sum(co))
            else:
                sig = torch.nn.functional.pad(
                    torch.stack([self.flip(self.st, s) for s in signs]),
                    (self.T0, self.T0), value=1.0).unsqueeze(1)
            X, Y, Y2, Z, Z2 = (torch.zeros((Q, n, K, J), dtype=torch.float64, device=DEVICE)
                               for _ in range(5))
            for t in range(I + self.T0):
                if self.face is not None:
                    if t < J:
                        X[:, :, 0, t] = torch.stack(
                            [(self.face[0] if s[0] > 0 else self.face[1])[t if s[1] > 0 else J - 1 - t]
                             for s in signs]).reshape(Q, 1)
                    if t < I:
                        Y[:, :, 0, 0] = torch.stack(
                            [(self.face[2] if s[1] > 0 else self.face[3])[t if s[0] > 0 else I - 1 - t]
                             for s in signs]).reshape(Q, 1)
                if mom == 0:
                    num = torch.addcmul(self.skewed(per, t), co[0], X)
                else:
                    v = [self.skewed(m, t) for m in srcs]
                    s0 = (v[0].repeat_interleave(n // S, 1) if self.even
                          else v[0].index_select(1, self.sid))
                    if mom == 3:
                        s0 = s0 + cx * v[1].index_select(1, self.sid) + cy * v[2].index_select(1, self.sid)
                    num = torch.addcmul(s0, co[0], X)
                num.addcmul_(co[1], Y)
                if self.dim3:
                    num.addcmul_(co[2], Z)
                psi = num.mul_(r) if self.uniform else num.div_(self.skewed(sig, t) + sum(co))
                if mom == 0:
                    self.skewed(out, t).copy_(psi)
                for a, wq in zip(acc, wm):
                    p = psi * wq
                    if self.even:
                        self.skewed(a, t).add_(p.reshape(Q, S, n // S, K, J).sum(2))
                    else:
                        self.skewed(a, t).index_add_(1, self.sid, p)
                # the edges on: x along the row, y and z to the next row and plane
                two = psi if step else psi.mul_(2)
                for old, new, lo, hi in ((X, X, np.s_[:], np.s_[:]),
                                         (Y, Y2, np.s_[..., 1:], np.s_[..., :-1]),
                                         (Z, Z2, np.s_[:, :, 1:], np.s_[:, :, :-1]))[:c["dim"]]:
                    if step:
                        new[lo].copy_(two[hi])
                    else:
                        torch.sub(two[hi], old[hi], out=new[lo])
                Y, Y2, Z, Z2 = Y2, Y, Z2, Z
            cut = slice(self.T0, self.T0 + I)
            part = [sum(self.flip(a[k][..., cut], s) for k, s in enumerate(signs)) for a in acc]
            total = part if total is None else [x + y for x, y in zip(total, part)]
            if mom == 0:
                for k, s in enumerate(signs):
                    psis[s] = self.flip(out[k][..., cut], s)
        return (total, psis) if mom == 0 else total

    def operator(self):
        """A[l][l'] = w_l' P(u_l', u_l), rows normalised, the Henyey-Greenstein kernel averaged
        over the mirror image in zeta; ordinates in the order of the signs, then of the first
        quadrant."""
        signs, m = self.groups[0], self.n // self.S
        g = self.c["g"]
        cx = torch.stack([s[0] * self.mu[0].reshape(self.S, m) for s in signs], 1).reshape(self.S, -1)
        cy = torch.stack([s[1] * self.mu[1].reshape(self.S, m) for s in signs], 1).reshape(self.S, -1)
        z = self.mu[2].reshape(self.S, 1, m).expand(-1, 4, -1).reshape(self.S, -1)
        w = self.w.reshape(self.S, 1, m).expand(-1, 4, -1).reshape(self.S, -1)
        flat = cx[:, :, None] * cx[:, None] + cy[:, :, None] * cy[:, None]
        zz = z[:, :, None] * z[:, None]
        G = lambda v: (1 - g * g) / (1 + g * g - 2 * g * v) ** 1.5  # noqa: E731
        A = 0.5 * (G(flat + zz) + G(flat - zz)) * w[:, None]
        return A / A.sum(2, keepdim=True)

    def solve(self):
        c, S, n = self.c, self.S, self.n
        shape = (S, self.K, self.J, self.I)
        phi = torch.zeros(shape, dtype=torch.float64, device=DEVICE)
        mom = {"iso": 1, "linear": 3, "hg": 0}[c["kernel"]]
        q = self.q.expand(shape).contiguous()
        if mom == 0:
            signs, m = self.groups[0], n // S
            A = self.operator()
            src = {s: self.q.expand((n,) + shape[1:]) for s in signs}
        else:
            src = [q] + [torch.zeros_like(q) for _ in range(mom - 1)]
        active = torch.ones(S, dtype=torch.bool, device=DEVICE)
        for it in range(c["fixed"] or 10000):
            if mom == 0:
                (new,), psis = self.sweep(src, 0)
            else:
                res = self.sweep(src, mom)
                new = res[0]
            keep = active.reshape(S, 1, 1, 1)
            d = (new - phi).flatten(1).norm(dim=1)
            nn = new.flatten(1).norm(dim=1)
            phi = torch.where(keep, new, phi)
            if not c["fixed"]:
                active = active & ~(d < c["tol"] * nn)
                if not bool(active.any()):
                    break
            if mom == 0:
                psi = torch.stack([psis[s].reshape(S, m, -1) for s in signs], 1).reshape(S, 4 * m, -1)
                del psis
                s2 = torch.empty_like(psi)
                for k in range(S):
                    torch.matmul(A[k], psi[k], out=s2[k])
                del psi
                s2 = s2.mul_(self.ss.reshape(1, 1, -1)).add_(self.q.reshape(1, 1, -1))
                s2 = s2.reshape((S, 4, m) + shape[1:])
                src = {s: s2[:, k].reshape((n,) + shape[1:]) for k, s in enumerate(signs)}
            else:
                src = [self.ss * new + self.q] + [c["g"] * self.ss * v for v in
                                                  (res[1:] if mom == 3 else [])]
        return phi.mean(0)


def _seconds(c):
    """About how long `exact` takes: launches of a step, or its arrays' bytes."""
    steps = (c["I"] + c["J"] + c["K"]) * (8 if c["dim"] == 3 else 1)
    n = _ordinate_count(c) * (1 / 8 if c["dim"] == 3 else 1) * c["J"] * c["K"] * 8
    ops = 14 + (12 if c["kernel"] == "linear" else 0)
    s = c["sweeps"] * steps * ops * max(8e-6, 3 * n / 4e12)
    return s + (_updates(c) * 8 * c["m"] / 0.8e12 if c["kernel"] == "hg" else 0)


def exact(case, seed):
    c = case
    if _seconds(c) > 20:
        return None
    if c["medium"] == "grids":
        out, first = [], 0
        for I, J, b, st, ss, q, count in _grids(c, seed):
            out.append(_Exact(c, seed, I, J, 1, b, st, ss, q, first, count).solve()[0])
            first += count
        return out
    phi = _Exact(c, seed, c["I"], c["J"], c["K"], _extent(c), *_medium(c, seed), 0,
                 c["samples"]).solve()
    return phi if c["dim"] == 3 else phi[0]
