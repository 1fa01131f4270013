"""The work that this framework is measured on, through its public entry points.

Each case is one call (or the few calls of one layer) that a user's program makes
again and again: WaveHoltz applies S v on the grids, orders, precisions and media
of the named workloads, two whole Krylov solves, a batch of shots, and the layers of
the warm-start network.  Sizes are those of the configurations, tests and benchmark
of this repository (64, 256..512 and 1024 squares, 48..256 cubes, 256 x 256
images); ragged ones stand for grids that no tile divides.

Results of the FP32-stencil form carry 32-bit accuracy in the solver's 64-bit
vectors; a program that keeps the wave fields of many shots stores them in 32
bits, so the cases of that form return them so.  FP64 results are returned as
they come.

``exact`` restates the method in plain torch, 64 bits, on whole grids: the
discrete operators from their energy forms (order 2: edges and centred
differences; order 4: summation by parts, also on mapped grids), the corrected
leapfrog with its Taylor start, the trapezoidal filter and CG.
"""
import math

import numpy as np
import torch

from paper_2205_12344_gb300 import _lib as L
from paper_2205_12344_gb300 import inputs
from paper_2205_12344_gb300.api import WaveHoltz, WaveHoltzBatch

VS_SPAN = 0.6  # largest |log Vs| of the smooth random media (three standard deviations of 0.2)


def listed():
    return [
        # the smallest problem of the repository (64 x 64, order 2, FP64): one operator
        # apply, where a level is a few microseconds of latency
        dict(name="apply_homog2d_64_f64", kind="apply", medium="homogeneous", nx=64, ny=64, nz=0, order=2,
             precision="fp64", sides="dirichlet", nrhs=1, ppw=0.0, mapped=False),
        # the same problem solved: CG to 1e-8, the call a new user makes first
        dict(name="solve_homog2d_64_f64", kind="solve", medium="homogeneous", nx=64, ny=64, nz=0, order=2,
             precision="fp64", sides="dirichlet", nrhs=1, ppw=0.0, mapped=False, tol=1e-8, maxit=200),
        # the layered seismic section, FP32 stencil: the operator apply of every CG
        # iteration of the benchmark
        dict(name="apply_layered2d_1024_f32", kind="apply", medium="layered", nx=1024, ny=1025, nz=0, order=4,
             precision="fp32", sides="free_top", nrhs=1, ppw=10.0, mapped=False),
        # the same section in FP64: right-hand sides, residual replacements and every
        # iteration of a plain FP64 solve
        dict(name="apply_layered2d_1024_f64", kind="apply", medium="layered", nx=1024, ny=1025, nz=0, order=4,
             precision="fp64", sides="free_top", nrhs=1, ppw=10.0, mapped=False),
        # a few CG iterations of the mixed-precision solve from a cold start (FP64 right-hand
        # side, FP32 iterations, FP64 residuals), as a frequency sweep makes them
        dict(name="solve_layered2d_384_f32", kind="solve", medium="layered", nx=384, ny=385, nz=0, order=4,
             precision="fp32", sides="free_top", nrhs=1, ppw=10.0, mapped=False, tol=1e-6, maxit=12),
        # one S apply of a batch of shots: three grid sizes and frequencies, 22 shots each
        dict(name="batch_layered2d_256_384_512_f32", kind="batch", medium="layered", n1=256, n2=384, n3=512, order=4,
             precision="fp32", sides="free_top", nrhs=22, ppw=10.0),
        # the layered section mapped onto an annular sector (curvilinear grid)
        dict(name="apply_sector2d_1024_f32", kind="apply", medium="layered", nx=1024, ny=1025, nz=0, order=4,
             precision="fp32", sides="free_top", nrhs=1, ppw=10.0, mapped=True),
        # the 3D cube of the configurations, FP32 stencil: the largest call
        dict(name="apply_grf3d_256_f32", kind="apply", medium="grf", nx=256, ny=256, nz=256, order=4,
             precision="fp32", sides="dirichlet", nrhs=1, ppw=10.0, mapped=False),
        # 3D in FP64 on a ragged box with a free top
        dict(name="apply_grf3d_ragged_f64", kind="apply", medium="grf", nx=101, ny=93, nz=87, order=4,
             precision="fp64", sides="free_top", nrhs=1, ppw=10.0, mapped=False),
        # 3D at order 2
        dict(name="apply_grf3d_o2_128_f32", kind="apply", medium="grf", nx=128, ny=128, nz=128, order=2,
             precision="fp32", sides="dirichlet", nrhs=1, ppw=10.0, mapped=False),
        # two layers of the warm-start network, forward and backward, as one training
        # step runs them: full resolution, few channels; and the widest one (after a
        # concatenation, a quarter of the resolution)
        dict(name="conv_256x256_32_32", kind="conv", batch=8, height=256, width=256, ci=32, co=32),
        dict(name="conv_64x64_256_128", kind="conv", batch=8, height=64, width=64, ci=256, co=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply2d", "apply2d", "apply3d", "apply3d", "mapped", "solve", "batch", "conv"])
    sides = rng.choice(["dirichlet", "free_top", "free"])
    precision = rng.choice(["fp32", "fp64"])
    if kind == "conv":
        level = rng.randrange(3)
        c = (32, 64, 128)[level]
        size = [2 * max(4, _log_int(rng, 24, 128) >> level) for _ in range(2)]
        return dict(kind="conv", batch=rng.randint(1, 8), height=size[0], width=size[1],
                    ci=rng.choice([16, c, 2 * c]) if level == 0 else rng.choice([c // 2, c, 2 * c]), co=c)
    if kind == "batch":
        return dict(kind="batch", medium="layered", n1=_log_int(rng, 96, 256), n2=_log_int(rng, 128, 384),
                    n3=_log_int(rng, 192, 512), order=4, precision="fp32", sides="free_top", nrhs=rng.randint(4, 22),
                    ppw=round(rng.uniform(10.0, 16.0), 2))
    if kind == "solve":
        n = _log_int(rng, 48, 384)
        return dict(kind="solve", medium="layered", nx=n, ny=n + rng.randint(-9, 9), nz=0, order=4,
                    precision=precision, sides="free_top", nrhs=1, ppw=round(rng.uniform(10.0, 14.0), 2), mapped=False,
                    tol=1e-6, maxit=rng.randint(4, 12))
    if kind == "mapped":
        return dict(kind="apply", medium="layered", nx=_log_int(rng, 96, 1024), ny=_log_int(rng, 96, 1024), nz=0,
                    order=4, precision=precision, sides=sides, nrhs=rng.randint(1, 2),
                    ppw=round(rng.uniform(10.0, 16.0), 2), mapped=True)
    if kind == "apply2d":
        return dict(kind="apply", medium=rng.choice(["layered", "grf"]), nx=_log_int(rng, 64, 1100),
                    ny=_log_int(rng, 64, 1100), nz=0, order=rng.choice([2, 4, 4]), precision=precision, sides=sides,
                    nrhs=rng.randint(1, 3), ppw=round(rng.uniform(10.0, 16.0), 2), mapped=False)
    hi = 180 if precision == "fp32" else 110
    return dict(kind="apply", medium="grf", nx=_log_int(rng, 40, hi), ny=_log_int(rng, 40, hi),
                nz=_log_int(rng, 40, hi), order=rng.choice([2, 4, 4]), precision=precision, sides=sides, nrhs=1,
                ppw=round(rng.uniform(10.0, 14.0), 2), mapped=False)


# ---- problems ----------------------------------------------------------------

def _sides(name, dim):
    bc = [inputs.DIRICHLET] * 6
    if name == "free_top":
        bc[2 * dim - 1] = inputs.FREE
    elif name == "free":
        bc[:2 * dim] = [inputs.FREE] * (2 * dim)
    return bc


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth_field(shape, corr, seed):
    """Gaussian random field (correlation length `corr` nodes), scaled to VS_SPAN at its largest value."""
    pad = [int(k + 3 * corr) for k in shape]
    noise = torch.randn(pad, dtype=torch.float32, device="cuda", generator=_generator(seed))
    spec = torch.fft.rfftn(noise)
    for a, k in enumerate(pad):
        f = torch.fft.rfftfreq(k, device="cuda") if a == len(pad) - 1 else torch.fft.fftfreq(k, device="cuda")
        g = torch.exp(-0.25 * (2 * math.pi * f * corr) ** 2)
        spec *= g.reshape([-1 if b == a else 1 for b in range(len(pad))])
    x = torch.fft.irfftn(spec, s=pad, dim=tuple(range(len(pad))))[tuple(slice(0, k) for k in shape)].double()
    x = x - x.mean()
    return x * (VS_SPAN / x.abs().max())


def _speeds(case):
    """(slowest Vs, largest sqrt((lambda + (dim + 1) mu) / rho)) of a case's medium, as its family defines them."""
    dim = 3 if case.get("nz") else 2
    if case["medium"] == "homogeneous":
        return 1.0, math.sqrt(2.0 + dim + 1)
    if case["medium"] == "layered":
        return 1.5 / math.sqrt(3.0), 4.5 / math.sqrt(3.0) * math.sqrt(1.0 + dim + 1)
    return math.exp(-VS_SPAN), math.exp(VS_SPAN) * math.sqrt(1.24 + dim + 1)


def _problem(case, seed, scale=1.0):
    """The synthetic problem of a case: its grid, medium and sources from the seed."""
    dim = 3 if case["nz"] else 2
    bc = _sides(case["sides"], dim)
    nu = [case["nx"], case["ny"], case["nz"]][:dim]
    n = [k + (bc[2 * a] == inputs.DIRICHLET) + (bc[2 * a + 1] == inputs.DIRICHLET) for a, k in enumerate(nu)]
    shape = tuple(reversed(n))
    rng = np.random.default_rng(seed)
    layered = case["medium"] == "layered"
    h = 0.01 if layered else 1.0 / (max(n) - 1)
    if case["medium"] == "homogeneous":
        rho, lam, mu = inputs.homogeneous(n)
    elif layered:
        rho, lam, mu = inputs.layered(n, h)
        rho *= 1.0 + 0.02 * rng.uniform(-1, 1, size=(shape[0],) + (1,) * (dim - 1))  # densities of another survey
    else:
        vs = torch.exp(_smooth_field(shape, 0.1 / h, seed))
        m = vs * vs
        rho, mu, lam = np.ones(shape), m.cpu().numpy(), (1.24 * m).cpu().numpy()
    if case["ppw"]:
        omega = scale * 2 * math.pi * _speeds(case)[0] / (case["ppw"] * h)
    else:
        omega = 10.0
    if layered:  # mu, lambda follow the density: Vs and Vp stay those of the layers
        base = inputs.layered(n, h)
        mu, lam = base[1 + 1] / base[0] * rho, base[1] / base[0] * rho
    # one source per right-hand side: a point force of a few nodes' width
    r, forcing = case["nrhs"], []
    width = case["ppw"] / 4.0 * h if case["ppw"] else 0.05
    for _ in range(r):
        at = [rng.uniform(0.25, 0.75) * (k - 1) * h for k in n]
        if layered:
            at[1] = 0.95 * (n[1] - 1) * h
        g = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for a in range(dim):
            x = torch.arange(n[a], dtype=torch.float64, device="cuda") * h - at[a]
            g = g + (x * x).reshape([-1 if b == dim - 1 - a else 1 for b in range(dim)])
        g = torch.exp(-g / (2 * width * width)).cpu().numpy()
        d = rng.standard_normal(dim)
        forcing.append(np.stack([c * g for c in d / np.linalg.norm(d)]))
    mapping = None
    if case.get("mapped"):  # about the extent of the square: radii 1.5 L to 2.5 L, an arc of the other side's length
        lq, lr = (n[0] - 1) * h, (n[1] - 1) * h
        mapping = inputs.annulus_mapping(n, h, span=lr / (2.0 * lq), r0=1.5 * lq, dr=lq)
    return inputs.Problem(case["medium"], dim, n, h, case["order"], bc, omega, rho, lam, mu, np.stack(forcing),
                          mapping=mapping)


def _wave_vector(p, seed):
    """A wave field of the problem's wavelengths (what the solver applies S to): plane
    waves in random directions with a little noise, [nrhs * dim * nodes]."""
    rng = np.random.default_rng(seed + 77)
    nu = p.unknowns_per_axis()
    k0 = p.omega * p.h / float(np.sqrt(p.mu / p.rho).mean())
    out = []
    for _ in range(p.nrhs * p.dim):
        v = 0.01 * torch.randn(tuple(reversed(nu)), dtype=torch.float64, device="cuda",
                               generator=_generator(rng.integers(1 << 30)))
        for _ in range(4):
            d = rng.standard_normal(p.dim)
            d *= k0 * rng.uniform(0.5, 1.2) / np.linalg.norm(d)
            z = torch.zeros((), dtype=torch.float64, device="cuda") + rng.uniform(0, 2 * math.pi)
            for a in range(p.dim):
                x = torch.arange(nu[a], dtype=torch.float64, device="cuda") * d[a]
                z = z + x.reshape([-1 if b == p.dim - 1 - a else 1 for b in range(p.dim)])
            v += rng.standard_normal() * torch.cos(z)
        out.append(v.reshape(-1))
    return torch.cat(out)


BATCH_SCALES = (0.5, 0.75, 1.0)  # frequencies of a batch's members, of the points-per-wavelength one


def _members(case, seed):
    out = []
    for k, scale in enumerate(BATCH_SCALES):
        one = dict(case, nx=case["n%d" % (k + 1)], ny=case["n%d" % (k + 1)] + 1, nz=0)
        out.append(_problem(one, seed + 1000 * k, scale))
    return out


def _conv_inputs(case, seed):
    g = _generator(seed)
    n, h, w, ci, co = (case[k] for k in ("batch", "height", "width", "ci", "co"))

    def rand(*shape):
        return torch.randn(shape, dtype=torch.float32, device="cuda", generator=g)

    x = torch.nn.functional.leaky_relu(rand(n, h, w, ci), 0.1).to(torch.bfloat16)  # the layer before's activations
    weight = (rand(co, 3, 3, ci) * math.sqrt(2.0 / (9 * ci))).to(torch.bfloat16)
    return dict(x=x, w=weight, bias=0.1 * rand(co), pre=rand(n, h, w, co), dy=rand(n, h, w, co) * 1e-3)


def prepare(case, seed):
    if case["kind"] == "conv":
        s = _conv_inputs(case, seed)
        s.update(case=case, scratch=torch.empty(9 * case["ci"] * case["co"], dtype=torch.bfloat16, device="cuda"))
        return s
    if case["kind"] == "batch":
        ps = _members(case, seed)
        return dict(case=case, solver=WaveHoltzBatch(ps, case["precision"]),
                    v=[_wave_vector(p, seed + 1000 * k) for k, p in enumerate(ps)])
    p = _problem(case, seed)
    s = dict(case=case, solver=WaveHoltz(p, case["precision"]))
    if case["kind"] == "apply":
        s["v"] = _wave_vector(p, seed)
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "conv":
        n, h, w, ci, co = (case[k] for k in ("batch", "height", "width", "ci", "co"))
        st = torch.cuda.current_stream().cuda_stream

        def new(shape, dtype):
            return torch.empty(shape, dtype=dtype, device="cuda")

        # forward: pre-activation and activation
        pre, act = new((n, h, w, co), torch.float32), new((n, h, w, co), torch.bfloat16)
        L.ewh_conv3x3_fwd(state["x"], state["w"], state["bias"], pre, act, 1, n, h, w, ci, co, st)
        # backward, from the gradient of the activation and the saved pre-activation
        g, gb = new((n, h, w, co), torch.float32), new((n, h, w, co), torch.bfloat16)
        L.ewh_leaky_relu_bwd(state["pre"], state["dy"], g, gb, n * h * w * co, st)
        db, dw = new((co,), torch.float32), new((co, 3, 3, ci), torch.float32)
        L.ewh_bias_grad(g, db, n * h * w, co, st)
        L.ewh_conv3x3_wgrad(state["x"], gb, dw, n, h, w, ci, co, st)
        dx = new((n, h, w, ci), torch.float32)
        L.ewh_conv3x3_dgrad(gb, state["w"], state["scratch"], dx, n, h, w, ci, co, st)
        return dict(pre=pre, act=act, db=db, dw=dw, dx=dx)
    if case["kind"] == "solve":
        v, _ = state["solver"].solve(tol=case["tol"], maxit=case["maxit"], raise_on_error=False)
        out = [v]
    elif case["kind"] == "batch":
        out = state["solver"].apply_S(state["v"])
    else:
        out = [state["solver"].apply_S(state["v"])]
    return [x.float() for x in out] if case["precision"] == "fp32" else out


def _levels(case, scale=1.0):
    """Time levels of one period (nt) of a case's problem, from its family's speeds."""
    slow, fast = _speeds(case)
    if case.get("mapped"):  # the narrowest cells of the sector, next to its inner radius
        fast *= 1.18
    if case["ppw"]:
        return math.ceil(case["ppw"] / (scale * slow) * fast / 0.5)
    return math.ceil(2 * math.pi / 10.0 * fast / 0.5 * (case["nx"] + 1))


def work(case):
    if case["kind"] == "conv":
        p = case["batch"] * case["height"] * case["width"]
        ci, co = case["ci"], case["co"]
        # read x twice (forward, weight gradient), w twice, the saved pre-activation and dy once; write pre, act, dx, dw, db
        data = p * (2 * 2 * ci + 4 * ci + (4 + 2 + 4 + 4) * co) + 9 * ci * co * (2 * 2 + 4)
        return dict(bytes=data, flops=3 * 2 * 9 * p * ci * co)
    if case["kind"] == "batch":
        nodes = [case["n%d" % k] * (case["n%d" % k] + 1) for k in (1, 2, 3)]
        levels = [_levels(case, s) for s in BATCH_SCALES]
        return dict(bytes=sum(m * (2 * 2 * 8 * case["nrhs"] + 3 * 4) for m in nodes),
                    flops=sum(52 * m * case["nrhs"] * t for m, t in zip(nodes, levels)))
    dim = 3 if case["nz"] else 2
    nodes = case["nx"] * case["ny"] * max(1, case["nz"])
    size = 4 if case["precision"] == "fp32" else 8
    per = {(2, 2): 70, (2, 4): 52, (3, 2): 160, (3, 4): 106}[(dim, case["order"])] + (26 if case["mapped"] else 0)
    applies = 1
    if case["kind"] == "solve":  # iterations, the right-hand side and a residual
        applies = (20 if case["medium"] == "homogeneous" else case["maxit"]) + 2
    media = (3 + (4 if case["mapped"] else 0)) * size
    return dict(bytes=applies * nodes * (2 * dim * 8 * case["nrhs"] + media),
                flops=applies * nodes * case["nrhs"] * per * _levels(case))


# ---- the same in plain torch, 64 bits -----------------------------------------------

def _cut(u, ax, a, b):
    return u.narrow(ax, a, b - a)


def _sbp(u, ax):
    """Fourth-order summation-by-parts first derivative along an axis (unit spacing)."""
    N = u.shape[ax]
    d = torch.empty_like(u)
    _cut(d, ax, 4, N - 4).copy_((8.0 * (_cut(u, ax, 5, N - 3) - _cut(u, ax, 3, N - 5)) -
                                 (_cut(u, ax, 6, N - 2) - _cut(u, ax, 2, N - 6))) / 12.0)
    rows = [{0: -24 / 17, 1: 59 / 34, 2: -4 / 17, 3: -3 / 34}, {0: -0.5, 2: 0.5},
            {0: 4 / 43, 1: -59 / 86, 3: 59 / 86, 4: -4 / 43}, {0: 3 / 98, 2: -59 / 98, 4: 32 / 49, 5: -4 / 49}]
    for i, row in enumerate(rows):
        _cut(d, ax, i, i + 1).copy_(sum(c * _cut(u, ax, j, j + 1) for j, c in row.items()))
        _cut(d, ax, N - 1 - i, N - i).copy_(sum(-c * _cut(u, ax, N - 1 - j, N - j) for j, c in row.items()))
    return d


def _sbp_divergence(f, ax):
    """-D f + H^-1 B f along an axis."""
    N = f.shape[ax]
    d = -_sbp(f, ax)
    _cut(d, ax, 0, 1).sub_(48 / 17 * _cut(f, ax, 0, 1))
    _cut(d, ax, N - 1, N).add_(48 / 17 * _cut(f, ax, N - 1, N))
    return d


class _Plain:
    """A problem's operator M^-1 K, time step, filter and mass on the full grid; fields are [rhs][z][y][x] per component."""

    def __init__(self, p):
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")  # noqa: E731
        self.p, dim = p, p.dim
        self.ax = [dim - a for a in range(dim)]  # tensor axis of grid axis a (axis 0: right-hand sides)
        self.rho, self.lam, self.mu = (t(a)[None] for a in (p.rho, p.lam, p.mu))
        shape = self.rho.shape
        self.known = torch.ones(shape, dtype=torch.float64, device="cuda")
        weight = torch.ones(shape, dtype=torch.float64, device="cuda")
        sbp_norm = [17 / 48, 59 / 48, 43 / 48, 49 / 48]
        for a in range(dim):
            N = p.n[a]
            w = torch.ones(N, dtype=torch.float64, device="cuda")
            for i in range(4):
                if p.order == 4:
                    w[i] = w[N - 1 - i] = sbp_norm[i]
            for side, i in ((0, 0), (1, N - 1)):
                if p.bc[2 * a + side] == inputs.DIRICHLET:
                    _cut(self.known, self.ax[a], i, i + 1).zero_()
                elif p.order == 2:
                    w[i] = 0.5
            weight = weight * w.reshape([-1 if b == self.ax[a] else 1 for b in range(dim + 1)])
        self.weight = weight
        speed = (self.lam + (dim + 1) * self.mu) / self.rho
        self.met = None
        J = 1.0
        if p.mapping is not None:
            X, Y = (t(a)[None] for a in p.mapping)
            xq, xr, yq, yr = (_sbp(c, self.ax[a]) / p.h for c in (X, Y) for a in (0, 1))
            J = xq * yr - xr * yq
            self.met, self.J = (yr, -xr, -yq, xq), J
            speed = speed * 0.5 * (yr ** 2 + xr ** 2 + yq ** 2 + xq ** 2) / J ** 2
        T = 2 * math.pi / p.omega
        self.nt = max(5, math.ceil(T / (0.5 * p.h / math.sqrt(float(speed.max())))))
        dt = T / self.nt
        wt = 2 * math.sin(p.omega * dt / 2) / dt
        self.kt = (wt / p.omega) ** 2 * dt * dt
        eta = [0.5 if k in (0, self.nt) else 1.0 for k in range(self.nt + 1)]
        self.w = [2 / self.nt * eta[k] * (math.cos(2 * math.pi * k / self.nt) - 0.25) for k in range(self.nt + 1)]
        self.mass = self.rho * J * weight * p.h ** dim * self.known

    def accel(self, u):
        """M^-1 K u at the unknown nodes."""
        p, ax, dim = self.p, self.ax, self.p.dim
        if p.order == 4 and self.met is None:
            g = [[_sbp(u[c], ax[a]) for a in range(dim)] for c in range(dim)]
            div = self.lam * sum(g[a][a] for a in range(dim))
            k = []
            for c in range(dim):
                k.append(sum(_sbp_divergence(self.mu * (g[c][a] + g[a][c]) + (div if a == c else 0.0), ax[a])
                             for a in range(dim)))
            scale = self.known / (self.rho * p.h ** 2)
        elif p.order == 4:
            yr, mxr, myq, xq = self.met
            d = [[_sbp(c, ax[0]), _sbp(c, ax[1])] for c in u]
            ux, uy, vx, vy = ((m0 * d[c][0] + m1 * d[c][1]) / self.J
                              for c in (0, 1) for m0, m1 in ((yr, myq), (mxr, xq)))
            sxx = self.lam * (ux + vy) + 2 * self.mu * ux
            syy = self.lam * (ux + vy) + 2 * self.mu * vy
            sxy = self.mu * (uy + vx)
            k = [_sbp_divergence(yr * a + mxr * b, ax[0]) + _sbp_divergence(myq * a + xq * b, ax[1])
                 for a, b in ((sxx, sxy), (sxy, syy))]
            scale = self.known / (self.rho * self.J * p.h ** 2)
        else:
            k = self._order2(u)
            scale = self.known / (self.rho * self.weight * p.h ** 2)
        return [scale * c for c in k]

    def _centred(self, u, a):
        x, N = self.ax[a], u.shape[self.ax[a]]
        d = torch.empty_like(u)
        _cut(d, x, 1, N - 1).copy_(0.5 * (_cut(u, x, 2, N) - _cut(u, x, 0, N - 2)))
        _cut(d, x, 0, 1).copy_(_cut(u, x, 1, 2) - _cut(u, x, 0, 1))
        _cut(d, x, N - 1, N).copy_(_cut(u, x, N - 1, N) - _cut(u, x, N - 2, N - 1))
        return d

    def _centred_t(self, v, a):
        x, N = self.ax[a], v.shape[self.ax[a]]
        d = torch.zeros_like(v)
        half = 0.5 * _cut(v, x, 1, N - 1)
        _cut(d, x, 2, N).add_(half)
        _cut(d, x, 0, N - 2).sub_(half)
        for i, j, k in ((0, 1, 0), (N - 1, N - 1, N - 2)):
            e = _cut(v, x, i, i + 1)
            _cut(d, x, j, j + 1).add_(e)
            _cut(d, x, k, k + 1).sub_(e)
        return d

    def _order2(self, u):
        p, dim = self.p, self.p.dim
        m = self.weight * self.known
        out = []
        for c in range(dim):
            k = torch.zeros_like(u[c])
            for a in range(dim):
                x, N = self.ax[a], u[c].shape[self.ax[a]]
                coef = self.lam + 2 * self.mu if a == c else self.mu
                edge = 0.5 * (_cut(coef, x, 0, N - 1) + _cut(coef, x, 1, N))
                # the weights of the other axes: those of this one's inner nodes are 1
                edge = edge * _cut(self.weight, x, 1, 2)
                f = edge * (_cut(u[c], x, 1, N) - _cut(u[c], x, 0, N - 1))
                _cut(k, x, 1, N).add_(f)
                _cut(k, x, 0, N - 1).sub_(f)
            for b in range(dim):
                if b != c:
                    k += self._centred_t(m * self.lam * self._centred(u[b], b), c)
                    k += self._centred_t(m * self.mu * self._centred(u[b], c), b)
            out.append(k)
        return out

    def wave(self, u, force=None):
        """The filtered leapfrog: Pi u with `force` = f / rho, S u without."""
        acc = [self.w[0] * c for c in u]
        delta = None
        for n in range(self.nt):
            a = self.accel(u)
            if force is not None:
                cn = math.cos(2 * math.pi * n / self.nt)
                a = [x + cn * f for x, f in zip(a, force)]
            delta = [-0.5 * self.kt * x for x in a] if n == 0 else [d - self.kt * x for d, x in zip(delta, a)]
            u = [x + d for x, d in zip(u, delta)]
            for s, x in zip(acc, u):
                s += self.w[n + 1] * x
        return acc

    def split(self, v):
        """Solver vector [rhs][comp][unknowns] -> full-grid fields per component."""
        p = self.p
        nu = tuple(reversed(p.unknowns_per_axis()))
        v = v.reshape((p.nrhs, p.dim) + nu)
        out = []
        for c in range(p.dim):
            f = torch.zeros((p.nrhs,) + tuple(self.rho.shape[1:]), dtype=torch.float64, device="cuda")
            self._inner(f).copy_(v[:, c])
            out.append(f)
        return out

    def _inner(self, f):
        for a in range(self.p.dim):
            lo = 1 if self.p.bc[2 * a] == inputs.DIRICHLET else 0
            f = f.narrow(self.ax[a], lo, self.p.unknowns_per_axis()[a])
        return f

    def join(self, u):
        return torch.stack([self._inner(c) for c in u], dim=1).reshape(-1)

    def solve(self, tol, maxit):
        """CG on (I - S) v = Pi 0 in the mass inner product, one right-hand side."""
        f = torch.as_tensor(self.p.forcing, dtype=torch.float64, device="cuda")
        force = [f[:, c] / self.rho * self.known for c in range(self.p.dim)]
        zero = [torch.zeros_like(c) for c in force]
        b = self.wave(zero, force)
        dot = lambda x, y: float(sum((self.mass * s * t).sum() for s, t in zip(x, y)))  # noqa: E731
        x, r = zero, b
        q = [c.clone() for c in b]
        rr = bb = dot(b, b)
        for _ in range(maxit):
            if math.sqrt(rr / bb) <= tol:
                break
            aq = [s - t for s, t in zip(q, self.wave(q))]
            alpha = rr / dot(q, aq)
            x = [s + alpha * t for s, t in zip(x, q)]
            r = [s - alpha * t for s, t in zip(r, aq)]
            new = dot(r, r)
            q = [s + new / rr * t for s, t in zip(r, q)]
            rr = new
        return x


def _exact_conv(case, seed):
    s = _conv_inputs(case, seed)
    x, w = s["x"].double(), s["w"].double()
    n, h, wd = case["batch"], case["height"], case["width"]

    def conv(v, taps):  # v [n, h, w, c] with zero padding, taps [co, 3, 3, c]
        v = torch.nn.functional.pad(v, (0, 0, 1, 1, 1, 1))
        return sum(v[:, i:i + h, j:j + wd] @ taps[:, i, j].T for i in range(3) for j in range(3))

    pre = conv(x, w) + s["bias"].double()
    act = torch.where(pre > 0, pre, 0.1 * pre)
    g32 = torch.where(s["pre"] > 0, s["dy"], torch.tensor(0.1, dtype=torch.float32, device="cuda") * s["dy"])
    g = g32.to(torch.bfloat16).double()
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    flat = g.reshape(-1, case["co"]).T
    dw = torch.stack([torch.stack([flat @ xp[:, i:i + h, j:j + wd].reshape(-1, case["ci"]) for j in range(3)], dim=1)
                      for i in range(3)], dim=1)
    dx = conv(g, w.flip(1, 2).permute(3, 1, 2, 0))
    return dict(pre=pre, act=act, db=g32.double().sum(dim=(0, 1, 2)), dw=dw, dx=dx)


def exact(case, seed):
    if case["kind"] == "conv":
        return _exact_conv(case, seed)
    if case["kind"] == "batch":
        out = []
        for k, p in enumerate(_members(case, seed)):
            q = _Plain(p)
            out.append(q.join(q.wave(q.split(_wave_vector(p, seed + 1000 * k)))))
        return out
    p = _problem(case, seed)
    q = _Plain(p)
    if case["kind"] == "solve":
        return [q.join(q.solve(case["tol"], case["maxit"]))]
    return [q.join(q.wave(q.split(_wave_vector(p, seed))))]
