"""Cases that stand for the framework's work: time stepping of one cavity in 2D and 3D in both
precisions, a batch of uneven cavities, driven and tracked-Delta-E runs, and the gradient of a
final-time misfit.  A pass is what a user's program does with a grid it keeps: set the initial
fields, advance them a number of steps, take the fields back (or, for a gradient, a forward run
and its reverse pass).

Fields of FP32_REFINED runs are returned as float32: the path computes in FP32 and its results
carry FP32 rounding noise, so a program that chose it goes on in that type.  FP64 runs return
float64.  exact() steps the same scheme in 64-bit torch with dense Pade matrices.
"""
import math

import torch

import paper_2306_17263_gb300 as ms
from paper_2306_17263_gb300.autograd import propagate_ez

PREC = {"fp64": ms.FP64, "fp32": ms.FP32_REFINED}
CLOS = {"paper": ms.CLOSURE_PAPER, "reflect": ms.CLOSURE_REFLECT}
SCHEME = {"c4": ms.SCHEME_C4, "c4_de": ms.SCHEME_C4_DE}

F64 = torch.float64


def case2d(n, steps, precision, closure="paper", r=0.5, z=1.0, scheme="c4", init="modes", sources=0, **more):
    return dict(kind="grid2d", n=n, steps=steps, precision=precision, closure=closure, r=r, z=z, scheme=scheme,
                init=init, sources=sources, **more)


def case3d(n, steps, precision, closure="paper", r=0.4, z=1.0, **more):
    return dict(kind="grid3d", n=n, steps=steps, precision=precision, closure=closure, r=r, z=z, **more)


def listed():
    return [
        # the smallest workload of the repository (64 cells a side, one time unit): launches and latency
        case2d(64, 128, "fp64", name="2d fp64 64"),
        # the headline grid: 2048 cells a side, modes up to 40, FP32_REFINED
        case2d(2048, 64, "fp32", name="2d fp32 2048"),
        # a ragged size near the stability limit (more sweeps of the solve), energy-conserving closure
        case2d(777, 50, "fp32", closure="reflect", r=0.65, z=1.7, init="field", name="2d fp32 777 reflect"),
        # full precision, a size between
        case2d(1024, 16, "fp64", init="field", name="2d fp64 1024"),
        # a driven cavity: two current sources on the headline grid's half size
        case2d(1024, 48, "fp32", z=1.3, sources=2, name="2d fp32 1024 driven"),
        # Delta E tracked as printed in the paper's Step 1 and Step 2
        case2d(1024, 32, "fp32", scheme="c4_de", name="2d fp32 1024 tracked"),
        # the 3D workload: 256^3, six components
        case3d(256, 10, "fp32", name="3d fp32 256"),
        # a small ragged 3D cavity, energy-conserving closure
        case3d(75, 40, "fp32", closure="reflect", r=0.5, z=1.7, name="3d fp32 75 reflect"),
        # 3D in full precision
        case3d(96, 8, "fp64", name="3d fp64 96"),
        # independent cavities of uneven sides from {64, 96, ..., 768}, advanced together
        dict(kind="batch", count=20, sizes_seed=0, lo=64, hi=768, steps=200, closure="paper", r=0.5, z=1.0,
             name="batch 20 cavities"),
        # gradient of a final-time misfit: forward run and FP32 reverse pass, 1024 cells a side
        dict(kind="gradient", n=1024, steps=64, precision="fp32", closure="paper", r=0.5, z=1.0, name="gradient fp32 1024"),
        # the same in full precision on a smaller odd grid
        dict(kind="gradient", n=321, steps=30, precision="fp64", closure="reflect", r=0.6, z=1.0,
             name="gradient fp64 321"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid2d", "grid2d", "grid2d", "grid2d", "grid3d", "grid3d", "batch", "gradient", "gradient"])
    closure = rng.choice(["paper", "reflect"])
    z = rng.choice([1.0, 1.3, 1.7, 2.5])
    if kind == "grid2d":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        n = _log_int(rng, 24, 2048 if precision == "fp32" else 1024)
        most = 1.2e8 if precision == "fp32" else 8e6  # cell updates of a pass
        steps = max(4, min(_log_int(rng, 8, 256), int(most / (n * n))))
        scheme = rng.choice(["c4", "c4", "c4", "c4_de"])
        sources = rng.choice([0, 0, 1, 2, 3]) if scheme == "c4" else 0
        return case2d(n, steps, precision, closure, round(rng.uniform(0.2, 0.68), 3), z, scheme,
                      rng.choice(["modes", "field"]), sources)
    if kind == "grid3d":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        n = _log_int(rng, 12, 224 if precision == "fp32" else 90)
        most = 8e7 if precision == "fp32" else 3e6
        steps = max(3, min(_log_int(rng, 8, 96), int(most / n ** 3)))
        return case3d(n, steps, precision, closure, round(rng.uniform(0.2, 0.55), 3), z)
    if kind == "batch":
        hi = 32 * rng.randint(8, 24)
        return dict(kind="batch", count=_log_int(rng, 4, 20), sizes_seed=rng.randrange(1, 1 << 20), lo=64, hi=hi,
                    steps=_log_int(rng, 16, 200), closure=closure, r=round(rng.uniform(0.2, 0.68), 3), z=z)
    precision = rng.choice(["fp32", "fp64"])
    n = _log_int(rng, 32, 1024 if precision == "fp32" else 512)
    steps = max(4, min(_log_int(rng, 8, 128), int((6e7 if precision == "fp32" else 3e6) / (n * n))))
    return dict(kind="gradient", n=n, steps=steps, precision=precision, closure=closure,
                r=round(rng.uniform(0.2, 0.68), 3), z=z)


# ---------------------------------------------------------------------------------------------
# Inputs

def _generator(seed):
    return torch.Generator().manual_seed(int(seed))


def _modes(gen, count, kmax):
    """`count` rows (m, n, amp): indices uniform in [1, kmax], amplitudes N(0, 1)."""
    mn = torch.randint(1, kmax + 1, (count, 2), generator=gen).tolist()
    amp = torch.randn(count, generator=gen, dtype=F64).tolist()
    return [(int(a), int(b), float(c)) for (a, b), c in zip(mn, amp)]


def _axis(n, k, node, dev):
    """sin(pi k x) at the n + 1 nodes, or cos(pi k x) at the n half-nodes, exact zeros on the walls."""
    if node:
        q = torch.remainder(torch.arange(n + 1, device=dev, dtype=torch.int64) * k, 2 * n).to(F64)
        v = torch.sin(math.pi * q / n)
        v[0] = v[n] = 0.0
        return v
    q = torch.remainder((2 * torch.arange(n, device=dev, dtype=torch.int64) + 1) * k, 4 * n).to(F64)
    return torch.cos(math.pi * q / (2 * n))


def mode_fields(n, r, z, modes, dev):
    """Cavity modes: E_z at t = 0, H_x and H_y at half a step."""
    t = 0.5 * r / n
    ez = torch.zeros(n + 1, n + 1, dtype=F64, device=dev)
    hx = torch.zeros(n, n + 1, dtype=F64, device=dev)
    hy = torch.zeros(n + 1, n, dtype=F64, device=dev)
    for m, k, a in modes:
        w = math.pi * math.hypot(m, k)
        s = a * math.sin(w * t) / (w * z)
        sx, sy = _axis(n, m, True, dev), _axis(n, k, True, dev)
        ez += a * torch.outer(sy, sx)
        hx -= s * math.pi * k * torch.outer(_axis(n, k, False, dev), sx)
        hy += s * math.pi * m * torch.outer(sy, _axis(n, m, False, dev))
    return ez, hx, hy


def random_ez(n, gen, dev, ell=0.05, mmax=96):
    """Gaussian random field of correlation length ell on the E_z nodes (sine series, unit RMS)."""
    mc = min(mmax, n - 1)
    k = torch.arange(1, mc + 1, dtype=F64, device=dev)
    env = torch.exp(-math.pi ** 2 * (k[:, None] ** 2 + k[None, :] ** 2) * ell ** 2 / 4.0)
    a = torch.randn(mc, mc, generator=gen, dtype=F64).to(dev) * env
    s = torch.stack([_axis(n, j, True, dev) for j in range(1, mc + 1)], 1)
    f = s @ a @ s.T
    return f / f[1:-1, 1:-1].square().mean().sqrt()


def random_h(n, gen, dev):
    """H of a Gaussian random potential that vanishes on the walls (divergence-free)."""
    p = random_ez(n, gen, dev)
    hx = torch.diff(p, dim=0) * n * 0.05
    hy = -torch.diff(p, dim=1) * n * 0.05
    hx[:, 0] = hx[:, -1] = 0.0
    hy[0, :] = hy[-1, :] = 0.0
    return hx, hy


def fields2d(case, seed, dev):
    gen = _generator(seed)
    n = case["n"]
    if case["init"] == "modes":
        return mode_fields(n, case["r"], case["z"], _modes(gen, 8, max(2, min(40, n // 6))), dev)
    return (random_ez(n, gen, dev),) + random_h(n, gen, dev)


def sources2d(case, seed):
    """Rows (m, n, amp, omega) of J_z = amp sin sin sin(omega t)."""
    gen = _generator(seed + 77)
    out = []
    for m, k, a in _modes(gen, case["sources"], 4):
        out.append((m, k, a, 2.0 + 12.0 * float(torch.rand(1, generator=gen, dtype=F64))))
    return out


def fields3d(case, seed, dev):
    """Two cavity modes A . (m, n, p) = 0, E at t = 0 and H at half a step."""
    gen = _generator(seed)
    n, z = case["n"], case["z"]
    t = 0.5 * case["r"] / n
    shapes = shapes3d(n)
    out = [torch.zeros(s, dtype=F64, device=dev) for s, _ in shapes]
    kmax = max(2, min(16, n // 6))
    for m, k, a in _modes(gen, 2, kmax):
        p = int(torch.randint(1, kmax + 1, (1,), generator=gen))
        K = (math.pi * m, math.pi * k, math.pi * p)
        w = math.sqrt(sum(v * v for v in K))
        u = torch.randn(3, generator=gen, dtype=F64).tolist()
        A = [a / w * (u[(e + 1) % 3] * K[(e + 2) % 3] - u[(e + 2) % 3] * K[(e + 1) % 3]) for e in range(3)]
        sh = -math.sin(w * t) / (z * w)
        amp = (A[0], A[1], A[2], sh * (A[2] * K[1] - A[1] * K[2]), sh * (A[0] * K[2] - A[2] * K[0]),
               sh * (A[1] * K[0] - A[0] * K[1]))
        for q, (_, node) in enumerate(shapes):
            x, y, zz = (_axis(n, i, node[e], dev) for e, i in enumerate((m, k, p)))
            out[q] += amp[q] * (zz[:, None, None] * y[None, :, None]) * x[None, None, :]
    return tuple(out)


def shapes3d(n):
    """Per component: its shape [z][y][x] and whether it sits on nodes along x, y, z."""
    out = []
    for c in range(6):
        node = [(a != c % 3) if c < 3 else (a == c % 3) for a in range(3)]
        out.append((tuple(n + 1 if q else n for q in reversed(node)), node))
    return out


def batch_sizes(case):
    gen = _generator(case["sizes_seed"])
    lo, hi = case["lo"] // 32, case["hi"] // 32
    return [32 * int(v) for v in torch.randint(lo, hi + 1, (case["count"],), generator=gen)]


def batch_modes(case, seed, sizes):
    gen = _generator(seed)
    return [_modes(gen, 4, min(30, s // 6)) for s in sizes]


def gradient_inputs(case, seed, dev):
    gen = _generator(seed)
    ez0 = random_ez(case["n"], gen, dev)
    lam = random_ez(case["n"], gen, dev)
    return ez0, lam


# ---------------------------------------------------------------------------------------------
# Passes

def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    stream = torch.cuda.Stream()
    st = dict(case=case, stream=stream)
    single = case.get("precision") != "fp64"
    st["single"] = single
    if kind == "batch":
        sizes = batch_sizes(case)
        with torch.cuda.stream(stream):
            b = ms.Batch(sizes, case["r"], z=case["z"], closure=CLOS[case["closure"]], stream="torch")
        for c, rows in enumerate(batch_modes(case, seed, sizes)):
            b.init_modes(c, rows)
        st["batch"] = b
        return st
    dim = 3 if kind == "grid3d" else 2
    scheme = SCHEME[case.get("scheme", "c4")]
    with torch.cuda.stream(stream):
        st["grid"] = ms.Grid(case["n"], case["r"], z=case["z"], precision=PREC[case["precision"]],
                             closure=CLOS[case["closure"]], scheme=scheme, stream="torch", dim=dim)
    if kind == "gradient":
        ez0, lam = gradient_inputs(case, seed, dev)
        st["ez0"], st["lam"] = ez0.requires_grad_(True), lam
    else:
        st["fields"] = fields3d(case, seed, dev) if dim == 3 else fields2d(case, seed, dev)
        st["out"] = tuple(torch.empty_like(f) for f in st["fields"])
        if case.get("sources"):
            st["grid"].set_sources(sources2d(case, seed))
    stream.wait_stream(torch.cuda.current_stream())
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    with torch.cuda.stream(st["stream"]):
        if kind == "batch":
            # the cavities go on from where the last pass left them, as in a run watched now and then
            b = st["batch"]
            b.run(case["steps"])
            return [[torch.from_numpy(a).to(torch.float32) for a in b.get_fields(c)] for c in range(case["count"])]
        if kind == "gradient":
            ez0 = st["ez0"]
            ez0.grad = None
            ez = propagate_ez(st["grid"], ez0, case["steps"])
            ez.backward(st["lam"])
            out = (ez.detach(), ez0.grad)
        else:
            g = st["grid"]
            g.set_fields_device(*st["fields"], step=0)
            g.run(case["steps"])
            g.get_fields_device(*st["out"])
            out = st["out"]
        return tuple(f.to(torch.float32) for f in out) if st["single"] else out


def work(case):
    """Bytes: the state read and written once a step (the least a step can do; 16 bytes a point for
    an FP64 or float-float state), and the fields of the pass in and out.  Operations: those of the
    scheme (filter, Pade recurrences, the solve's stencils, the update), not of any one way to do it."""
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        cells = sum(s * s for s in batch_sizes(case))
        return {"bytes": 48.0 * cells * steps + 12.0 * cells, "flops": 150.0 * cells * steps}
    n = case["n"]
    if kind == "grid3d":
        cells = n ** 3
        return {"bytes": 96.0 * cells * steps + 72.0 * cells, "flops": 500.0 * cells * steps}
    cells = n * n
    if kind == "gradient":
        return {"bytes": 2 * 48.0 * cells * steps + 32.0 * cells, "flops": 2 * 150.0 * cells * steps}
    more = 16.0 if case["scheme"] == "c4_de" else 0.0  # the tracked plane is state too
    return {"bytes": (48.0 + more) * cells * steps + 36.0 * cells, "flops": 150.0 * cells * steps}


# ---------------------------------------------------------------------------------------------
# The scheme in 64-bit torch

class Scheme:
    def __init__(self, n, r, z, closure, dev):
        self.n, self.r, self.z, self.dev = n, r, z, dev
        self.h = 1.0 / n
        self.ht = r * self.h
        self.k2 = 24.0 / self.ht ** 2
        self.beta = 1.0 + self.k2 * self.h ** 2 / 12.0
        self.c1h2 = self.k2 * self.beta * self.h ** 2
        self.w = {"h2n": self.pade(n - 1, closure, False), "n2h": self.pade(n, closure, True)}
        rho = (16.0 / 3.0) / (2.0 * self.c1h2 + 16.0 / 3.0)
        self.sweeps = 2 + math.ceil(math.log(1e-18) / math.log(rho))

    def pade(self, m, closure, node_to_half):
        """W = A^-1 D (M x M+1), A = [1, 22, 1]/24 with the closure's end rows."""
        a = torch.zeros(m, m, dtype=F64, device=self.dev)
        i = torch.arange(m, device=self.dev)
        a[i, i] = 22.0
        a[i[1:], i[:-1]] = 1.0
        a[i[:-1], i[1:]] = 1.0
        if closure == "paper":
            e = torch.tensor([26.0, -5.0, 4.0, -1.0], dtype=F64, device=self.dev)
            a[0], a[-1] = 0.0, 0.0
            a[0, :4] = e
            a[-1, -4:] = e.flip(0)
        else:
            a[0, 0] = a[-1, -1] = 23.0 if node_to_half else 22.0
        d = torch.zeros(m, m + 1, dtype=F64, device=self.dev)
        d[i, i] = -1.0
        d[i, i + 1] = 1.0
        return torch.linalg.solve(a / 24.0, d)

    @staticmethod
    def along(mat, u, dim):
        return torch.movedim(torch.tensordot(mat, u, dims=([1], [dim])), 0, dim)

    def delta(self, u, dim, half):
        """Derivative along a dimension; half: from half-nodes to the inner nodes (walls 0)."""
        v = self.along(self.w["h2n" if half else "n2h"], u, dim) * self.n
        return self.pad0(v, dim) if half else v

    def delta_t(self, v, dim, half):
        """Transpose of delta."""
        if half:
            v = v.narrow(dim, 1, v.shape[dim] - 2)
        return self.along(self.w["h2n" if half else "n2h"].T, v, dim) * self.n

    @staticmethod
    def pad0(v, dim):
        z = torch.zeros_like(v.narrow(dim, 0, 1))
        return torch.cat([z, v, z], dim)

    @staticmethod
    def second(u, dim, neu):
        a, b = u.narrow(dim, 0, 1), u.narrow(dim, u.shape[dim] - 1, 1)
        if not neu:
            a, b = torch.zeros_like(a), torch.zeros_like(b)
        p = torch.cat([a, u, b], dim)
        m = u.shape[dim]
        return p.narrow(dim, 0, m) - 2.0 * u + p.narrow(dim, 2, m)

    def neu(self, u):
        return [s == self.n for s in u.shape]

    def inner(self, v):
        """v with 0 on the walls of its node dimensions."""
        for dim, neu in enumerate(self.neu(v)):
            if not neu:
                v = self.pad0(v.narrow(dim, 1, v.shape[dim] - 2), dim)
        return v

    def lap(self, u):
        return sum(self.second(u, d, neu) for d, neu in enumerate(self.neu(u)))

    def filt(self, u):
        return self.inner(self.beta * u + self.lap(u) / 12.0)

    def solve(self, b):
        """P1 x = b by Richardson sweeps to below 64-bit rounding."""
        b = self.inner(b) * self.h ** 2
        om = 2.0 / (2.0 * self.c1h2 + 16.0 / 3.0)
        x = om * b
        neu = self.neu(b)
        nd = len(neu)
        for _ in range(self.sweeps):
            l = [self.second(x, d, neu[d]) for d in range(nd)]
            p = self.c1h2 * x - sum(l)
            for d in range(nd):
                for e in range(d):
                    p = p - self.second(l[d], e, neu[e]) / 6.0
            x = self.inner(x + om * (b - p))
        return x


def _sin_sources(sc, rows):
    n, dev = sc.n, sc.dev
    out = []
    for m, k, a, w in rows:
        f = sc.beta - sc.h ** 2 / 12.0 * math.pi ** 2 * (m * m + k * k)
        sx, sy = _axis(n, m, True, dev), _axis(n, k, True, dev)
        out.append((-sc.z * (sc.k2 - w * w) * f * a * torch.outer(sy, sx),
                    f * a * w * math.pi * k * torch.outer(_axis(n, k, False, dev), sx),
                    -f * a * w * math.pi * m * torch.outer(sy, _axis(n, m, False, dev)), w))
    return out


def _steps2d(sc, ez, hx, hy, steps, scheme="c4", rows=()):
    src = _sin_sources(sc, rows)
    ez, hx, hy = (sc.inner(v) for v in (ez, hx, hy))
    de = sc.inner(sc.lap(ez)) / sc.h ** 2 if scheme == "c4_de" else None
    for s in range(steps):
        gx, gy = sc.filt(hx), sc.filt(hy)
        rhs = sc.k2 * sc.z * (sc.delta(gy, 1, True) - sc.delta(gx, 0, True))
        for e, _, _, w in src:
            rhs = rhs + math.sin(w * (s + 0.5) * sc.ht) * e
        es = sc.solve(rhs)
        ez = ez + sc.ht * es
        if de is None:
            ge = sc.filt(ez)
        else:
            de = sc.inner(de + sc.k2 * sc.ht * es - sc.z * (24.0 / sc.ht) * (sc.delta(hy, 1, True) - sc.delta(hx, 0, True)))
            ge = sc.beta * ez + sc.h ** 2 / 12.0 * de
        rx = -sc.k2 / sc.z * sc.delta(ge, 0, False)
        ry = sc.k2 / sc.z * sc.delta(ge, 1, False)
        for _, ax, ay, w in src:
            c = math.cos(w * (s + 1.0) * sc.ht)
            rx, ry = rx + c * ax, ry + c * ay
        hx = hx + sc.ht * sc.solve(rx)
        hy = hy + sc.ht * sc.solve(ry)
    return ez, hx, hy


def _steps3d(sc, f, steps):
    f = [sc.inner(v) for v in f]
    for _ in range(steps):
        g = [sc.filt(f[3 + c]) for c in range(3)]
        for e in range(3):
            p, q = (e + 1) % 3, (e + 2) % 3  # dimension of axis a is 2 - a
            r = sc.k2 * sc.z * (sc.delta(g[q], 2 - p, True) - sc.delta(g[p], 2 - q, True))
            f[e] = f[e] + sc.ht * sc.solve(r)
        g = [sc.filt(f[c]) for c in range(3)]
        for c in range(3):
            p, q = (c + 1) % 3, (c + 2) % 3
            r = -sc.k2 / sc.z * (sc.delta(g[q], 2 - p, False) - sc.delta(g[p], 2 - q, False))
            f[3 + c] = f[3 + c] + sc.ht * sc.solve(r)
    return tuple(f)


def _gradient(sc, ez0, lam, steps):
    """E_z after `steps` steps from E_z^0 (H^{1/2} by its Taylor series) and the transposed map of lam."""
    t = 0.5 * sc.ht
    c3 = t ** 3 / 6.0 / sc.h ** 2

    def taylor(v):
        return sc.inner((t * v + c3 * sc.lap(v)) / sc.z)

    e0 = sc.inner(ez0)
    hx, hy = taylor(sc.inner(-sc.delta(e0, 0, False))), taylor(sc.inner(sc.delta(e0, 1, False)))
    ez = _steps2d(sc, e0, hx, hy, steps)[0]
    le = sc.inner(lam)
    lx, ly = torch.zeros_like(hx), torch.zeros_like(hy)
    for _ in range(steps):
        ux, uy = sc.solve(lx), sc.solve(ly)
        v = sc.k2 / sc.z * (sc.delta_t(uy, 1, False) - sc.delta_t(ux, 0, False))
        le = le + sc.ht * sc.filt(sc.inner(v))
        ue = sc.solve(le)
        ly = ly + sc.ht * sc.filt(sc.inner(sc.k2 * sc.z * sc.delta_t(ue, 1, True)))
        lx = lx - sc.ht * sc.filt(sc.inner(sc.k2 * sc.z * sc.delta_t(ue, 0, True)))
    wx, wy = taylor(lx), taylor(ly)
    g = le + sc.inner(sc.delta_t(wy, 1, False) - sc.delta_t(wx, 0, False))
    return ez, g


def exact(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "batch":
        out = []
        sizes = batch_sizes(case)
        for n, rows in zip(sizes, batch_modes(case, seed, sizes)):
            sc = Scheme(n, case["r"], case["z"], case["closure"], dev)
            f = mode_fields(n, case["r"], case["z"], rows, dev)
            out.append([v.cpu() for v in _steps2d(sc, *f, case["steps"])])
        return out
    sc = Scheme(case["n"], case["r"], case["z"], case["closure"], dev)
    if kind == "gradient":
        return _gradient(sc, *gradient_inputs(case, seed, dev), case["steps"])
    if kind == "grid3d":
        return _steps3d(sc, fields3d(case, seed, dev), case["steps"])
    rows = sources2d(case, seed) if case["sources"] else ()
    return _steps2d(sc, *fields2d(case, seed, dev), case["steps"], case["scheme"], rows)
