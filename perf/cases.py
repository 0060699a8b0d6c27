"""The work whose time counts: calls of this package as a reconstruction program makes them.

A case is a dict of plain values: the operation (``op``), the image and grid sizes and
neighbours per axis, the trajectory and its length, and what the operation needs besides
(batch size, coils, iterations).  ``prepare`` makes what such a program holds before the
call (the plan, the images, the samples), ``run`` is one pass through the public entry
points, ``exact`` is the same min-max operator written in plain torch in 64 bits.

Ranges that ``draw`` covers: 1D, 2D and 3D; images of 16 to 512 points per axis, even and
odd multiples, grids 1.25 to 2 times that in products of 2, 3 and 5; 4 to 7 neighbours (6
most often, the usual choice); a few hundred to two million points on radial, spiral,
kooshball, stack-of-stars and uniformly random trajectories.

Inputs: images are smooth-phase ellipses with noise, samples are the analytic transform of
a sum of Gaussian blobs plus noise, so that the centre of k-space is a thousand times
stronger than its edge, as measured data are.
"""
import itertools
import math

import torch

import paper_1710_03197_gb300 as nf

DEV = "cuda"
GOLDEN = math.radians(111.2461)


def _case(name, op, N, K, J, traj, shots, samples, nb=1, iters=0):
    c = {} if name is None else {"name": name}
    c.update(op=op, d=len(N), traj=traj, shots=shots, samples=samples, nb=nb, iters=iters)
    for a in range(len(N)):
        c["N%d" % a], c["K%d" % a], c["J%d" % a] = N[a], K[a], J[a]
    return c


def listed():
    return [
        # a small frame of a real-time or interactive loop: launches and latency
        _case("pair2d_64", "pair", (64, 64), (128, 128), (6, 6), "radial", 64, 128),
        # the usual slice: one forward and one adjoint, golden-angle radial
        _case("pair2d_256", "pair", (256, 256), (512, 512), (6, 6), "radial", 403, 512),
        # a rectangular field of view on a lean 1.5x grid, five neighbours, spirals of odd length
        _case("pair2d_ragged", "pair", (240, 192), (360, 288), (5, 5), "spiral", 13, 3001),
        # the largest 2D grid there is
        _case("pair2d_512", "pair", (512, 512), (1024, 1024), (6, 6), "radial", 805, 1024),
        # the usual volume: 128^3 kooshball, two million points
        _case("pair3d_128", "pair", (128, 128, 128), (256, 256, 256), (6, 6, 6), "koosh", 8192, 256),
        # an anisotropic volume, stack of stars, 1.25x to 1.5x grid, four neighbours
        _case("pair3d_ragged", "pair", (96, 80, 24), (144, 100, 36), (4, 4, 4), "stars", 1101, 145),
        # the inner step of every iterative volume reconstruction
        _case("normal3d_64", "normal", (64, 64, 64), (128, 128, 128), (6, 6, 6), "koosh", 2400, 128),
        # a stack of slices that share a trajectory, forward and adjoint
        _case("batch2d_16", "batch", (192, 192), (384, 384), (6, 6), "radial", 150, 384, nb=16),
        # a dynamic series: 8 frames of uneven length, 32 coils, the normal operator of all of them
        _case("frames_32coils", "frames", (256, 256), (512, 512), (6, 6), "frames", 8, 512, nb=32),
        # trajectory optimisation: new trajectory, loss, gradients of image and trajectory
        _case("grad_spiral", "grad", (256, 256), (512, 512), (6, 6), "spiral", 16, 2048),
        # parallel imaging: multi-coil conjugate gradients
        _case("cg_8coils", "cg_coils", (128, 128), (256, 256), (6, 6), "radial", 101, 256, nb=8, iters=4),
        # compressed sensing: total-variation solver on incoherent samples
        _case("l1tv_random", "l1tv", (128, 128), (256, 256), (6, 6), "random", 1, 40009, iters=3),
    ]


def _smooth(v, most=1024):
    """The smallest even product of 2, 3 and 5 from v up."""
    v = max(16, int(v) + (int(v) & 1))
    while True:
        r = v
        for f in (2, 3, 5):
            while r % f == 0:
                r //= f
        if r == 1:
            return min(v, most)
        v += 2


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["pair", "pair", "pair", "normal", "batch", "frames", "grad", "cg_coils", "l1tv"])
    d = rng.choice([1, 2, 2, 2, 3, 3]) if op == "pair" else rng.choice([2, 3]) if op in ("normal", "batch", "grad") else 2
    hi = {1: 512, 2: 512 if op in ("pair", "normal") else 256, 3: 112 if op in ("pair", "normal") else 48}[d]
    lo = {1: 64, 2: 32, 3: 16}[d]
    n = _log(rng, lo, hi)
    N = tuple(2 * max(8, int(n * rng.uniform(0.7, 1.0)) // 2) for _ in range(d))
    over = rng.choice([1.25, 1.5, 2.0, 2.0])
    K = tuple(_smooth(over * v) for v in N)
    J = (rng.choice([4, 5, 6, 6, 6, 7]),) * d
    traj = rng.choice({1: ["random"], 2: ["radial", "radial", "spiral", "random"], 3: ["koosh", "stars", "random"]}[d])
    nb = {"batch": rng.randint(2, 24), "frames": rng.randint(4, 32), "cg_coils": rng.randint(2, 12)}.get(op, 1)
    iters = {"cg_coils": rng.randint(2, 4), "l1tv": rng.randint(1, 3)}.get(op, 0)
    pts = 1
    for v in N:
        pts *= v
    most = {1: 200_000, 2: 800_000, 3: 1_500_000}[d] // (nb if op in ("batch", "cg_coils") else 1)
    M = max(300, min(most, int(pts * math.exp(rng.uniform(math.log(0.2), math.log(2.5))))))
    samples = max(32, min(M, max(K) + rng.choice([0, 1, -3])))
    shots = max(1, M // samples)
    if op == "frames":
        traj, shots = "frames", rng.randint(2, 8)
    elif op == "l1tv":
        # two points for each pixel, or nearly: what a few iterations solve without magnifying rounding
        traj, samples, shots = "random", max(300, int(2.2 * pts) | 1), 1
    elif traj == "random":
        samples, shots = samples * shots + 1, 1
    return _case(None, op, N, K, J, traj, shots, samples, nb, iters)


# ---------------------------------------------------------------- inputs

def _dims(c):
    return tuple(tuple(c["%s%d" % (k, a)] for a in range(c["d"])) for k in "NKJ")


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _radial(shots, samples, turn, first=0):
    th = turn + GOLDEN * (first + torch.arange(shots, device=DEV, dtype=torch.float64))
    rho = -math.pi + 2 * math.pi * torch.arange(samples, device=DEV, dtype=torch.float64) / samples
    return torch.stack([torch.cos(th)[:, None] * rho, torch.sin(th)[:, None] * rho], -1).reshape(-1, 2)


def _counts(c, seed):
    """Spokes of each frame of a dynamic series: 13 to 89."""
    return torch.randint(13, 90, (c["shots"],), generator=torch.Generator().manual_seed(int(seed) + 17)).tolist()


def _trajectories(c, seed):
    """The trajectories of a case (several for a series), float32 (M, d), in radians."""
    g = _gen(seed)
    S, n, d = c["shots"], c["samples"], c["d"]
    turn = float(_rand(g, 1, hi=math.pi))
    if c["traj"] == "frames":
        out, first = [], 0
        for s in _counts(c, seed):
            out.append(_radial(s, n, turn, first))
            first += s
        return [o.float() for o in out]
    if c["traj"] == "radial":
        om = _radial(S, n, turn)
    elif c["traj"] == "spiral":
        tau = torch.arange(n, device=DEV, dtype=torch.float64) / n
        ang = 2 * math.pi * 8 * tau[None] + 2 * math.pi * torch.arange(S, device=DEV)[:, None] / S + turn
        om = torch.stack([math.pi * tau * torch.cos(ang), math.pi * tau * torch.sin(ang)], -1).reshape(-1, 2)
        om = om + 1e-3 * torch.randn(om.shape, generator=g, device=DEV, dtype=torch.float64)
    elif c["traj"] == "koosh":
        i = torch.arange(S, device=DEV, dtype=torch.float64)
        z = 1 - (2 * i + 1) / S
        phi = turn + i * math.pi * (3 - math.sqrt(5))
        r = torch.sqrt(1 - z * z)
        rho = -math.pi + 2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n
        om = (torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], 1)[:, None] * rho[:, None]).reshape(-1, 3)
    elif c["traj"] == "stars":
        om = _radial(S, n, turn)
        kz = 2 * math.pi * ((torch.arange(S, device=DEV) % c["N2"]) / c["N2"] - 0.5)
        om = torch.cat([om, kz.repeat_interleave(n)[:, None].double()], 1)
    else:
        om = _rand(g, S * n, d, lo=-math.pi, hi=math.pi)
    return [om.float().contiguous()]


def _noise(g, *shape):
    return torch.complex(torch.randn(*shape, generator=g, device=DEV), torch.randn(*shape, generator=g, device=DEV))


def _images(g, nb, N):
    """nb images: ellipses of their own values under a smooth phase, a little noise."""
    ax = torch.meshgrid(*[torch.linspace(-1, 1, n, device=DEV) for n in N], indexing="ij")
    out = []
    for _ in range(nb):
        p = _rand(g, 7, 2 * len(N) + 1, lo=-1.0).float().tolist()
        img = torch.zeros(N, device=DEV)
        for q in p:
            r2 = sum(((x - 0.6 * q[2 * a]) / (0.15 + 0.5 * abs(q[2 * a + 1]))) ** 2 for a, x in enumerate(ax))
            img = img + (0.4 + q[-1]) * (r2 <= 1)
        ph = sum(p[a][0] * x for a, x in enumerate(ax))
        out.append(torch.polar(img, 2 * ph) + 0.01 * _noise(g, *N))
    return torch.stack(out) if nb > 1 else out[0]


def _samples(g, om, nb, N):
    """Samples of nb sums of Gaussian blobs (their analytic transform) plus noise: (nb, M) or (M,)."""
    M, d = om.shape
    y = []
    for _ in range(nb):
        v = torch.zeros(M, device=DEV, dtype=torch.complex64)
        for q in _rand(g, 6, d + 2, lo=-1.0).tolist():
            sig = [(0.02 + 0.1 * abs(q[d])) * n for n in N]
            decay = sum((om[:, a] * sig[a]) ** 2 for a in range(d))
            ph = sum(om[:, a] * (0.4 * q[a] * N[a]) for a in range(d))
            v = v + (0.5 + 0.5 * q[d + 1]) * math.prod(sig) * torch.polar(torch.exp(-0.5 * decay), -ph)
        y.append(v + 0.3 * _noise(g, M))
    return torch.stack(y) if nb > 1 else y[0]


def _coils(g, nc, N):
    ax = torch.meshgrid(*[torch.linspace(-1, 1, n, device=DEV) for n in N], indexing="ij")
    out = []
    for i, q in enumerate(_rand(g, nc, len(N) + 1, lo=-1.0).tolist()):
        cen = [0.8 * math.cos(2 * math.pi * i / nc), 0.8 * math.sin(2 * math.pi * i / nc)] + [0.0] * (len(N) - 2)
        r2 = sum((x - m) ** 2 for x, m in zip(ax, cen))
        out.append(torch.polar(torch.exp(-r2 / 0.9), sum(2 * b * x for b, x in zip(q, ax)) + 3 * q[-1]))
    return torch.stack(out)


def _inputs(c, seed):
    """Everything made from the seed: trajectories, images, samples, coil maps."""
    N, _, _ = _dims(c)
    op, nb = c["op"], c["nb"]
    oms = _trajectories(c, seed)
    g = _gen(seed + 1)
    i = {"oms": oms}
    if op in ("pair", "normal", "batch", "grad"):
        i["x"] = _images(g, nb if op == "batch" else 1, N)
    if op in ("pair", "batch", "grad", "l1tv"):
        i["y"] = _samples(g, oms[0], nb if op == "batch" else 1, N)
    if op == "frames":
        i["x"] = _images(g, len(oms), N).reshape((len(oms),) + N)
        i["coils"] = _coils(g, nb, N)
    if op == "cg_coils":
        i["coils"] = _coils(g, nb, N)
        i["y"] = _samples(g, oms[0], nb, N).reshape(-1)
    return i


def prepare(case, seed):
    """The plan (or plans) of the trajectory, the inputs, and the buffers a loop writes to."""
    N, K, J = _dims(case)
    s = _inputs(case, seed)
    s["case"], s["dims"] = case, (N, K, J)
    s["plans"] = [nf.NufftPlan(om, N, K, J) for om in s["oms"]]
    if case["op"] == "frames":
        s["frames"] = nf.NufftFrames(s["plans"])
        s["out"] = torch.empty_like(s["x"])
    elif case["op"] in ("pair", "batch"):
        s["yo"], s["xo"] = torch.empty_like(s["y"]), torch.empty_like(s["x"])
    elif case["op"] == "normal":
        s["out"] = torch.empty_like(s["x"])
    elif case["op"] == "grad":
        s["om"] = s["oms"][0].clone().requires_grad_(True)
        s["xv"] = s["x"].clone().requires_grad_(True)
    return s


def run(s):
    c, plan = s["case"], s["plans"][0]
    op = c["op"]
    if op == "pair":
        return [nf.nufft_forward(plan, s["x"], s["yo"]), nf.nufft_adjoint(plan, s["y"], s["xo"])]
    if op == "normal":
        return nf.nufft_selfadjoint(plan, s["x"], s["out"])
    if op == "batch":
        return [nf.nufft_forward_batch(plan, s["x"], s["yo"]), nf.nufft_adjoint_batch(plan, s["y"], s["xo"])]
    if op == "frames":
        return s["frames"].selfadjoint_multicoil(s["coils"], s["x"], s["out"])
    if op == "grad":
        N, K, J = s["dims"]
        y = nf.nufft_apply(s["om"], s["xv"], N, K, J, plan=plan, refresh=True)
        r = y - s["y"]
        loss = 0.5 * torch.view_as_real(r).square().sum()
        gom, gx = torch.autograd.grad(loss, (s["om"], s["xv"]))
        return {"y": y.detach(), "gom": gom, "gx": gx}
    if op == "cg_coils":
        return nf.solve_cg_multicoil(plan, s["coils"], s["y"], maxiter=c["iters"])
    # 1/lam lies inside the range of the images' gradients
    return nf.solve_l1tv_ols(plan, s["y"], maxiter=c["iters"], inner=1, cg_iters=3, mu=1.0, lam=5.0)


def work(case):
    """Bytes: each image, sample and frequency once per transform that the operation is made of.
    Operations: 5 K log2 K for a transform of the grid, 8 for a tap."""
    N, K, J = _dims(case)
    n, k, taps, d = math.prod(N), math.prod(K), math.prod(J), case["d"]
    op, nb, it = case["op"], case["nb"], case["iters"]
    M = case["shots"] * case["samples"] if op != "frames" else 51 * case["samples"] * case["shots"]
    fft = 5.0 * k * math.log2(k)
    one = fft + 8.0 * taps * M
    if op in ("pair", "batch"):
        return {"bytes": 2 * nb * 8 * (n + M) + 2 * 4 * d * M, "flops": 2 * nb * one}
    if op == "normal":
        return {"bytes": 16 * n + 4 * d * M, "flops": 2 * one}
    if op == "frames":
        f = case["shots"]
        return {"bytes": 16 * n * f + 8 * n * nb + 4 * d * M, "flops": 2 * nb * (f * fft + 8.0 * taps * M)}
    if op == "grad":
        return {"bytes": 16 * n + 16 * M + 8 * d * M, "flops": 2 * one + 8.0 * d * taps * M}
    if op == "cg_coils":
        return {"bytes": 8 * nb * (M + n) + 8 * n + 4 * d * M, "flops": nb * one * (1 + 2 * (it + 1))}
    return {"bytes": 8 * M + 8 * n + 4 * d * M, "flops": one * (1 + it * 2 * (4 + 1))}


# ---------------------------------------------------------------- 64 bits

class _Exact:
    """A = V F S of the min-max interpolator in complex128, in plain torch."""

    def __init__(self, om, N, K, J):
        self.N, self.K, self.J, self.d = N, K, J, len(N)
        self.om = om.double()
        self.tab = [self._axis(a) for a in range(self.d)]
        self.k, self.c = [], []
        for a in range(self.d):
            k, c = self._coef(a, False)
            self.k.append(k)
            self.c.append(c)
        s = torch.ones((), device=DEV, dtype=torch.float64)
        for t in self.tab:
            s = s[..., None] * t[1]
        self.s = s
        self.place = [(torch.arange(n, device=DEV) - n // 2) % m for n, m in zip(N, K)]

    def _axis(self, a):
        N, K, J = self.N[a], self.K[a], self.J[a]
        t = torch.arange(N, device=DEV, dtype=torch.float64) - N / 2
        q = (2.34 * J) ** 2 - (math.pi * J * t / K) ** 2
        z = q.abs().sqrt()
        ft = torch.where(q > 0, torch.sinh(z) / z, torch.where(q < 0, torch.sin(z) / z, torch.ones_like(z)))
        s = 1 / ft
        s = s / s.max()
        j = torch.arange(1, J + 1, device=DEV, dtype=torch.float64)
        ph = (2 * math.pi / K) * (j[:, None] - j[None])[..., None] * t
        G = torch.complex((torch.cos(ph) * s * s).sum(-1), (torch.sin(ph) * s * s).sum(-1))
        return t, s, torch.linalg.inv(G)

    def _coef(self, a, deriv):
        N, K, J = self.N[a], self.K[a], self.J[a]
        t, s, T = self.tab[a]
        gamma = (2.0 * math.pi) / K
        w = self.om[:, a]
        u = w / gamma
        k0 = torch.floor(u + 0.5) - (J + 1) // 2 if J & 1 else torch.floor(u) - J // 2
        j = torch.arange(1, J + 1, device=DEV, dtype=torch.float64)
        out = torch.empty(w.numel(), J, device=DEV, dtype=torch.complex128)
        for lo in range(0, w.numel(), 1 << 16):
            sl = slice(lo, lo + (1 << 16))
            ph = (w[sl, None] - gamma * (k0[sl, None] + j))[..., None] * t
            v = s * t if deriv else s
            re, im = torch.cos(ph) @ v, -(torch.sin(ph) @ v)
            out[sl] = (torch.complex(im, -re) if deriv else torch.complex(re, im)) @ T.T
        return ((k0[:, None] + j).long() % K), out

    def _taps(self, c):
        """(grid index, weight) of each tap, for all points."""
        for js in itertools.product(*[range(J) for J in self.J]):
            idx, w = None, None
            for a, j in enumerate(js):
                idx = self.k[a][:, j] if idx is None else idx * self.K[a] + self.k[a][:, j]
                w = c[a][:, j] if w is None else w * c[a][:, j]
            yield idx, w

    def spectrum(self, x):
        z = torch.zeros(self.K, device=DEV, dtype=torch.complex128)
        ix = torch.meshgrid(*self.place, indexing="ij")
        z[ix] = self.s * x.to(torch.complex128)
        return torch.fft.fftn(z).reshape(-1)

    def interp(self, grid, c=None):
        y = torch.zeros(self.om.shape[0], device=DEV, dtype=torch.complex128)
        for idx, w in self._taps(self.c if c is None else c):
            y += w * grid[idx]
        return y

    def forward(self, x):
        return self.interp(self.spectrum(x))

    def adjoint(self, y):
        grid = torch.zeros(math.prod(self.K), 2, device=DEV, dtype=torch.float64)
        y = y.to(torch.complex128)
        for idx, w in self._taps(self.c):
            grid.index_add_(0, idx, torch.view_as_real(w.conj() * y))
        z = torch.fft.ifftn(torch.view_as_complex(grid).reshape(self.K), norm="forward")
        return self.s * z[torch.meshgrid(*self.place, indexing="ij")]

    def normal(self, x):
        return self.adjoint(self.forward(x))


def _cg(apply, b, x, iters):
    r = b - apply(x)
    p = r.clone()
    rr = torch.vdot(r.reshape(-1), r.reshape(-1)).real
    for _ in range(iters):
        q = apply(p)
        alpha = rr / torch.vdot(p.reshape(-1), q.reshape(-1)).real
        x = x + alpha * p
        r = r - alpha * q
        new = torch.vdot(r.reshape(-1), r.reshape(-1)).real
        p = r + (new / rr) * p
        rr = new
    return x


def _l1tv(E, y, maxiter, inner, cg_iters, mu, lam):
    axes = range(E.d)
    diff = lambda v, a: torch.roll(v, -1, a) - v  # noqa: E731
    diff_t = lambda v, a: torch.roll(v, 1, a) - v  # noqa: E731

    def K(v):
        out = mu * E.normal(v)
        for a in axes:
            out = out + lam * diff_t(diff(v, a), a)
        return out

    ahy = E.adjoint(y)
    ahyk, x = ahy.clone(), torch.zeros_like(ahy)
    d, b = [torch.zeros_like(x) for _ in axes], [torch.zeros_like(x) for _ in axes]
    for _ in range(maxiter):
        for _ in range(inner):
            rhs = mu * ahyk
            for a in axes:
                rhs = rhs + lam * diff_t(d[a] - b[a], a)
            x = _cg(K, rhs, x, cg_iters)
            for a in axes:
                g = diff(x, a)
                z = g + b[a]
                m = z.abs()
                d[a] = z / m.clamp_min(1e-300) * (m - 1 / lam).clamp_min(0)
                b[a] = b[a] + (g - d[a])
        ahyk = ahyk + ahy - E.normal(x)
    return x


def exact(case, seed):
    N, K, J = _dims(case)
    i = _inputs(case, seed)
    op, nb = case["op"], case["nb"]
    E = _Exact(i["oms"][0], N, K, J)
    if op == "pair":
        return [E.forward(i["x"]), E.adjoint(i["y"])]
    if op == "normal":
        return E.normal(i["x"])
    if op == "batch":
        return [torch.stack([E.forward(v) for v in i["x"]]), torch.stack([E.adjoint(v) for v in i["y"]])]
    coils = i["coils"].to(torch.complex128) if "coils" in i else None
    sense = lambda e, v: sum(m.conj() * e.normal(m * v) for m in coils)  # noqa: E731
    if op == "frames":
        return torch.stack([sense(_Exact(om, N, K, J), v) for om, v in zip(i["oms"], i["x"].to(torch.complex128))])
    if op == "grad":
        grid = E.spectrum(i["x"])
        y = E.interp(grid)
        r = y - i["y"].to(torch.complex128)
        gom = []
        for a in range(E.d):
            c = list(E.c)
            c[a] = E._coef(a, True)[1]
            gom.append((r.conj() * E.interp(grid, c)).real)
        return {"y": y, "gom": torch.stack(gom, 1), "gx": E.adjoint(r)}
    if op == "cg_coils":
        ys = i["y"].reshape(nb, -1)
        b = sum(m.conj() * E.adjoint(v) for m, v in zip(coils, ys))
        return _cg(lambda v: sense(E, v), b, torch.zeros_like(b), case["iters"])
    return _l1tv(E, i["y"], case["iters"], 1, 3, 1.0, 5.0)
