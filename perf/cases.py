"""Performance cases: calls a program makes of this package, with their inputs and exact values.

A case is a dict of plain values:
  op      step     new sample locations, forward, and both gradients (one step of trajectory learning)
          gram     forward and adjoint at unchanged locations (the inner loop of a reconstruction)
          forward, adjoint, vjp   one of them at unchanged locations
          jvp      directional derivative in the locations, with the forward values
          inverse  regularised least-squares image by CG and its implicit gradient (autograd layer)
  shape   image size, "320x320"; C coils, or C images when maps is false; M sample locations
  traj    "radial" (golden-angle spokes in 2-D, Fibonacci-sphere spokes with a random walk in 3-D,
          readouts of twice the longest side, the last one cut) or "uniform"
  sigma, J, deterministic   plan options

The inputs are random, but shaped like the package's workloads: complex Gaussian images and incoming
gradients, smooth Gaussian-bump coil maps, spokes through the k-space centre.
"""
import math

import torch

from paper_2111_02912_gb300 import Plan
from paper_2111_02912_gb300.autograd import NufftOperator, psd_inverse

CG_ITERS = 10        # CG iterations of the forward and of the implicit backward of op "inverse"
CG_LAMBDA = 0.1      # its regularisation, times M
GOLDEN = math.radians(111.246117975)


def _case(name, op, shape, C, M, maps=True, traj="radial", sigma=2.0, J=6, deterministic=False):
    return dict(name=name, op=op, shape=shape, C=C, M=M, maps=maps, traj=traj, sigma=sigma, J=J,
                deterministic=deterministic)


def listed():
    return [
        # one spoke on a 40^2 image: the smallest step, all launches and host time
        _case("spoke40_step", "step", "40x40", 8, 80),
        # a small image without maps at random locations
        _case("uniform64_step", "step", "64x64", 1, 4096, maps=False, traj="uniform"),
        # an uneven image, an odd coil count, an odd number of samples, a grid edge (450) that is no round number
        _case("ragged150x218_step", "step", "150x218", 5, 30011),
        # the ordinary case: 320^2, 16 coils, 80 spokes of 640 samples, one trajectory-learning step
        _case("radial320_step", "step", "320x320", 16, 51200),
        # the same at the low-accuracy setting (grid ratio 1.25, five taps)
        _case("radial320_low_step", "step", "320x320", 16, 51200, sigma=1.25, J=5),
        # the same as the inner loop of a reconstruction: fixed trajectory, forward and adjoint
        _case("radial320_gram", "gram", "320x320", 16, 51200),
        # the largest 2-D problem of a batch: 384^2, 32 coils, 200,000 samples
        _case("coils32_384_step", "step", "384x384", 32, 200000),
        # a short series of images without maps (frames of one trajectory)
        _case("frames256_gram", "gram", "256x256", 4, 65537, maps=False),
        # forward-mode derivative with the forward values, on a rectangle (Gauss-Newton, sensitivity)
        _case("jvp192x256", "jvp", "192x256", 12, 99999),
        # regularised inverse by CG and its implicit gradient through the autograd layer, trajectory updated
        _case("inverse320", "inverse", "320x320", 16, 51200),
        # 3-D radial, 8 coils, two million samples: one trajectory-learning step
        _case("radial3d_step", "step", "128x128x96", 8, 2000000),
        # an uneven 3-D volume (grid edges 180, 200 and 144), six coils: reconstruction inner loop
        _case("ragged3d_gram", "gram", "90x100x70", 6, 500003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    D = 3 if rng.random() < 0.25 else 2
    if D == 2:
        a = 2 * _log_int(rng, 16, 192)
        b = a if rng.random() < 0.5 else 2 * _log_int(rng, 16, 192)
        shape = "%dx%d" % (a, b)
        C, M = _log_int(rng, 1, 32), _log_int(rng, 80, 200000)
        op = rng.choice(["step", "step", "step", "gram", "gram", "forward", "adjoint", "vjp", "jvp", "inverse"])
    else:
        shape = "%dx%dx%d" % tuple(2 * _log_int(rng, 10, top) for top in (64, 64, 48))
        C, M = _log_int(rng, 1, 8), _log_int(rng, 4000, 2000000)
        op = rng.choice(["step", "step", "gram", "gram", "forward", "adjoint", "vjp"])
    sigma, J = rng.choice([(2.0, 6), (2.0, 6), (2.0, 6), (2.0, 6), (1.25, 5), (2.0, 4)])
    c = _case("", op, shape, C, M, maps=op == "inverse" or rng.random() < 0.7, traj=rng.choice(["radial", "radial", "uniform"]),
              sigma=sigma, J=J, deterministic=op in ("step", "gram") and rng.random() < 0.15)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------- inputs

def _shape(case):
    return tuple(int(n) for n in case["shape"].split("x"))


def _trajectory(case, g, dev):
    shape, M = _shape(case), case["M"]
    D = len(shape)
    if case["traj"] == "uniform":
        return (torch.rand((D, M), generator=g, device=dev, dtype=torch.float64) * (2 * math.pi) - math.pi).float()
    n_read = 2 * max(shape)
    n_spokes = -(-M // n_read)
    turn = float(torch.rand((), generator=g, device=dev)) * 2 * math.pi
    i = torch.arange(n_spokes, device=dev, dtype=torch.float64)
    kr = math.pi * (2.0 * torch.arange(n_read, device=dev, dtype=torch.float64) / n_read - 1.0)
    if D == 2:
        th = GOLDEN * i + turn
        dirs = torch.stack([torch.cos(th), torch.sin(th)])
        sd = 5e-4 * math.pi
    else:
        z = 1.0 - 2.0 * (i + 0.5) / n_spokes
        phi = math.pi * (3.0 - math.sqrt(5.0)) * (i + 0.5) + turn
        s = torch.sqrt(1.0 - z * z)
        dirs = torch.stack([s * torch.cos(phi), s * torch.sin(phi), z])
        sd = 2e-3 * math.pi
    om = dirs[:, :, None] * kr
    step = torch.randn(om.shape, generator=g, device=dev, dtype=torch.float64) * sd
    om = om + torch.cumsum(step, dim=2)
    om = torch.remainder(om + math.pi, 2 * math.pi) - math.pi
    return om.reshape(D, -1)[:, :M].float().contiguous()


def _maps(case, g, dev):
    shape, C = _shape(case), case["C"]
    D, ref = len(shape), float(max(shape))
    turn = float(torch.rand((), generator=g, device=dev)) * 2 * math.pi
    c = torch.arange(C, device=dev, dtype=torch.float32)
    ang = 2 * math.pi * c / C + turn
    z = 1.0 - (2.0 * c + 1.0) / C if D == 3 else torch.zeros_like(c)
    s = torch.sqrt(1.0 - z * z)
    centre = 0.4 * ref * torch.stack([s * torch.cos(ang), s * torch.sin(ang), z])[:D]
    d2 = torch.zeros((C,) + shape, device=dev)
    for d in range(D):
        r = torch.arange(shape[d], device=dev, dtype=torch.float32) - shape[d] // 2
        v = (r[None] - centre[d][:, None]) ** 2
        d2 = d2 + v.reshape((C,) + tuple(shape[d] if e == d else 1 for e in range(D)))
    ph = (2 * math.pi * c / C).reshape((C,) + (1,) * D)
    return torch.polar(torch.exp(-d2 / (2 * (0.35 * ref) ** 2)), ph.expand_as(d2).contiguous())


def _inputs(case, seed):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(1_000_003 + seed)
    shape, C, M = _shape(case), case["C"], case["M"]
    cplx = lambda *n: torch.randn(n, generator=g, device=dev, dtype=torch.complex64)
    q = dict(omega=_trajectory(case, g, dev), smaps=_maps(case, g, dev) if case["maps"] else None)
    q["x"] = cplx(*(shape if case["maps"] else (C,) + shape))
    q["v"] = cplx(C, M)
    if case["op"] == "jvp":
        q["domega"] = torch.randn((len(shape), M), generator=g, device=dev) * 1e-2
    if case["op"] == "inverse":
        q["b"], q["g"] = q["x"], cplx(*shape)
    return q


def prepare(case, seed):
    s = _inputs(case, seed)
    s["op"] = case["op"]
    shape, C = _shape(case), case["C"]
    if case["op"] == "inverse":
        s["param"] = s["omega"].clone().requires_grad_(True)
        s["b"] = s["b"].requires_grad_(True)
        s["lam"] = CG_LAMBDA * case["M"]
        s["E"] = NufftOperator(shape, s["param"], s["smaps"], J=case["J"], sigma=case["sigma"], max_coils=C)
    else:
        s["plan"] = Plan(shape, s["omega"], J=case["J"], sigma=case["sigma"], max_coils=C,
                         deterministic=case["deterministic"])
        if case["op"] != "step":
            s["plan"].sort_points()
    return s


def run(s):
    op = s["op"]
    if op == "inverse":
        with torch.no_grad():
            s["param"].copy_(s["omega"])     # where a training loop's optimiser writes the trajectory
        z = psd_inverse(s["b"], s["param"], s["E"], s["lam"], CG_ITERS)
        gb, go = torch.autograd.grad(z, (s["b"], s["param"]), s["g"])
        return z, gb, go
    plan, x, smaps = s["plan"], s["x"], s["smaps"]
    if op == "step":
        plan.set_points(s["omega"])
        y = plan.forward(x, smaps)
        go, gx = plan.vjp_omega_x(x, s["v"], smaps)
        return y, go, gx
    if op == "gram":
        y = plan.forward(x, smaps)
        return y, plan.adjoint(y, smaps)
    if op == "forward":
        return plan.forward(x, smaps)
    if op == "adjoint":
        return plan.adjoint(s["v"], smaps)
    if op == "vjp":
        return plan.vjp_omega_x(x, s["v"], smaps)
    return plan.jvp_omega(x, s["domega"], smaps, want_y=True)


# ------------------------------------------------------------------------------- what it takes

def _grid(n, sigma):
    k = math.ceil(sigma * n - 1e-9)
    while True:
        q = k
        for p in (2, 3, 5):
            while q % p == 0:
                q //= p
        if k % 2 == 0 and q == 1:
            return k
        k += 1


def work(case):
    shape, C, M, J, op = _shape(case), case["C"], case["M"], case["J"], case["op"]
    D, n = len(shape), math.prod(shape)
    images = n if case["maps"] else C * n
    img, maps, om, ksp = 8 * images, 8 * C * n if case["maps"] else 0, 4 * D * M, 8 * C * M
    K = math.prod(_grid(m, case["sigma"]) for m in shape)
    one = 4 * M * J ** D + 5 * K * math.log2(K)        # one channel: taps and the grid's transform
    nbytes, channels = {
        "step": (img + maps + om + ksp + ksp + om + img, C * (2 + D)),
        "gram": (img + maps + om + ksp + img, 2 * C),
        "forward": (img + maps + om + ksp, C),
        "adjoint": (ksp + maps + om + img, C),
        "vjp": (img + maps + om + ksp + om + img, C * (1 + D)),
        "jvp": (img + maps + 2 * om + 2 * ksp, C * (1 + D)),
        "inverse": (4 * img + maps + 2 * om, C * (2 * 2 * CG_ITERS + 2 + 2 * D)),
    }[op]
    return {"bytes": nbytes, "flops": channels * one}


# ------------------------------------------------------------------------------- exact values
# The same operator in 64 bits: Kaiser-Bessel interpolation of the zero-padded, scaled image's
# transform and its transpose, by torch's FFT, gathers and index_add.

class _Exact:
    def __init__(self, case, omega):
        self.shape, self.D = _shape(case), len(_shape(case))
        self.K = tuple(_grid(n, case["sigma"]) for n in self.shape)
        J, dev = case["J"], omega.device
        beta = math.pi * math.sqrt((J / case["sigma"]) ** 2 * (case["sigma"] - 0.5) ** 2 - 0.8)
        self.scale = torch.ones(self.shape, dtype=torch.float64, device=dev)
        self.r = []
        self.start, self.w = [], []
        taps = torch.arange(J, device=dev)
        for d in range(self.D):
            r = torch.arange(self.shape[d], device=dev, dtype=torch.float64) - self.shape[d] // 2
            a = torch.sqrt(beta ** 2 - (math.pi * J * r / self.K[d]) ** 2)
            along = tuple(-1 if e == d else 1 for e in range(self.D))
            self.scale = self.scale * (a / (J * torch.sinh(a))).reshape(along)
            self.r.append(r.reshape(along))
            t = omega[d].double() * (self.K[d] / (2 * math.pi))
            k = (torch.floor(t - J / 2).long() + 1)[:, None] + taps
            u = t[:, None] - k
            z = torch.clamp(1.0 - (2.0 * u / J) ** 2, min=0.0)
            self.w.append(torch.where(u.abs() < J / 2, torch.special.i0(beta * torch.sqrt(z)), torch.zeros_like(z)))
            self.start.append(torch.remainder(k, self.K[d]))
        self.M, self.chunk = omega.shape[1], max(1, (1 << 23) // J ** self.D)

    def _taps(self, lo):
        hi = min(self.M, lo + self.chunk)
        idx, w = self.start[0][lo:hi], self.w[0][lo:hi]
        for d in range(1, self.D):
            idx = (idx[:, :, None] * self.K[d] + self.start[d][lo:hi, None, :]).reshape(hi - lo, -1)
            w = (w[:, :, None] * self.w[d][lo:hi, None, :]).reshape(hi - lo, -1)
        return hi, idx, w

    def forward(self, imgs):
        C, dims = imgs.shape[0], tuple(range(1, self.D + 1))
        g = torch.zeros((C,) + self.K, dtype=torch.complex128, device=imgs.device)
        g[(slice(None),) + tuple(slice(0, n) for n in self.shape)] = imgs * self.scale
        g = torch.fft.fftn(torch.roll(g, [-(n // 2) for n in self.shape], dims), dim=dims)
        g = g.reshape(C, -1).t().contiguous()
        y = torch.empty((C, self.M), dtype=torch.complex128, device=imgs.device)
        for lo in range(0, self.M, self.chunk):
            hi, idx, w = self._taps(lo)
            for c in range(0, C, 8):
                y[c:c + 8, lo:hi] = (w[:, :, None] * g[idx, c:c + 8]).sum(1).t()
        return y

    def adjoint(self, y):
        C, K = y.shape[0], math.prod(self.K)
        g = torch.zeros((K, 2 * C), dtype=torch.float64, device=y.device)
        for lo in range(0, self.M, self.chunk):
            hi, idx, w = self._taps(lo)
            for c in range(0, C, 8):
                v = torch.view_as_real(y[c:c + 8, lo:hi].t().contiguous()).reshape(hi - lo, 1, -1)
                part = g[:, 2 * c:2 * c + 16] if C > 8 else g
                part.index_add_(0, idx.reshape(-1), (w[:, :, None] * v).reshape(-1, v.shape[2]))
        g = torch.view_as_complex(g.reshape(K, C, 2)).t().reshape((C,) + self.K)
        dims = tuple(range(1, self.D + 1))
        x = torch.roll(torch.fft.ifftn(g, dim=dims, norm="forward"), [n // 2 for n in self.shape], dims)
        return x[(slice(None),) + tuple(slice(0, n) for n in self.shape)] * self.scale


def exact(case, seed):
    q = _inputs(case, seed)
    S = q["smaps"].to(torch.complex128) if q["smaps"] is not None else None
    up = lambda t: t.to(torch.complex128)
    E = _Exact(case, q["omega"])
    fwd = lambda x: E.forward(S * x if S is not None else x)
    adj = lambda y: (E.adjoint(y) * S.conj()).sum(0) if S is not None else E.adjoint(y)
    # d/d omega_d of E x is -i E (r_d x)
    vjp = lambda x, v: torch.stack([(v.conj() * -1j * fwd(x * r)).real.sum(0) for r in E.r])
    op = case["op"]
    if op == "inverse":
        lam = CG_LAMBDA * case["M"]

        def cg(b):
            x, r = torch.zeros_like(b), b.clone()
            p, rr = r.clone(), (b.conj() * b).sum().real
            for _ in range(CG_ITERS):
                Fp = adj(fwd(p)) + lam * p
                alpha = rr / (p.conj() * Fp).sum().real
                x, r = x + alpha * p, r - alpha * Fp
                new = (r.conj() * r).sum().real
                p, rr = r + (new / rr) * p, new
            return x

        z, u = cg(up(q["b"])), cg(up(q["g"]))
        return z, u, -(vjp(z, fwd(u)) + vjp(u, fwd(z)))
    x, v = up(q["x"]), up(q["v"])
    if op == "step":
        return fwd(x), vjp(x, v), adj(v)
    if op == "gram":
        y = fwd(x)
        return y, adj(y)
    if op == "forward":
        return fwd(x)
    if op == "adjoint":
        return adj(v)
    if op == "vjp":
        return vjp(x, v), adj(v)
    dom = q["domega"].double()
    return sum(dom[d] * -1j * fwd(x * E.r[d]) for d in range(E.D)), fwd(x)
