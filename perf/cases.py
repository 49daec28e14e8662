"""The work that users of this library have it do, as cases to be timed.

A case is one call of a public entry point (``claire.Registration``,
``claire.solve_batch``, ``autograd.transport_mismatch``) on inputs shaped like
the repository's workloads: "brain-like" blob images (overlapping ellipsoids,
smoothed with sigma = 2 voxels), band-limited velocities that displace by a
few voxels, beta = 1e-2, gamma = 1.  Inputs are made on the GPU from the seed.
``exact`` evaluates the same discrete method in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2008_12820_gb300 import claire
from paper_2008_12820_gb300.autograd import transport_mismatch

TWO_PI = 2.0 * math.pi
BETA, GAMMA = 1e-2, 1.0


def _case(kind, shape, nt=4, disp=4.0, precision="fp32", scheme="spectral", name=None, **more):
    c = dict(kind=kind, n1=shape[0], n2=shape[1], n3=shape[2], nt=nt, disp=disp, precision=precision,
             scheme=scheme, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the preconditioner of the 32^3 plain-method workload: five launches
        # on a grid that a few SMs hold, so launches and host calls count
        _case("precond", (32, 32, 32), name="precond_32"),
        # the preconditioner at the headline grid: one application per PCG iteration
        _case("precond", (256, 256, 256), name="precond_256"),
        # forward transport + mismatch of a small pair of a batch (a line-search trial)
        _case("forward", (64, 64, 64), name="forward_64"),
        # reduced gradient with objective, the start of every Gauss-Newton step
        _case("gradient", (128, 128, 128), name="gradient_128"),
        # the FP16-storage form, more time steps and large displacements
        # (tiles whose foot points spread over several cells)
        _case("gradient", (160, 160, 160), nt=8, disp=12.0, precision="fp16", name="gradient_fp16_160"),
        # the Gauss-Newton Hessian matvec of the headline workload
        _case("matvec", (256, 256, 256), name="matvec_256"),
        # the same on an odd grid: lengths with factors 3 and 5, rows that are
        # not a whole number of 16-byte chunks, ragged tiles
        _case("matvec", (120, 135, 150), name="matvec_120x135x150"),
        # the paper's own GPU discretization: trilinear interpolation, FD8 derivatives
        _case("matvec", (192, 192, 192), scheme="linear_fd8", name="matvec_linear_192"),
        # differentiable transport inside a training step: forward and backward,
        # states recomputed from checkpoints, a ragged anisotropic grid
        _case("autograd", (160, 128, 192), stride=2, name="autograd_160x128x192"),
        # several small registrations of uneven grids at once
        _case("batch", (64, 96, 80), pairs=4, name="batch_4"),
        # a full registration with the two-level preconditioner
        _case("solve", (128, 128, 128), precond="2LinvH0", name="solve_2l_128"),
        # the headline: a full Gauss-Newton-Krylov registration of a 256^3 pair
        _case("solve", (256, 256, 256), precond="invA", name="solve_256"),
    ]


# grid lengths of the range: products of 2, 3 and 5
_LENGTHS = sorted(a * b * c for a in (1, 2, 4, 8, 16, 32, 64, 128, 256) for b in (1, 3, 9, 27) for c in (1, 5, 25)
                  if 32 <= a * b * c <= 256)


def _length(rng, lo, hi):
    """a valid length near a size drawn evenly over the logarithm of [lo, hi]"""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ok = [n for n in _LENGTHS if lo <= n <= hi]
    return min(ok, key=lambda n: (abs(math.log(n / x)), n))


def draw(rng):
    kind = rng.choice(["precond", "forward", "gradient", "matvec", "matvec", "autograd", "batch", "solve"])
    disp = round(math.exp(rng.uniform(math.log(1.0), math.log(12.0))), 2)
    if kind == "batch":
        return _case(kind, tuple(_length(rng, 48, 128) for _ in range(3)), disp=min(disp, 4.0),
                     pairs=rng.randint(2, 6))
    if kind == "solve":
        n = _length(rng, 48, 160)
        even = [m for m in (64, 80, 96, 120, 128, 144, 160) if m <= max(n, 64)]
        pc = rng.choice(["invA", "2LinvH0"])
        shape = (n, _length(rng, 48, 160), _length(rng, 48, 160)) if pc == "invA" else \
            (even[-1], rng.choice(even), rng.choice(even))
        return _case(kind, shape, disp=min(disp, 4.0), precond=pc)
    lo, hi = (32, 256) if kind in ("precond", "matvec") else (48, 200)
    if rng.random() < 0.4:
        shape = (_length(rng, lo, hi),) * 3
    else:
        shape = tuple(_length(rng, lo, hi) for _ in range(3))
    if kind == "precond":
        return _case(kind, shape)
    nt = rng.choice([3, 4, 4, 8])
    if kind == "autograd":
        return _case(kind, shape, nt=nt, disp=disp, stride=rng.choice([1, 2, 2, 3]))
    if kind == "forward":
        return _case(kind, shape, nt=nt, disp=disp, scheme=rng.choice(["spectral", "spectral", "linear_fd8"]))
    return _case(kind, shape, nt=nt, disp=disp, precision=rng.choice(["fp32", "fp32", "fp16"]),
                 scheme=rng.choice(["spectral", "spectral", "linear_fd8"]))


# ------------------------------------------------------------------ inputs --

def _axes(shape, dtype=torch.float32):
    ax = [torch.arange(n, device="cuda", dtype=dtype) for n in shape]
    return torch.meshgrid(*ax, indexing="ij")


def _smooth_field(shape, rng, kmax=6, comps=3):
    """random periodic fields with wavenumbers up to kmax and a 1/(1+|k|^2)
    amplitude decay (float32 [comps, *shape])"""
    kmax = min(kmax, min(shape) // 2 - 1)
    k = np.arange(-kmax, kmax + 1)
    k3 = np.arange(0, kmax + 1)
    amp = 1.0 / (1.0 + k[:, None, None] ** 2 + k[None, :, None] ** 2 + k3[None, None, :] ** 2)
    z = (rng.standard_normal((comps,) + amp.shape) + 1j * rng.standard_normal((comps,) + amp.shape)) * amp
    z = torch.from_numpy(z.astype(np.complex64)).cuda()
    E = [torch.polar(torch.ones((), device="cuda"),
                     (TWO_PI / n) * torch.outer(torch.arange(n, device="cuda").float(),
                                                torch.from_numpy(kk).cuda().float()))
         for n, kk in zip(shape, (k, k, k3))]
    out = []
    for c in range(comps):
        f = torch.einsum("abc,zc->abz", z[c], E[2])
        f = torch.einsum("abz,yb->ayz", f, E[1])
        # the real part of the last contraction as two real products
        out.append(torch.einsum("ayz,xa->xyz", f.real.contiguous(), E[0].real.contiguous())
                   - torch.einsum("ayz,xa->xyz", f.imag.contiguous(), E[0].imag.contiguous()))
    return torch.stack(out)


def _velocity(shape, rng, disp):
    """band-limited velocity that moves points by at most disp voxels over unit time"""
    v = _smooth_field(shape, rng)
    return v * (disp * (TWO_PI / min(shape)) / v.square().sum(0).sqrt().max())


def _blur(img, sigma=2.0):
    w = [torch.exp(-0.5 * (sigma * TWO_PI * torch.fft.fftfreq(n, device="cuda")) ** 2) for n in img.shape[:2]]
    w.append(torch.exp(-0.5 * (sigma * TWO_PI * torch.fft.rfftfreq(img.shape[2], device="cuda")) ** 2))
    F = torch.fft.rfftn(img) * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
    return torch.fft.irfftn(F, s=img.shape).contiguous()


def _images(shape, rng, v):
    """template of 12 overlapping ellipsoids and the same ellipsoids displaced by v"""
    ext = torch.tensor(shape, device="cuda", dtype=torch.float32)
    grid = torch.stack(_axes(shape))
    scale = torch.tensor([n / TWO_PI for n in shape], device="cuda")[:, None, None, None]
    moved = grid - v * scale
    imgs = [torch.zeros(shape, device="cuda"), torch.zeros(shape, device="cuda")]
    n = np.array(shape, dtype=np.float64)
    for _ in range(12):
        centre = torch.from_numpy((rng.uniform(0.15, 0.85, 3) * n).astype(np.float32)).cuda()
        semi = torch.from_numpy((rng.uniform(0.06, 0.14, 3) * n).astype(np.float32)).cuda()
        q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
        R = torch.from_numpy(q.astype(np.float32)).cuda()
        value = float(rng.uniform(0.2, 1.0))
        for img, pts in zip(imgs, (grid, moved)):
            rel = pts - centre[:, None, None, None]
            rel = rel - ext[:, None, None, None] * torch.round(rel / ext[:, None, None, None])
            r2 = 0.0
            for a in range(3):
                r2 = r2 + ((R[0, a] * rel[0] + R[1, a] * rel[1] + R[2, a] * rel[2]) / semi[a]).square()
            img[r2 <= 1.0] = value
    return _blur(imgs[0]), _blur(imgs[1])


def _shape(case):
    return case["n1"], case["n2"], case["n3"]


def _problem(shape, seed, disp):
    """images of a pair, the velocity that relates them, and an iterate on the way to it"""
    rng = np.random.default_rng(seed)
    v = _velocity(shape, rng, disp)
    m0, m1 = _images(shape, rng, v)
    return m0, m1, (0.7 * v).contiguous(), rng


def _inputs(case, seed):
    """every input tensor of a case, from the seed alone"""
    shape = _shape(case)
    if case["kind"] == "precond":
        # a PCG residual: smooth structure plus broad-band roughness
        rng = np.random.default_rng(seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        return dict(r=_smooth_field(shape, rng) +
                    0.1 * torch.randn((3,) + shape, generator=gen, device="cuda"))
    m0, m1, v, rng = _problem(shape, seed, case["disp"])
    d = dict(m0=m0, m1=m1, v=v)
    if case["kind"] == "matvec":
        d["vt"] = _velocity(shape, rng, case["disp"])  # a PCG direction
    return d


def _registration(case, shape, stream=None):
    reg = claire.Registration(shape, case["nt"], BETA, GAMMA, stream=stream, precision=case["precision"])
    if case["scheme"] == "linear_fd8":
        reg.set_discretization("linear", "fd8")
    return reg


def _batch_shapes(case):
    """uneven grids from the case's three lengths"""
    a = _shape(case)
    every = [(a[0],) * 3, (a[1],) * 3, (a[0], a[1], a[2]), (a[2], a[0], a[1]), (a[2],) * 3, (a[1], a[2], a[0])]
    return every[:case["pairs"]]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        s = dict(case=case, regs=[], vs=[])
        for i, shape in enumerate(_batch_shapes(case)):
            m0, m1, v, _ = _problem(shape, seed + 1000003 * i, case["disp"])
            reg = _registration(case, shape)
            reg.set_images(m0, m1)
            s["regs"].append(reg)
            s["vs"].append(torch.zeros_like(v))
        return s
    shape = _shape(case)
    x = _inputs(case, seed)
    s = dict(case=case)
    if kind == "solve":
        # the solver runs on a stream of its own, as the README advises (its
        # loops then run as CUDA graphs)
        s["stream"] = torch.cuda.Stream()
        s["reg"] = _registration(case, shape, s["stream"])
        s["stream"].wait_stream(torch.cuda.current_stream())
        s["reg"].set_images(x["m0"], x["m1"])
        s["v"] = torch.zeros((3,) + shape, device="cuda")
        torch.cuda.synchronize()
        return s
    s["reg"] = _registration(case, shape)
    if kind == "precond":
        s["r"], s["out"] = x["r"], torch.empty_like(x["r"])
        return s
    s["reg"].set_images(x["m0"], x["m1"])
    s["v"] = x["v"]
    if kind == "matvec":
        s["reg"].linearize(x["v"])
        s["vt"], s["out"] = x["vt"], torch.empty_like(x["vt"])
    elif kind == "gradient":
        s["out"] = torch.empty_like(x["v"])
    elif kind == "autograd":
        s["v"] = x["v"].requires_grad_(True)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "precond":
        return s["reg"].precond(s["r"], out=s["out"])
    if kind == "forward":
        m, mis = s["reg"].forward(s["v"])
        return [m, mis]
    if kind == "gradient":
        g, J = s["reg"].gradient(s["v"], out=s["out"])
        return [g, J]
    if kind == "matvec":
        return s["reg"].hess_matvec(None, s["vt"], out=s["out"])
    if kind == "autograd":
        v = s["v"]
        v.grad = None
        mis, m = transport_mismatch(v, s["reg"], case["stride"])
        # mismatch plus a brightness term of the warped image
        loss = mis.float() + 5.0 * m.square().mean()
        loss.backward()
        return [loss.detach(), m.detach(), v.grad]
    if kind == "batch":
        for v in s["vs"]:
            v.zero_()
        claire.solve_batch(s["regs"], s["vs"], max_gn=4)
        return list(s["vs"])
    v, st = s["v"], s["stream"]
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        v.zero_()
        rep = s["reg"].solve(v, precond=case["precond"], max_gn=4)
    torch.cuda.current_stream().wait_stream(st)
    return [v, rep.J]


# -------------------------------------------------------------------- work --

def work(case):
    """Bytes and operations of one pass: inputs and the kept linearization
    read once, outputs written once; 64 (or 8) taps per interpolation, the
    transforms at 2.5 N log2 N operations per real field."""
    kind, nt = case["kind"], case["nt"]
    if kind == "batch":
        total = dict(bytes=0.0, flops=0.0)
        for shape in _batch_shapes(case):
            w = _work_solve(shape, case)
            total = {k: total[k] + w[k] for k in total}
        return total
    if kind == "solve":
        return _work_solve(_shape(case), case)
    return _work_one(kind, _shape(case), case, nt)


def _work_one(kind, shape, case, nt):
    N = float(shape[0] * shape[1] * shape[2])
    interp = 2.0 * 8 if case["scheme"] == "linear_fd8" else 2.0 * 64
    fft = 2.5 * math.log2(N)
    deriv = 2 * 2.5 * math.log2(N) / 3  # one axis, forward and back
    tb = 2 if case["precision"] == "fp16" else 4  # bytes of a stored trajectory value
    foot = 3 * interp
    if kind == "precond":
        return dict(bytes=24 * N, flops=N * (6 * fft + 30))
    if kind == "forward":  # v, m0, m1 in; m(1) out
        return dict(bytes=24 * N, flops=N * (foot + nt * interp))
    if kind == "matvec":  # vt, X-, X+, c, grad m^j in; the product out
        return dict(bytes=N * (12 + 24 + 4 + 3 * tb * (nt + 1) + 12), flops=N * (2 * nt * interp + 6 * fft))
    lin = N * (2 * foot + (nt + 1) * interp + (3 * (nt + 1) + 3) * deriv)
    if kind == "autograd":  # v, m0, m1 in; m(1), its gradient and grad v out
        return dict(bytes=40 * N, flops=lin + N * nt * interp)
    # gradient: v, m0, m1 in; g and the linearization kept for the matvecs out
    # (X-, X+, m^j, grad m^j, div v, c, lambda^j)
    return dict(bytes=N * (20 + 12 + 24 + 8 + 5 * tb * (nt + 1)), flops=lin + N * (nt * interp + 6 * fft))


def _work_solve(shape, case):
    """three Gauss-Newton steps with four PCG iterations each, the usual count
    of these pairs: a gradient, a line-search trial, matvecs, preconditioners"""
    total = dict(bytes=0.0, flops=0.0)
    for kind, times in (("gradient", 4), ("forward", 3), ("matvec", 11), ("precond", 11)):
        w = _work_one(kind, shape, case, case["nt"])
        total = {k: total[k] + times * w[k] for k in total}
    return total


# ------------------------------------------------------------------- exact --

class _Exact:
    """The discrete method in 64 bits with plain torch operations."""

    def __init__(self, case, shape):
        self.shape, self.nt, self.linear = shape, case["nt"], case["scheme"] == "linear_fd8"
        self.dt = 1.0 / self.nt
        self.idx = [torch.arange(n, device="cuda").view([-1 if a == b else 1 for b in range(3)])
                    for a, n in enumerate(shape)]
        self.ih = [n / TWO_PI for n in shape]
        self.h3 = math.prod(TWO_PI / n for n in shape)

    def interp(self, f, disp):
        n1, n2, n3 = self.shape
        strides = (n2 * n3, n3, 1)
        offs, wts = [], []
        for a in range(3):
            fl = torch.floor(disp[a])
            t = disp[a] - fl
            if self.linear:
                w, first = [1 - t, t], 0
            else:
                w = [-t * (t - 1) * (t - 2) / 6, (t + 1) * (t - 1) * (t - 2) / 2, -(t + 1) * t * (t - 2) / 2,
                     (t + 1) * t * (t - 1) / 6]
                first = -1
            base = self.idx[a] + fl.long() + first
            offs.append([torch.remainder(base + k, self.shape[a]) * strides[a] for k in range(len(w))])
            wts.append(w)
        flat, out = f.reshape(-1), 0.0
        for o1, w1 in zip(offs[0], wts[0]):
            for o2, w2 in zip(offs[1], wts[1]):
                row, w12 = o1 + o2, w1 * w2
                for o3, w3 in zip(offs[2], wts[2]):
                    out = out + w12 * w3 * flat[row + o3]
        return out

    def foot(self, v, s):
        q = [s * self.dt * v[a] * self.ih[a] for a in range(3)]
        return [0.5 * s * self.dt * (v[a] + self.interp(v[a], q)) * self.ih[a] for a in range(3)]

    def freq(self, a, nyquist):
        n = self.shape[a]
        k = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
        if not nyquist and n % 2 == 0:
            k[n // 2] = 0.0
        return k.view([-1 if a == b else 1 for b in range(3)])

    def deriv(self, f, a):
        if self.linear:
            r = 0.0
            for j, c in enumerate((4 / 5, -1 / 5, 4 / 105, -1 / 280), 1):
                r = r + c * (torch.roll(f, -j, a) - torch.roll(f, j, a))
            return r * self.ih[a]
        return torch.fft.ifft(1j * self.freq(a, False) * torch.fft.fft(f, dim=a), dim=a).real

    def grad(self, f):
        return torch.stack([self.deriv(f, a) for a in range(3)])

    def regular(self, v, inverse):
        F = torch.stack([torch.fft.fftn(v[c]) for c in range(3)])
        k = [self.freq(a, True) for a in range(3)]
        kd = [self.freq(a, False) for a in range(3)]
        kk = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
        kd2 = kd[0] ** 2 + kd[1] ** 2 + kd[2] ** 2
        kv = kd[0] * F[0] + kd[1] * F[1] + kd[2] * F[2]
        if inverse:
            bk = torch.where(kk == 0, 1.0, BETA * kk)  # identity on the zero wavenumber
            diag, coup = 1.0 / bk, -GAMMA / bk / (bk + GAMMA * kd2)
        else:
            diag, coup = BETA * kk, GAMMA
        return torch.stack([torch.fft.ifftn(diag * F[c] + coup * kd[c] * kv).real for c in range(3)])

    def weight(self, j):
        return self.dt * (0.5 if j in (0, self.nt) else 1.0)

    def states(self, m0, xm):
        m = [m0]
        for _ in range(self.nt):
            m.append(self.interp(m[-1], xm))
        return m

    def factor(self, v, xp):
        div = sum(self.deriv(v[a], a) for a in range(3))
        dx = self.interp(div, xp)
        return 1 + 0.5 * self.dt * (dx + div) + 0.5 * self.dt ** 2 * div * dx

    def adjoint(self, lam, c, xp, grads):
        """body force of the adjoint that ends in lam; grads(j) is grad m^j"""
        b = self.weight(self.nt) * lam * grads(self.nt)
        for j in range(self.nt - 1, -1, -1):
            lam = c * self.interp(lam, xp)
            b = b + self.weight(j) * lam * grads(j)
        return b


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch"):
        return None  # a whole Gauss-Newton solve in 64 bits takes too long
    ex = _Exact(case, _shape(case))
    x = {k: t.detach().double() for k, t in _inputs(case, seed).items()}
    if kind == "precond":
        return ex.regular(x["r"], True)
    v, m0, m1 = x["v"], x["m0"], x["m1"]
    m = ex.states(m0, ex.foot(v, -1.0))
    mis = 0.5 * ex.h3 * float((m[-1] - m1).square().sum())
    if kind == "forward":
        return [m[-1], mis]
    xp = ex.foot(v, 1.0)
    c = ex.factor(v, xp)
    if kind == "autograd":
        loss = mis + 5.0 * float(m[-1].square().mean())
        upstream = 10.0 * m[-1] / m[-1].numel()
        b = ex.adjoint(m1 - m[-1] - upstream / ex.h3, c, xp, lambda j: ex.grad(m[j]))
        return [loss, m[-1], ex.h3 * b]
    if kind == "gradient":
        Av = ex.regular(v, False)
        J = mis + 0.5 * ex.h3 * float((v * Av).sum())
        return [Av + ex.adjoint(m1 - m[-1], c, xp, lambda j: ex.grad(m[j])), J]
    vt, xm, dt = x["vt"], ex.foot(v, -1.0), ex.dt
    grads = [ex.grad(f) for f in m]
    src = [-(vt * g).sum(0) for g in grads]
    u = 0.5 * dt * src[0]
    for j in range(ex.nt):
        u = ex.interp(u, xm) + dt * src[j + 1]
    mt = u - 0.5 * dt * src[-1]
    return ex.regular(vt, False) + ex.adjoint(-mt, c, xp, lambda j: grads[j])
