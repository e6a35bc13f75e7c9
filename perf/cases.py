"""Timed cases of the imaging library: what a program that images with it calls.

The calls are the measurement operator Phi, its adjoint and the normal
operator, the SARA dictionary in both directions, the SDMM and primal-dual
solvers, and the learned warm start's network forward and backward. Sizes are
those of the package's workloads (64 x 64 in double precision, 256 x 256 with
8 blocks, 512 x 512 channels, 1024 x 1024 with 64 blocks, the 256 x 256
warm-start network) and rectangular or odd ones between them; draw() spreads
over the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_1502_05037_gb300 as pk
from paper_1502_05037_gb300 import problem, synth

IMAGING = dict(L=4, R=1, dtype="f32", uniform=0.0, snr=30.0, mask=0x1FF, iters=0)
CG_ITERS = 8
GAMMA = 3e-4          # SDMM step for skies of peak 1: about 1e-3 of the largest coefficient
UV_SIGMA = math.pi / 4


def _imaging(name, op, nx, ny, M, J, **kw):
    return dict(IMAGING, name=name, op=op, nx=nx, ny=ny, M=M, J=J, **kw)


def listed():
    return [
        # the smallest call: predicting a snapshot's visibilities from a 64 x 64 image
        _imaging("phi_64", "phi", 64, 64, 8192, 4, L=3),
        # the largest prediction: ten million visibilities of a 1024 x 1024 image
        _imaging("phi_1024", "phi", 1024, 1024, 10_485_760, 6, L=5, R=64, uniform=0.1, snr=20.0),
        # one spectral channel's dirty image, an odd number of visibilities
        _imaging("phi_adj_512", "phi_adj", 512, 512, 917_503, 6, R=7),
        # the normal operator of a solver of the caller's own, rectangular field, odd kernel
        _imaging("normal_256x512", "normal", 512, 256, 655_361, 5, R=8),
        # analysis coefficients of a 1024 x 1024 image in all nine bases (reweighting, objectives)
        _imaging("psi_adj_1024", "psi_adj", 1024, 1024, 4096, 6, L=5),
        # synthesis from the coefficients of a rectangular image
        _imaging("psi_512x1024", "psi", 1024, 512, 4096, 6, L=4),
        # double precision: the small problem solved to check a pipeline
        _imaging("sdmm_64_f64", "sdmm", 64, 64, 8192, 4, L=3, dtype="f64", iters=2),
        # SDMM on the 256 x 256 workload, a few iterations of a solve
        _imaging("sdmm_256", "sdmm", 256, 256, 655_360, 6, R=8, iters=4),
        # SDMM on the 1024 x 1024 workload with 64 blocks
        _imaging("sdmm_1024", "sdmm", 1024, 1024, 10_485_760, 6, L=5, R=64, uniform=0.1, snr=20.0, iters=2),
        # a reweighted pass of the primal-dual solver on a 512 x 512 channel
        _imaging("pd_512", "pd", 512, 512, 786_433, 6, R=9, iters=10),
        # training the warm-start network: a mini-batch's loss and gradients
        dict(name="unet_grad_256", op="unet_grad", nx=256, ny=256, levels=4, base=32, batch=8),
        # the warm start of one solve: the network's prediction from one dirty image
        dict(name="unet_forward_256", op="unet_forward", nx=256, ny=256, levels=4, base=32, batch=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["phi", "phi", "phi_adj", "phi_adj", "normal", "psi_adj", "psi", "sdmm", "sdmm", "pd",
                     "unet_grad", "unet_forward"])
    if op.startswith("unet"):
        levels = rng.choice([3, 4])
        step = 1 << (levels - 1)
        return dict(op=op, nx=step * rng.randint(64 // step, 256 // step), ny=step * rng.randint(64 // step, 256 // step),
                    levels=levels, base=rng.choice([16, 24, 32]), batch=rng.randint(1, 8) if op == "unet_grad" else rng.randint(1, 4))
    double = rng.random() < 0.25
    nx = 2 ** rng.randint(5, 8 if double else 10)
    ny = max(32, min(1024, int(nx * rng.choice([0.5, 1, 1, 1, 2]))))
    if double:
        ny = min(ny, 256)
    N = nx * ny
    M = _log_int(rng, N // 2, 10 * N) | 1
    if double:
        M = min(M, 262_145)
    if op in ("sdmm", "pd"):
        M = min(M, 2_621_441)
    if op in ("psi", "psi_adj"):
        M = 4096
    return dict(IMAGING, op=op, nx=nx, ny=ny, M=M, J=rng.choice([4, 5, 6, 6, 6, 7, 8]), L=rng.randint(2, 5),
                R=_log_int(rng, 1, 64), dtype="f64" if double else "f32", uniform=rng.choice([0.0, 0.1]),
                snr=rng.choice([20.0, 30.0]), mask=rng.choice([0x1FF, 0x1FF, 0x1FF, 0x01F, 0x1FE]),
                iters=rng.randint(2, 4) if op == "sdmm" else rng.randint(5, 10) if op == "pd" else 0)


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _generator(seed, role):
    g = torch.Generator(device=_device())
    g.manual_seed(100_003 * (int(seed) + 1) + role)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device=_device(), generator=g)


def _randn(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device=_device(), generator=g)


def _real(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _cplx(case):
    return torch.complex64 if case["dtype"] == "f32" else torch.complex128


def _coverage(case, seed):
    """(u, v) on [-pi, pi): Gaussian about the centre, a fraction of it uniform."""
    g = _generator(seed, 1)
    out = []
    uniform = _rand(g, case["M"]) < case["uniform"]
    for _ in range(2):
        gauss, flat = UV_SIGMA * _randn(g, case["M"]), math.pi * (2 * _rand(g, case["M"]) - 1)
        c = torch.where(uniform | (gauss.abs() >= 3.14159), flat, gauss)
        out.append(c.clamp(-3.14159, 3.14159).to(_real(case)))
    return out


def _sky(nx, ny, seed, role=2):
    """Point sources and Gaussian blobs on a zero background, peak 1."""
    g = _generator(seed, role)
    dev = _device()
    img = torch.zeros(ny, nx, dtype=torch.float64, device=dev)
    n = max(20, nx * ny // 2048)
    py, px = (0.1 + 0.8 * _rand(g, n)) * ny, (0.1 + 0.8 * _rand(g, n)) * nx
    img.view(-1).index_put_((py.long() * nx + px.long(),), -torch.log(1 - _rand(g, n)), accumulate=True)
    iy, ix = torch.arange(ny, device=dev, dtype=torch.float64), torch.arange(nx, device=dev, dtype=torch.float64)
    k = 12
    cy, cx = _rand(g, k) * ny, _rand(g, k) * nx
    s, a = (1 + 2 * _rand(g, k)) * max(nx, ny) / 64, 0.2 + 0.8 * _rand(g, k)
    ey = torch.exp(-(iy[None] - cy[:, None]) ** 2 / (2 * s[:, None] ** 2))
    ex = torch.exp(-(ix[None] - cx[:, None]) ** 2 / (2 * s[:, None] ** 2))
    img += torch.einsum("k,ki,kj->ij", a, ey, ex)
    return img / img.max()


def _offsets(case):
    R = min(case["R"], case["M"])
    return synth.block_offsets(synth.block_sizes(case["M"], R, 4000 + R))


def _nu(case):
    """||Phi|| of a dense Gaussian coverage (its peak density), which a program knows in advance."""
    return math.sqrt(case["M"] * 2 * math.pi / UV_SIGMA ** 2)


def _imaging_inputs(case, seed):
    """Everything but the plan, from the seed alone."""
    rt, ct = _real(case), _cplx(case)
    d = {"op": case["op"], "M": case["M"], "iters": case["iters"]}
    d["u"], d["v"] = _coverage(case, seed)
    sky = _sky(case["nx"], case["ny"], seed)
    op = case["op"]
    g = _generator(seed, 3)
    if op in ("phi", "normal", "psi_adj"):
        d["x"] = sky.to(rt)
    elif op == "psi":
        d["c"] = _psi_adj64(sky + 0.01 * _randn(g, case["ny"], case["nx"]), case["L"], case["mask"]).to(rt)
    else:
        # data: the sky's visibilities plus noise at the case's signal-to-noise ratio
        y0 = _Nufft64(case, d["u"], d["v"]).phi(sky)
        sigma = problem.noise_sigma_from_norm(float(torch.linalg.vector_norm(y0)), case["M"], case["snr"])
        noise = torch.view_as_complex(_randn(g, case["M"], 2)) * (sigma / math.sqrt(2))
        d["y"] = (y0 + noise).to(ct)
        d["offsets"] = _offsets(case)
        d["eps"] = problem.chi2_epsilon(sigma, np.diff(d["offsets"]))
        d["nu"] = _nu(case)
        # solves start from a blurred image; the reweighted pass has weights
        d["x0"] = _blur(sky, 1.5).to(rt)
        if op == "pd":
            c = _psi_adj64(sky, case["L"], case["mask"])
            rho = c.std()
            d["w"] = (rho / (rho + c.abs())).to(rt)
    return d


def _blur(img, width):
    """Periodic Gaussian blur over the last two axes."""
    ny, nx = img.shape[-2:]
    fy = torch.fft.fftfreq(ny, device=img.device, dtype=torch.float64)[:, None]
    fx = torch.fft.fftfreq(nx, device=img.device, dtype=torch.float64)[None]
    return torch.fft.ifft2(torch.fft.fft2(img) * torch.exp(-2 * (math.pi * width) ** 2 * (fy * fy + fx * fx))).real


def _unet_shapes(levels, base):
    """(Cout, k, Cin) of the network's convolutions in the parameter vector's order."""
    shapes, cin = [], 1
    for l in range(levels - 1):
        c = base << l
        shapes += [(c, 3, cin), (c, 3, c)]
        cin = c
    cb = base << (levels - 1)
    shapes += [(cb, 3, cin), (cb, 3, cb)]
    for l in range(levels - 2, -1, -1):
        c = base << l
        shapes += [(c, 3, 2 * c), (c, 3, 2 * c), (c, 3, c)]
    return shapes + [(1, 1, base)]


def _unet_inputs(case, seed):
    g = _generator(seed, 4)
    p = []
    for co, k, ci in _unet_shapes(case["levels"], case["base"]):
        p += [_randn(g, co * k * k * ci) * math.sqrt(2.0 / (k * k * ci)), 0.01 * _randn(g, co)]
    target = torch.stack([_sky(case["nx"], case["ny"], seed, 10 + b) for b in range(case["batch"])])
    x = _blur(target, 2.0) + 0.01 * _randn(g, *target.shape)
    return {"op": case["op"], "params": torch.cat(p).float(), "x": x.float().contiguous(), "target": target.float().contiguous()}


def prepare(case, seed):
    if case["op"].startswith("unet"):
        d = _unet_inputs(case, seed)
        d["net"] = pk.Unet(case["ny"], case["nx"], levels=case["levels"], base=case["base"], max_batch=case["batch"])
        d["net"].set_params(d["params"])
        d["out"] = torch.empty_like(d["params"] if case["op"] == "unet_grad" else d["x"])
        return d
    d = _imaging_inputs(case, seed)
    d["plan"] = pk.Plan(case["nx"], case["ny"], d["u"], d["v"], kb_width=case["J"], levels=case["L"],
                        block_offsets=_offsets(case), basis_mask=case["mask"],
                        dtype=pk.PURIFY_F32 if case["dtype"] == "f32" else pk.PURIFY_F64)
    shape = {"phi": (case["M"],), "psi_adj": (bin(case["mask"]).count("1"), case["ny"], case["nx"])}
    d["out"] = torch.empty(shape.get(case["op"], (case["ny"], case["nx"])), device=_device(),
                           dtype=_cplx(case) if case["op"] in ("phi", "phi_adj") else _real(case))
    return d


def run(state):
    op, out = state["op"], state["out"]
    if op == "phi":
        pk.purify_phi(state["plan"], state["x"], out)
    elif op == "phi_adj":
        pk.purify_phi_adj(state["plan"], state["y"], out)
    elif op == "normal":
        pk.purify_phi_normal(state["plan"], state["x"], out)
    elif op == "psi":
        pk.purify_psi(state["plan"], state["c"], out)
    elif op == "psi_adj":
        pk.purify_psi_adj(state["plan"], state["x"], out)
    elif op == "sdmm":
        out.copy_(state["x0"])
        st = pk.purify_sdmm_solve(state["plan"], state["y"], state["eps"], out, max_iter=state["iters"],
                                  cg_iters=CG_ITERS, gamma=GAMMA, nu=state["nu"])
        return {"x": out, "objective": st.objective, "residual": st.max_resid_over_eps}
    elif op == "pd":
        out.copy_(state["x0"])
        st = pk.purify_pd_solve(state["plan"], state["y"], state["eps"], out, w=state["w"], iters=state["iters"],
                                nu=state["nu"])
        return {"x": out, "objective": st.objective, "residual": st.max_resid_over_eps}
    elif op == "unet_forward":
        state["net"].forward(state["x"], out)
    else:
        loss = state["net"].gradients(state["x"], state["target"], out)
        return {"loss": loss, "grads": out}
    return out


# -------------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once; the multiply-adds of the
    transforms, the interpolation (2 J^2 complex terms per visibility) and the
    filters."""
    if case["op"].startswith("unet"):
        shapes = _unet_shapes(case["levels"], case["base"])
        pix, macs, L = case["batch"] * case["nx"] * case["ny"], 0.0, case["levels"]
        level = [l for l in range(L - 1) for _ in range(2)] + [L - 1] * 2 + [l for l in range(L - 2, -1, -1) for _ in range(3)] + [0]
        for (co, k, ci), l in zip(shapes, level):
            macs += co * k * k * ci * pix / 4 ** l
        params = sum(co * k * k * ci + co for co, k, ci in shapes)
        if case["op"] == "unet_forward":
            return {"bytes": 4.0 * (2 * pix + params), "flops": 2 * macs}
        return {"bytes": 4.0 * (2 * pix + 2 * params), "flops": 6 * macs}
    rb = 4 if case["dtype"] == "f32" else 8
    N, M, J, op, n = case["nx"] * case["ny"], case["M"], case["J"], case["op"], max(1, case["iters"])
    q = bin(case["mask"]).count("1")
    fft = 5.0 * 4 * N * math.log2(4 * N) * 0.75          # half of the row transforms are of zero rows
    one = fft + M * (4.0 * J * J + 40 * J)                # one of Phi, Phi^H
    wavelet = sum(2.0 * N * 2 * 2 * 2 * p * 4 / 3 for p in range(1, 9) if case["mask"] >> p & 1)
    if op in ("phi", "phi_adj"):
        return {"bytes": rb * (N * (1.0 if op == "phi" else 2.0) + 4.0 * M), "flops": one}
    if op == "normal":
        return {"bytes": rb * (2.0 * N + 2.0 * M), "flops": 2 * one}
    if op in ("psi", "psi_adj"):
        return {"bytes": rb * (1.0 + q) * N, "flops": wavelet}
    if op == "sdmm":
        return {"bytes": rb * (2.0 * N + 4.0 * M), "flops": n * (2 * one * (1 + CG_ITERS) + 2 * wavelet + 20 * M)}
    return {"bytes": rb * ((2.0 + q) * N + 4.0 * M), "flops": n * (2 * one + 2 * wavelet + 20 * M)}


# ------------------------------------------------- the same in 64 bits
class _Nufft64:
    """Phi = G F Z S with the Kaiser-Bessel kernel, in double precision."""

    def __init__(self, case, u, v):
        J = self.J = case["J"]
        self.nx, self.ny, self.beta = case["nx"], case["ny"], 2.34 * case["J"]
        self.Kx, self.Ky = 2 * self.nx, 2 * self.ny
        self.dev = u.device
        self.ax = self._taps(u.double(), self.Kx)
        self.ay = self._taps(v.double(), self.Ky)
        self.s = self._correction(self.ny, self.Ky)[:, None] * self._correction(self.nx, self.Kx)[None]
        n1, n2 = torch.arange(self.nx, device=self.dev) - self.nx // 2, torch.arange(self.ny, device=self.dev) - self.ny // 2
        self.at = ((n2 % self.Ky)[:, None] * self.Kx + (n1 % self.Kx)[None]).reshape(-1)
        assert J >= 2

    def _taps(self, coord, K):
        kappa = coord * (K / (2 * math.pi))
        k0 = torch.floor(kappa - self.J / 2) + 1
        i0b = torch.special.i0(torch.tensor(self.beta, dtype=torch.float64, device=self.dev))
        taps = []
        for a in range(self.J):
            t = kappa - (k0 + a)
            r = (1 - (2 * t / self.J) ** 2).clamp_min(0)
            taps.append(((k0 + a).long() % K, torch.special.i0(self.beta * r.sqrt()) / i0b))
        return taps

    def _correction(self, n, K):
        nu = torch.arange(n, dtype=torch.float64, device=self.dev) - n // 2
        a = self.beta ** 2 - (math.pi * self.J * nu / K) ** 2
        z = a.abs().sqrt().clamp_min(1e-300)
        return 1 / (self.J / torch.special.i0(torch.tensor(self.beta, dtype=torch.float64, device=self.dev)) * torch.where(a > 0, torch.sinh(z), torch.sin(z)) / z)

    def phi(self, x):
        grid = torch.zeros(self.Ky * self.Kx, dtype=torch.complex128, device=self.dev)
        grid[self.at] = (self.s * x.double()).reshape(-1).to(torch.complex128)
        grid = torch.fft.fft2(grid.view(self.Ky, self.Kx)).reshape(-1)
        y = torch.zeros(self.ax[0][0].numel(), dtype=torch.complex128, device=self.dev)
        for ky, wy in self.ay:
            row = torch.zeros_like(y)
            for kx, wx in self.ax:
                row += wx * grid[ky * self.Kx + kx]
            y += wy * row
        return y

    def phi_adj(self, y):
        grid = torch.zeros(self.Ky * self.Kx, 2, dtype=torch.float64, device=self.dev)
        for ky, wy in self.ay:
            row = wy * y
            for kx, wx in self.ax:
                grid.index_add_(0, ky * self.Kx + kx, torch.view_as_real(wx * row))
        img = torch.fft.ifft2(torch.view_as_complex(grid).view(self.Ky, self.Kx), norm="forward")
        return self.s * img.reshape(-1)[self.at].view(self.ny, self.nx)


def _daubechies(p):
    """Minimum-phase Daubechies low-pass filter of p vanishing moments."""
    zeros = [-1.0] * p
    if p > 1:
        c = np.array([math.comb(p - 1 + k, k) for k in range(p)][::-1], dtype=np.longdouble)
        for y in np.roots(c.astype(np.float64)):
            y = np.clongdouble(y)
            for _ in range(4):
                y = y - np.polyval(c, y) / np.polyval(np.polyder(c), y)
            b = 1 - 2 * y
            z = b + np.sqrt(b * b - 1)
            zeros.append(z if abs(z) < 1 else 1 / z)
    h = np.array([1], dtype=np.clongdouble)
    for z in zeros:
        h = np.convolve(h, np.array([1, -z], dtype=np.clongdouble))
    h = h.real
    return (h * (np.sqrt(np.longdouble(2)) / h.sum())).astype(np.float64)


def _bases(mask):
    return [p for p in range(9) if mask >> p & 1]


def _level(n, p, dev):
    """One periodic analysis level of db_p on length n: [n][n], low-pass rows first."""
    h = _daubechies(p)
    g = (-1.0) ** np.arange(2 * p) * h[::-1]
    A = np.zeros((n, n))
    k = np.arange(n // 2)
    for i in range(2 * p):
        np.add.at(A, (k, (2 * k + i) % n), h[i])
        np.add.at(A, (n // 2 + k, (2 * k + i) % n), g[i])
    return torch.from_numpy(A).to(dev)


def _psi_adj64(x, levels, mask):
    out, q = [], len(_bases(mask))
    for p in _bases(mask):
        c = x.double().clone()
        for l in range(levels if p else 0):
            ny, nx = x.shape[0] >> l, x.shape[1] >> l
            c[:ny, :nx] = _level(ny, p, x.device) @ c[:ny, :nx] @ _level(nx, p, x.device).T
        out.append(c)
    return torch.stack(out) / math.sqrt(q)


def _psi64(c, levels, mask):
    x = torch.zeros(c.shape[1:], dtype=torch.float64, device=c.device)
    for i, p in enumerate(_bases(mask)):
        b = c[i].double().clone()
        for l in reversed(range(levels if p else 0)):
            ny, nx = c.shape[1] >> l, c.shape[2] >> l
            b[:ny, :nx] = _level(ny, p, c.device).T @ b[:ny, :nx] @ _level(nx, p, c.device)
        x += b
    return x / math.sqrt(c.shape[0])


class _Solve64:
    """Problem (3): the pieces both solvers share."""

    def __init__(self, case, d):
        self.A, self.L, self.mask, self.nu = _Nufft64(case, d["u"], d["v"]), case["L"], case["mask"], d["nu"]
        off = torch.from_numpy(d["offsets"]).to(_device())
        self.block = torch.repeat_interleave(torch.arange(len(off) - 1, device=off.device), off[1:] - off[:-1])
        self.y = d["y"].to(torch.complex128) / self.nu
        self.eps = torch.from_numpy(d["eps"]).to(_device()) / self.nu

    def phi(self, x):
        return self.A.phi(x) / self.nu

    def adj(self, y):
        return self.A.phi_adj(y).real / self.nu

    def norms(self, r):
        return torch.zeros_like(self.eps).index_add_(0, self.block, r.real ** 2 + r.imag ** 2).sqrt()

    def ball(self, v):
        r = v - self.y
        n = self.norms(r)
        return self.y + r * torch.where(n > self.eps, self.eps / n, torch.ones_like(n))[self.block]

    def answer(self, x, w):
        objective = (w * _psi_adj64(x, self.L, self.mask)).abs().sum()
        return {"x": x, "objective": float(objective), "residual": float((self.norms(self.phi(x) - self.y) / self.eps).max())}


def _sdmm64(case, d):
    S, x = _Solve64(case, d), d["x0"].double()
    z1, z2, z3 = 0.0, 0.0, 0.0
    for _ in range(case["iters"]):
        v1, v2 = _psi_adj64(x, S.L, S.mask), S.phi(x)
        t = v1 + z1
        s1, s2, s3 = t.sign() * (t.abs() - GAMMA).clamp_min(0), S.ball(v2 + z2), (x + z3).clamp_min(0)
        z1, z2, z3 = t - s1, z2 + v2 - s2, z3 + x - s3
        r = _psi64(s1 - z1, S.L, S.mask) + S.adj(s2 - z2 - v2) + s3 - z3 - 2 * x
        p, rs = r.clone(), (r * r).sum()
        for _ in range(CG_ITERS):
            Ap = 2 * p + S.adj(S.phi(p))
            a = rs / (p * Ap).sum()
            x, r = x + a * p, r - a * Ap
            rs, old = (r * r).sum(), rs
            p = r + (rs / old) * p
    return S.answer(x, 1.0)


def _pd64(case, d, tau=0.05, sigma=9.8):
    S, x, w = _Solve64(case, d), d["x0"].double(), d["w"].double()
    bar, p1, p2 = x, 0.0, 0.0
    for _ in range(case["iters"]):
        p1 = torch.maximum(torch.minimum(p1 + sigma * _psi_adj64(bar, S.L, S.mask), w), -w)
        t = p2 + sigma * S.phi(bar)
        p2 = t - sigma * S.ball(t / sigma)
        new = (x - tau * (_psi64(p1, S.L, S.mask) + S.adj(p2))).clamp_min(0)
        bar, x = 2 * new - x, new
    return S.answer(x, w)


def _unet64(case, d):
    flat = d["params"].double().requires_grad_(case["op"] == "unet_grad")
    layers, at = [], 0
    for co, k, ci in _unet_shapes(case["levels"], case["base"]):
        n = co * k * k * ci
        layers.append((flat[at:at + n].view(co, k, k, ci).permute(0, 3, 1, 2), flat[at + n:at + n + co]))
        at += n + co
    todo = iter(layers)

    def conv(t):
        w, b = next(todo)
        return F.relu(F.conv2d(t, w, b, padding=1))

    x = d["x"].double()[:, None]
    t, skips = x, []
    for _ in range(case["levels"] - 1):
        t = conv(conv(t))
        skips.append(t)
        t = F.max_pool2d(t, 2)
    t = conv(conv(t))
    for s in reversed(skips):
        t = conv(conv(torch.cat([s, conv(F.interpolate(t, scale_factor=2, mode="nearest"))], 1)))
    w, b = next(todo)
    out = (x + F.conv2d(t, w, b))[:, 0]
    if case["op"] == "unet_forward":
        return out
    loss = ((out - d["target"].double()) ** 2).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grads": flat.grad}


def exact(case, seed):
    if case["op"].startswith("unet"):
        return _unet64(case, _unet_inputs(case, seed))
    d = _imaging_inputs(case, seed)
    op = case["op"]
    if op == "sdmm":
        return _sdmm64(case, d)
    if op == "pd":
        return _pd64(case, d)
    if op == "psi":
        return _psi64(d["c"], case["L"], case["mask"])
    if op == "psi_adj":
        return _psi_adj64(d["x"], case["L"], case["mask"])
    A = _Nufft64(case, d["u"], d["v"])
    if op == "phi":
        return A.phi(d["x"])
    if op == "phi_adj":
        return A.phi_adj(d["y"].to(torch.complex128))
    return A.phi_adj(A.phi(d["x"])).real
