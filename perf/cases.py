"""The work this framework is used for, as cases of one pass each: the acoustic operators A, A^T and
C of compressed-sensing photoacoustic tomography over small, ordinary and large grids, their autograd
pair, the TV proximal operator, a TV-Bregman reconstruction, and the learned warm start's network.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU and the handle a user's program keeps
    run(state)           one pass through the public entry points, and its outputs
    work(case)           bytes and operations one pass cannot do without
    exact(case, seed)    the outputs in 64 bits, restated with plain torch

Grids, sampling ratios, step counts and schedules are those of the named workloads (presets.py), the
tests and bench.py, or lie between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1605_00133_gb300 import _lib, autograd, unet
from paper_1605_00133_gb300.operators import PatOperator
from paper_1605_00133_gb300.presets import (KIND_FULL, KIND_RSP, KIND_SHD01, KIND_SHDPM, Grid,
                                            Sampling)

KINDS = {"full": KIND_FULL, "rsp": KIND_RSP, "shd01": KIND_SHD01, "shdpm": KIND_SHDPM}
DX, C0, CFL = 100e-6, 1500.0, 0.3


def _op(name, op, grid, T, kind, m, batch=1, **extra):
    return {"name": name, "op": op, "nz": grid[0], "ny": grid[1], "nx": grid[2], "T": T, "kind": kind,
            "m": m, "batch": batch, **extra}


def listed():
    return [
        # one forward projection of a small test volume: quick experiments, dense sweeps of phantoms
        _op("forward_32", "forward", (32, 32, 32), 64, "rsp", 256),
        # simulating the data of the ordinary 64x128x128 scan: 12.5 % random single points
        _op("forward_128", "forward", (64, 128, 128), 400, "rsp", 2048),
        # back-projection of such a scan, the first image a user looks at
        _op("adjoint_128", "adjoint", (64, 128, 128), 400, "rsp", 2048),
        # the gradient of the data misfit of a scan with scrambled-Hadamard 0/1 patterns through
        # autograd: one forward, one adjoint, as an iterative or learned reconstruction calls it
        _op("gradient_patterns_128", "gradient", (64, 128, 128), 400, "shd01", 2048),
        # conventional full scan of three volumes at once on a slab-shaped grid, an odd number of steps
        _op("forward_batch_slab", "forward", (32, 256, 64), 75, "full", 0, batch=3),
        # the misfit gradient on the large 128x256x256 grid, 1/16 of the points; a part of its 800 steps
        _op("gradient_256", "gradient", (128, 256, 256), 200, "rsp", 4096),
        # the pattern operator C and its transpose alone, on a recorded series of 400 planes
        _op("patterns_128", "sample", (16, 128, 128), 400, "shd01", 2048),
        # positivity-constrained TV denoising: the proximal step of a reconstruction (50 iterations)
        {"name": "prox_128", "op": "prox", "nz": 64, "ny": 128, "nx": 128, "alpha": 0.02, "iters": 50, "batch": 1},
        # the same on the large grid, whose fields do not fit the L2
        {"name": "prox_256", "op": "prox", "nz": 128, "ny": 256, "nx": 256, "alpha": 0.02, "iters": 20, "batch": 1},
        # a short TV-Bregman reconstruction of the small volume (latency: many short kernels and
        # reductions the host decides on)
        _op("solve_32", "solve", (32, 32, 32), 64, "rsp", 256, lam=2e-4, outer=2, inner=5, prox_iters=40),
        # one decoder layer of the warm-start network on an odd volume: convolution with ReLU, its data
        # gradient and its weight gradient
        {"name": "conv_48_16_odd", "op": "conv", "cin": 48, "cout": 16, "D": 33, "H": 70, "W": 101},
        # one training pass of the warm-start network on the ordinary volume: output, loss, gradients
        {"name": "network_128", "op": "network", "D": 64, "H": 128, "W": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forward", "adjoint", "gradient", "forward", "adjoint", "gradient", "sample", "prox",
                     "solve", "conv", "network"])
    if op in ("forward", "adjoint", "gradient"):
        while True:
            nz, ny, nx = (2 ** rng.randint(4, 7) for _ in range(3))
            if rng.random() < 0.3:
                ny = nx = 256
            T = _log_int(rng, 24, 800)
            batch = rng.choice([1, 1, 1, 2, 3, 4])
            if nz * ny * nx * T * batch * (2 if op == "gradient" else 1) <= 128 * 256 * 256 * 400:
                break
        kind = rng.choice(["full", "rsp", "rsp", "shd01", "shdpm"])
        if ny * nx > 32768 and kind.startswith("shd"):
            kind = "rsp"
        m = 0 if kind == "full" else max(1, int(ny * nx * rng.uniform(1 / 16, 1 / 3)))
        return _op("", op, (nz, ny, nx), T, kind, m, batch)
    if op == "sample":
        ny, nx = (2 ** rng.randint(4, 7) for _ in range(2))
        kind = rng.choice(["rsp", "shd01", "shdpm"])
        m = max(1, int(ny * nx * rng.uniform(1 / 16, 1 / 3)))
        return _op("", op, (16, ny, nx), _log_int(rng, 16, 800), kind, m, rng.choice([1, 2]))
    if op == "prox":
        nz, ny, nx = (2 ** rng.randint(4, 7) for _ in range(3))
        return {"name": "", "op": op, "nz": nz, "ny": ny, "nx": nx, "alpha": math.exp(rng.uniform(-6, -2)),
                "iters": _log_int(rng, 10, 100), "batch": rng.choice([1, 1, 2])}
    if op == "solve":
        nz, ny, nx = (2 ** rng.randint(4, 6) for _ in range(3))
        return _op("", op, (nz, ny, nx), rng.randint(40, 96), "rsp", max(1, int(ny * nx * rng.uniform(1 / 8, 1 / 4))),
                   lam=2e-4, outer=rng.randint(1, 2), inner=rng.randint(3, 6), prox_iters=rng.randint(20, 50))
    if op == "conv":
        cin, cout = rng.choice([(16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (192, 64),
                                (96, 32), (48, 16)])
        D, H, W = (_log_int(rng, 9, 100) for _ in range(3))
        return {"name": "", "op": op, "cin": cin, "cout": cout, "D": D, "H": H, "W": W}
    D, H, W = (8 * rng.randint(2, n) for n in (8, 16, 16))
    return {"name": "", "op": op, "D": D, "H": H, "W": W}


# ------------------------------------------------------------------------------------ inputs

def _dev():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


def _pml(shape):
    return min(10, min(shape) // 2 - 2)


def _grid(c):
    shape = (c["nz"], c["ny"], c["nx"])
    return Grid(*shape, dx=DX, c=C0, cfl=CFL, T=c.get("T", 1), pml_size=_pml(shape), batch=c["batch"])


def _sampling(c, seed):
    g = torch.Generator().manual_seed(seed + 1)
    M, m, kind = c["ny"] * c["nx"], c.get("m", 0), KINDS[c.get("kind", "full")]
    if kind == KIND_FULL:
        return Sampling(kind, M)
    if kind == KIND_RSP:
        idx = torch.randperm(M, generator=g)[:m].sort().values
        return Sampling(kind, m, indices=idx.numpy().astype(np.int32))
    perm, rows = torch.randperm(M, generator=g), torch.randperm(M, generator=g)[:m]
    return Sampling(kind, m, perm=perm.numpy().astype(np.int32), rows=rows.numpy().astype(np.int32))


def _vessels(c, seed):
    """Initial pressure [B][nz][ny][nx] in [0, 1]: straight vessel pieces of radius 1 to 4 voxels with
    soft walls, zero in the absorbing layer (float32)."""
    dev, shape, P = _dev(), (c["nz"], c["ny"], c["nx"]), _pml((c["nz"], c["ny"], c["nx"]))
    z, y, x = (torch.arange(n, device=dev, dtype=torch.float32) for n in shape)
    z, y, x = z[:, None, None], y[None, :, None], x[None, None, :]
    out = torch.zeros((c["batch"],) + shape, device=dev)
    for b in range(c["batch"]):
        rng = np.random.default_rng(1000 * seed + b)
        for _ in range(24):
            lo, hi = np.full(3, P + 1.0), np.array(shape) - P - 2.0
            a = lo + rng.random(3) * (hi - lo)
            d = rng.standard_normal(3)
            d *= rng.uniform(8, 40) / np.linalg.norm(d)
            r, v = rng.uniform(1, 4), rng.uniform(0.1, 1)
            t = ((z - a[0]) * d[0] + (y - a[1]) * d[1] + (x - a[2]) * d[2]) / float(d @ d)
            t = t.clamp_(0, 1)
            dist2 = (z - a[0] - t * d[0]) ** 2 + (y - a[1] - t * d[1]) ** 2 + (x - a[2] - t * d[2]) ** 2
            torch.maximum(out[b], v * torch.sigmoid(2.0 * (r - dist2.sqrt())), out=out[b])
    mask = torch.zeros(shape, device=dev)
    mask[P:shape[0] - P, P:shape[1] - P, P:shape[2] - P] = 1
    return out * mask


def _plane_data(c, seed):
    """Plane pressure series [B][T][ny*nx]: the spherical waves of a dozen Gaussian balls below the
    detection plane, p = a (r - ct) / (2 r) exp(-(r - ct)^2 / (2 s^2)), plus 1 % noise (float32)."""
    dev, g = _dev(), _grid(c)
    y, x = torch.meshgrid(torch.arange(g.ny, device=dev, dtype=torch.float64),
                          torch.arange(g.nx, device=dev, dtype=torch.float64), indexing="ij")
    t = CFL * torch.arange(g.T, device=dev, dtype=torch.float64)[:, None]  # in voxels
    gen = torch.Generator(device=dev).manual_seed(seed + 7)
    out = torch.empty((g.batch, g.T, g.m_plane), device=dev)
    for b in range(g.batch):
        rng = np.random.default_rng(1000 * seed + 500 + b)
        p = torch.zeros((g.T, g.m_plane), device=dev, dtype=torch.float64)
        for _ in range(12):
            cz = rng.uniform(3, max(4, g.nz - 2 * g.pml_size - 2))
            cy, cx = rng.uniform(g.pml_size, g.ny - g.pml_size), rng.uniform(g.pml_size, g.nx - g.pml_size)
            r = ((y - cy) ** 2 + (x - cx) ** 2 + cz ** 2).sqrt().reshape(1, -1)
            s, a = rng.uniform(1.5, 3), rng.uniform(0.2, 1)
            p += a * (r - t) / (2 * r) * torch.exp(-(r - t) ** 2 / (2 * s * s))
        noise = torch.randn(p.shape, generator=gen, device=dev, dtype=torch.float64)
        out[b] = (p + 0.01 * p.abs().max() * noise).float()
    return out


def _data(c, seed):
    """Measured data [B][T][m] of that series (float32)."""
    f = _sample64(_plane_data(c, seed).double(), c, _sampling(c, seed))
    return f.float().contiguous()


def _bf16(shape, seed, scale):
    g = torch.Generator(device=_dev()).manual_seed(seed)
    return (torch.randn(shape, generator=g, device=_dev()) * scale).bfloat16()


def _conv_inputs(c, seed):
    V, cin, cout = c["D"] * c["H"] * c["W"], c["cin"], c["cout"]
    x = _bf16((V, cin), 3 * seed, 1.0).relu()  # activations behind a ReLU
    w = _bf16((27, cout, cin), 3 * seed + 1, (2.0 / (27 * cin)) ** 0.5)
    dy = _bf16((V, cout), 3 * seed + 2, 0.1)
    return x, w, dy


def _net_inputs(c, seed):
    shape = (c["D"], c["H"], c["W"])
    params = {k: (v.bfloat16().float() if k != "head" else v) for k, v in unet.init_params(seed).items()}
    vol = _vessels({"nz": shape[0], "ny": shape[1], "nx": shape[2], "batch": 1}, seed)[0]
    g = torch.Generator(device=_dev()).manual_seed(seed + 3)
    # a back-projection is a blurred, noisy image of the target
    xin = 0.7 * vol + 0.1 * torch.randn(shape, generator=g, device=_dev())
    return params, xin.contiguous(), vol


# ------------------------------------------------------------------------------------ prepare, run

class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    s.case = c
    if c["op"] == "conv":
        L = _lib.load()
        s.x, s.w, s.dy = _conv_inputs(c, seed)
        V, cin, cout, dims = s.x.shape[0], c["cin"], c["cout"], (c["D"], c["H"], c["W"])
        dev = s.x.device
        s.wt = torch.empty((27, cin, cout), dtype=torch.bfloat16, device=dev)
        w32, wb = s.w.float(), torch.empty_like(s.w)
        _lib.check(L.pat_unet_cast_weights(w32.data_ptr(), cin, cout, wb.data_ptr(), s.wt.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        s.y = torch.empty((V, cout), dtype=torch.bfloat16, device=dev)
        s.dx = torch.empty((V, cin), dtype=torch.bfloat16, device=dev)
        s.dw = torch.empty((27, cout, cin), dtype=torch.float32, device=dev)
        s.scratch = torch.empty(L.pat_unet_wgrad_scratch(cin, cout, *dims), dtype=torch.float32, device=dev)
        return s
    if c["op"] == "network":
        params, s.xin, s.target = _net_inputs(c, seed)
        s.net = unet.WarmStartUNet(c["D"], c["H"], c["W"], params=params)
        return s
    s.op = PatOperator(_grid(c), _sampling(c, seed))
    if c["op"] in ("forward", "gradient", "prox"):
        s.p0 = _vessels(c, seed)
    if c["op"] == "prox":
        g = torch.Generator(device=_dev()).manual_seed(seed + 3)
        s.p0 += 0.05 * torch.randn(s.p0.shape, generator=g, device=s.p0.device)
        s.out = torch.empty_like(s.p0)
    if c["op"] in ("adjoint", "gradient", "solve", "sample"):
        s.f = _data(c, seed)
    if c["op"] == "sample":
        s.planes = _plane_data(c, seed)
    if c["op"] == "gradient":
        s.p0.requires_grad_(True)
    return s


def run(state):
    s, c = state, state.case
    op = c["op"]
    if op == "forward":
        return s.op.forward(s.p0)
    if op == "adjoint":
        return s.op.adjoint(s.f)
    if op == "gradient":
        s.p0.grad = None
        f = autograd.pat_forward(s.p0, s.op)
        (0.5 * (f - s.f).square().sum()).backward()
        return f.detach(), s.p0.grad
    if op == "sample":
        return s.op.sample(s.planes), s.op.sample_adjoint(s.f)
    if op == "prox":
        return s.op.tv_prox(s.p0, c["alpha"], c["iters"], out=s.out)
    if op == "solve":
        # 4.4 bounds ||A^T C^T C A|| on these grids
        p, rep = s.op.bregman_solve(s.f, c["lam"], outer=c["outer"], inner=c["inner"], prox_iters=c["prox_iters"],
                                    L=4.4)
        return p, np.asarray(rep["residuals"], dtype=np.float64)
    if op == "conv":
        L, st, dims = _lib.load(), torch.cuda.current_stream().cuda_stream, (c["D"], c["H"], c["W"])
        cin, cout = c["cin"], c["cout"]
        _lib.check(L.pat_unet_conv3(s.x.data_ptr(), cin, cin, s.w.data_ptr(), cout, s.y.data_ptr(), cout, *dims, 1, st))
        _lib.check(L.pat_unet_conv3(s.dy.data_ptr(), cout, cout, s.wt.data_ptr(), cin, s.dx.data_ptr(), cin, *dims,
                                    0, st))
        _lib.check(L.pat_unet_conv3_wgrad(s.x.data_ptr(), cin, cin, s.dy.data_ptr(), cout, cout, *dims,
                                          s.scratch.data_ptr(), s.dw.data_ptr(), st))
        return s.y, s.dx, s.dw
    out = s.net.forward(s.xin)
    loss = s.net.backward(s.target)
    return out, loss, s.net.G


# ------------------------------------------------------------------------------------ work

def _pass_flops(c):
    """One time step: per axis four complex line transforms (5 L log2 L) and 38 operations a line
    point, on half spectra; times the steps of one direction."""
    n = (c["nz"], c["ny"], c["nx"])
    points = n[0] * n[1] * n[2] / 2
    return c["batch"] * (c["T"] - 1) * sum(points * (20 * math.log2(L) + 38) for L in n)


def work(case):
    c = case
    if c["op"] == "conv":
        V, ci, co = c["D"] * c["H"] * c["W"], c["cin"], c["cout"]
        return {"bytes": 2 * V * (ci + co) * 2 + 8 * 27 * ci * co, "flops": 3 * 2 * 27 * V * ci * co}
    if c["op"] == "network":
        V = c["D"] * c["H"] * c["W"]
        macs = sum(27 * ci * co * V / 8 ** lev for ci, co, lev in unet.LAYERS.values())
        n_par = sum(27 * ci * co for ci, co, _ in unet.LAYERS.values())
        return {"bytes": 12 * V + 8 * n_par, "flops": 6 * macs}
    N, M = c["batch"] * c["nz"] * c["ny"] * c["nx"], c["ny"] * c["nx"]
    if c["op"] == "prox":
        return {"bytes": 8 * N, "flops": 40 * N * c["iters"]}
    D = c["batch"] * c["T"] * (c["m"] or M)
    if c["op"] in ("forward", "adjoint"):
        return {"bytes": 4 * (N + D), "flops": _pass_flops(c)}
    if c["op"] == "gradient":
        return {"bytes": 4 * (2 * N + 2 * D), "flops": 2 * _pass_flops(c)}
    if c["op"] == "sample":
        planes = c["batch"] * c["T"]
        fwht = M * math.log2(M) if c["kind"].startswith("shd") else 0
        return {"bytes": 8 * (planes * M + D), "flops": 2 * planes * fwht}
    pairs = c["outer"] * (c["inner"] + 0.5)
    return {"bytes": 4 * (N + D), "flops": pairs * 2 * _pass_flops(c) + c["outer"] * c["inner"] * c["prox_iters"] * 40 * N}


# ------------------------------------------------------------------------------------ exact (64 bits)

class _Wave:
    """The k-space scheme of include/pat.h and its transpose, with torch.fft in float64."""

    def __init__(self, c):
        g = self.g = _grid(c)
        dev = _dev()
        self.dt, self.c2 = g.dt, g.c * g.c
        n = (g.nz, g.ny, g.nx)

        def wn(L, half):
            m = np.arange(L // 2 + 1 if half else L)
            return 2 * np.pi * np.where(m < L // 2, m, m - L) / (L * g.dx)

        k = [torch.tensor(wn(L, ax == 2), device=dev).reshape([-1 if i == ax else 1 for i in range(3)])
             for ax, L in enumerate(n)]
        arg = 0.5 * g.c * g.dt * (k[0] ** 2 + k[1] ** 2 + k[2] ** 2).sqrt()
        self.kappa = torch.where(arg == 0, torch.ones_like(arg), arg.sin() / arg.clamp_min(1e-300))
        self.dp = [torch.polar(torch.ones_like(q), q * g.dx / 2) * 1j * q for q in k]
        self.dm = [torch.polar(torch.ones_like(q), -q * g.dx / 2) * 1j * q for q in k]

        def pml(L, shift):
            pos = np.arange(L) + shift
            P = g.pml_size
            d = np.where(pos < P, P - pos, np.where(pos > L - 1 - P, pos - (L - 1 - P), 0.0)) / max(P, 1)
            return np.exp(-g.pml_alpha * (g.c / g.dx) * d ** 4 * g.dt / 2)

        self.a, self.s = ([torch.tensor(pml(L, h), device=dev).reshape([-1 if i == ax else 1 for i in range(3)])
                           for ax, L in enumerate(n)] for h in (0.0, 0.5))
        self.n = n

    def spec(self, f):
        return torch.fft.rfftn(f) * self.kappa

    def real(self, F):
        return torch.fft.irfftn(F, s=self.n)

    def forward(self, p0):
        g, dt, r0 = self.g, self.dt, self.g.rho0
        out = torch.empty((g.T, g.m_plane), device=p0.device, dtype=torch.float64)
        out[0] = p0[g.sensor_z].reshape(-1)
        P = self.spec(p0)
        rho = [p0 / (3 * self.c2) for _ in range(3)]
        u = [dt / (2 * r0) * self.real(self.dp[i] * P) for i in range(3)]
        for t in range(1, g.T):
            for i in range(3):
                u[i] = self.s[i] * (self.s[i] * u[i] - dt / r0 * self.real(self.dp[i] * P))
                div = self.real(self.dm[i] * self.spec(u[i]))
                rho[i] = self.a[i] * (self.a[i] * rho[i] - dt * r0 * div)
            p = self.c2 * (rho[0] + rho[1] + rho[2])
            out[t] = p[g.sensor_z].reshape(-1)
            P = self.spec(p)
        return out

    def adjoint(self, y):
        g, dt, r0 = self.g, self.dt, self.g.rho0
        y = y.reshape(g.T, g.ny, g.nx)
        q = [torch.zeros(self.n, device=y.device, dtype=torch.float64) for _ in range(3)]
        v = [torch.zeros_like(q[0]) for _ in range(3)]
        for t in range(g.T - 1, 0, -1):
            lam = 0
            for i in range(3):
                q[i][g.sensor_z] += self.c2 * y[t]
                back = self.real(self.dm[i].conj() * self.spec(self.a[i] * q[i]))
                q[i] = self.a[i] ** 2 * q[i]
                v[i] = v[i] - dt * r0 * back
                lam = lam + self.dp[i].conj() * self.spec(self.s[i] * v[i])
                v[i] = self.s[i] ** 2 * v[i]
            lam = self.c2 * (-dt / r0) * self.real(lam)
            for i in range(3):
                q[i] = q[i] + lam
        p = torch.zeros_like(q[0])
        p[g.sensor_z] += y[0]
        for i in range(3):
            p += q[i] / (3 * self.c2) + dt / (2 * r0) * self.real(self.dp[i].conj() * self.spec(v[i]))
        return p


def _fwht(v):
    """Unnormalised Walsh-Hadamard transform of the last axis (Sylvester order)."""
    n, h = v.shape[-1], 1
    while h < n:
        w = v.reshape(*v.shape[:-1], n // (2 * h), 2, h)
        v = torch.stack([w[..., 0, :] + w[..., 1, :], w[..., 0, :] - w[..., 1, :]], dim=-2).reshape(v.shape)
        h *= 2
    return v


def _sample64(planes, c, s):
    M = c["ny"] * c["nx"]
    if s.kind == KIND_FULL:
        return planes
    if s.kind == KIND_RSP:
        return planes[..., torch.tensor(s.indices, device=planes.device, dtype=torch.long)]
    perm = torch.tensor(s.perm, device=planes.device, dtype=torch.long)
    w = _fwht(planes[..., perm])
    sel = w[..., torch.tensor(s.rows, device=planes.device, dtype=torch.long)]
    return sel / math.sqrt(M) if s.kind == KIND_SHDPM else 0.5 * (w[..., :1] + sel)


def _sample64_adjoint(f, c, s):
    M = c["ny"] * c["nx"]
    if s.kind == KIND_FULL:
        return f
    out = torch.zeros(f.shape[:-1] + (M,), device=f.device, dtype=torch.float64)
    if s.kind == KIND_RSP:
        out[..., torch.tensor(s.indices, device=f.device, dtype=torch.long)] = f
        return out
    out[..., torch.tensor(s.rows, device=f.device, dtype=torch.long)] = f
    w = _fwht(out)
    w = w / math.sqrt(M) if s.kind == KIND_SHDPM else 0.5 * (f.sum(-1, keepdim=True) + w)
    res = torch.empty_like(w)
    res[..., torch.tensor(s.perm, device=f.device, dtype=torch.long)] = w
    return res


def _diff(q):
    g = torch.zeros((3,) + q.shape, device=q.device, dtype=q.dtype)
    g[0, :-1] = q[1:] - q[:-1]
    g[1, :, :-1] = q[:, 1:] - q[:, :-1]
    g[2, :, :, :-1] = q[:, :, 1:] - q[:, :, :-1]
    return g


def _diff_t(x):
    o = torch.zeros_like(x[0])
    o[:-1] -= x[0, :-1]
    o[1:] += x[0, :-1]
    o[:, :-1] -= x[1, :, :-1]
    o[:, 1:] += x[1, :, :-1]
    o[:, :, :-1] -= x[2, :, :, :-1]
    o[:, :, 1:] += x[2, :, :, :-1]
    return o


def _prox64(p, alpha, iters):
    q = p.clamp_min(0)
    qb, xi = q.clone(), torch.zeros((3,) + p.shape, device=p.device, dtype=torch.float64)
    if alpha <= 0:
        return q
    tau = 1 / math.sqrt(12)
    sigma = 1 / (12 * tau)
    for _ in range(iters):
        theta = 1 / math.sqrt(1 + 2 * tau)
        xi = xi + sigma * _diff(qb)
        xi = xi / (xi.square().sum(0).sqrt() / alpha).clamp_min(1)
        new = ((q - tau * _diff_t(xi) + tau * p) / (1 + tau)).clamp_min(0)
        qb, q = new + theta * (new - q), new
        tau, sigma = theta * tau, sigma / theta
    return q


def _solve64(c, f, fwd, adj, L):
    """Bregman steps around FISTA with restart and step halving (include/pat.h, pat_bregman_solve)."""
    lam, eta = c["lam"], 1.8 / L

    def energy(ax, x, d):
        return float(0.5 * (ax - d).square().sum() + lam * _diff(x).square().sum(0).sqrt().sum())

    xp, b, residuals = torch.zeros((c["nz"], c["ny"], c["nx"]), device=f.device, dtype=torch.float64), 0 * f, []
    for _ in range(c["outer"]):
        d = f + b
        axp = fwd(xp)
        ep, y, ay, t = energy(axp, xp, d), xp, axp, 1.0
        best, stale = ep, 0
        for _ in range(c["inner"]):
            x = _prox64(y - eta * adj(ay - d), eta * lam, c["prox_iters"])
            ax = fwd(x)
            e = energy(ax, x, d)
            if e > ep:
                t, grad, h = 1.0, adj(axp - d), eta
                for _ in range(6):
                    x = _prox64(xp - h * grad, h * lam, c["prox_iters"])
                    ax = fwd(x)
                    e = energy(ax, x, d)
                    if e <= ep:
                        break
                    h *= 0.5
                if e > ep:
                    x, ax, e = xp, axp, ep
            same = bool((x == xp).all())
            tn = 0.5 * (1 + math.sqrt(1 + 4 * t * t))
            beta = (t - 1) / tn
            y, ay = x + beta * (x - xp), ax + beta * (ax - axp)
            xp, axp, ep, t = x, ax, e, tn
            best, stale = (e, 0) if e < best else (best, stale + 1)
            if same or stale >= 5:
                break
        b = b + f - axp
        residuals.append(float((axp - f).norm()))
    return xp, np.asarray(residuals)


def _conv64(x, w, shape):
    """x [V][cin], w [27][cout][cin] -> [V][cout]: 3x3x3 convolution, zero padding 1."""
    D, H, W = shape
    xp = torch.nn.functional.pad(x.reshape(D, H, W, -1), (0, 0, 1, 1, 1, 1, 1, 1))
    y = 0
    for t in range(27):
        dz, dy, dx = t // 9, (t // 3) % 3, t % 3
        y = y + xp[dz:dz + D, dy:dy + H, dx:dx + W].reshape(D * H * W, -1) @ w[t].T
    return y


def _network64(params, xin, target, s_in=1.0):
    p = {k: v.to(xin.device).double().requires_grad_(True) for k, v in params.items()}
    dims = [tuple(n >> k for n in xin.shape) for k in range(4)]

    def conv(x, name):
        return torch.relu(_conv64(x, p[name], dims[unet.LAYERS[name][2]]))

    def pool(x, lev):
        d, h, w = dims[lev + 1]
        return x.reshape(d, 2, h, 2, w, 2, -1).mean((1, 3, 5)).reshape(d * h * w, -1)

    def up(x, lev):
        d, h, w = dims[lev]
        return x.reshape(d, 1, h, 1, w, 1, -1).expand(-1, 2, -1, 2, -1, 2, -1).reshape(8 * d * h * w, -1)

    x = torch.zeros((xin.numel(), 16), device=xin.device, dtype=torch.float64)
    x[:, 0] = s_in * xin.reshape(-1).double()
    s1 = conv(conv(x, "e1a"), "e1b")
    s2 = conv(conv(pool(s1, 0), "e2a"), "e2b")
    s3 = conv(conv(pool(s2, 1), "e3a"), "e3b")
    u = conv(conv(pool(s3, 2), "e4a"), "e4b")
    u = conv(conv(torch.cat([up(u, 3), s3], 1), "d3a"), "d3b")
    u = conv(conv(torch.cat([up(u, 2), s2], 1), "d2a"), "d2b")
    h = conv(conv(torch.cat([up(u, 1), s1], 1), "d1a"), "d1b")
    out = p["head"][16] + h @ p["head"][:16]
    loss = (out - target.reshape(-1).double()).square().mean()
    loss.backward()
    grads = torch.cat([p[k].grad.reshape(-1) for k in list(unet.LAYERS) + ["head"]])
    return out.detach(), loss.detach().reshape(1), grads


def exact(case, seed):
    c = case
    if c["op"] == "conv":
        shape = (c["D"], c["H"], c["W"])
        x, w, dy = (t.double() for t in _conv_inputs(c, seed))
        x.requires_grad_(True)
        w.requires_grad_(True)
        y = _conv64(x, w, shape)
        (y * dy).sum().backward()
        return torch.relu(y.detach()), x.grad, w.grad
    if c["op"] == "network":
        return _network64(*_net_inputs(c, seed))
    if c["op"] == "prox":
        g = torch.Generator(device=_dev()).manual_seed(seed + 3)
        p0 = _vessels(c, seed)
        p0 += 0.05 * torch.randn(p0.shape, generator=g, device=p0.device)
        return torch.stack([_prox64(p.double(), c["alpha"], c["iters"]) for p in p0])
    if c["op"] in ("forward", "adjoint", "gradient") and c["nz"] * c["ny"] * c["nx"] * c["T"] * c["batch"] > 2.0e9:
        return (None, None) if c["op"] == "gradient" else None
    s = _sampling(c, seed)
    if c["op"] == "sample":
        return (_sample64(_plane_data(c, seed).double(), c, s), _sample64_adjoint(_data(c, seed).double(), c, s))
    w = _Wave(c)

    def fwd(p):
        return _sample64(w.forward(p), c, s)

    def adj(f):
        return w.adjoint(_sample64_adjoint(f, c, s))

    if c["op"] == "forward":
        return torch.stack([fwd(p.double()) for p in _vessels(c, seed)])
    f = _data(c, seed).double()
    if c["op"] == "adjoint":
        return torch.stack([adj(y) for y in f])
    if c["op"] == "solve":
        p, r = _solve64(c, f[0], fwd, adj, 4.4)
        return p[None], r
    ax = torch.stack([fwd(p.double()) for p in _vessels(c, seed)])
    return ax, torch.stack([adj(y) for y in ax - f])
