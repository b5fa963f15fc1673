"""Host-side model of the TV prox's two-iteration kernel (tv_step2_kernel and tv2_plan in pat_solver.cu), no GPU.

A CTA owns H rows of y (and 128 columns of lines longer than that) over a run of z planes.  A thread holds four
consecutive x of one of the H + 3 rows y0 - 2 .. y0 + H; split lines have one more thread on each side.  Marching along
z from two planes before the run, it does the first iteration at plane z and the second at plane z - 1.  This test
restates, per plane and for all threads at once, the global reads, the exchanges through shared memory (poisoned where
nothing was written) and the stores, in FP64, and checks over the plans of the kernel that every read is inside its
buffer, every voxel is stored exactly once, nothing undefined reaches a stored value, and pairs of iterations equal the
oracle's prox (App. B)."""
import math

import numpy as np
import pytest

COLS, THREADS = 128, 384


def plan(nz, ny, nx, B):
    split = nx > COLS
    ntx = COLS // 4 + 2 if split else nx // 4
    H = 16
    while H > 8 and (H + 3) * ntx > THREADS:
        H //= 2
    H = min(H, ny)
    if H > 8 and (H + 3) * ntx > 128 and ((ny + 7) // 8) * nz * B <= 152:
        H = 8
    gx, gy = (nx + COLS - 1) // COLS if split else 1, (ny + H - 1) // H
    threads = (H + 3) * ntx
    resident = 152 * max(1, 14 // -(-threads // 32))
    best = None
    for run in range(1, nz + 1):
        n = (nz + run - 1) // run
        if B * n > 65535:
            continue
        cost = -(-(gx * gy * B * n) // resident) * (run + 3)
        if best is None or cost < best[0]:
            best = cost, run, n
    assert threads <= THREADS
    return split, ntx, H, gx, gy, best[1], best[2]


def dual(sigma, alpha, d, gz, gy, gx):
    e = d[0] + sigma * gz, d[1] + sigma * gy, d[2] + sigma * gx
    with np.errstate(invalid="ignore", divide="ignore"):
        n = np.sqrt(e[0] ** 2 + e[1] ** 2 + e[2] ** 2)
        s = np.where(n > alpha, alpha / n, 1.0)
    return [v * s for v in e]


def launch(qb_in, xi_in, q_in, p, alpha, par, dims, B, the_plan):
    nz, ny, nx = dims
    split, ntx, H, gxn, gyn, zrun, nruns = the_plan
    n, N, plane, rows, cols = nz * ny * nx, B * nz * ny * nx, ny * nx, H + 3, 4 * ntx
    out = {"q": np.full(N, np.nan), "qb": np.full(N, np.nan), "xi": np.full(3 * N, np.nan)}
    written = np.zeros(N, int)
    undefined = np.full((rows, cols), np.nan)

    def read(buf, idx, mask):
        assert ((idx >= 0) & (idx < len(buf)))[mask].all()
        return np.where(mask, buf[np.where(mask, idx, 0)], 0.0)

    def right(a, last):     # the value at x + 1: within a thread, and `last` for its fourth voxel
        r = np.roll(a, -1, 1)
        r[:, 3::4] = last
        return r

    def left(a):            # at x - 1: the thread before's fourth voxel, 0 before the first thread
        r = np.roll(a, 1, 1)
        r[:, 0] = 0.0
        return r

    def above(a, first):    # at y - 1
        return np.concatenate([first, a[:-1]])

    for bx in range(gxn):
        for by in range(gyn):
            for bz in range(B * nruns):
                b, run = divmod(bz, nruns)
                z0, z1 = run * zrun, min(run * zrun + zrun, nz)
                tx = np.arange(cols)[None, :] // 4
                x = np.arange(cols)[None, :] + (bx * COLS - 4 if split else 0) + np.zeros((rows, 1), int)
                y = by * H - 2 + np.arange(rows)[:, None] + np.zeros((1, cols), int)
                x4 = x - x % 4 if not split else x - (np.arange(cols)[None, :] % 4)
                inn = (x4 >= 0) & (x4 < nx) & (y >= 0) & (y < ny)
                rr = np.arange(rows)[:, None]
                own = inn & (rr >= 2) & (rr < H + 2) & ((tx > 0) & (tx < ntx - 1) if split else True)
                yn, xn = y + 1 < ny, x + 1 < nx
                base = b * n + y * nx + x

                def primal(k, z, q, pv, dz, pz, dy, dyl, dx):
                    gt = np.where(z + 1 < nz, -dz, 0.0) + (pz if z > 0 else 0.0)
                    gt = gt - np.where(yn, dy, 0.0) + np.where(y > 0, dyl, 0.0)
                    gt = gt - np.where(xn, dx, 0.0) + np.where(x > 0, left(dx), 0.0)
                    v = np.maximum(0.0, (q + par["tau"][k] * pv - par["tau"][k] * gt) / (1.0 + par["tau"][k]))
                    return v, v + par["theta"][k] * (v - q)

                zs = z0 - 2 if z0 > 1 else 0
                qc = read(qb_in, base + zs * plane, inn)
                zero = np.zeros((rows, cols))
                pz1 = pz2 = zero
                d1, q1, qb1, p1 = [zero] * 3, zero, zero, zero
                sqb = [undefined, undefined]
                for z in range(zs, z1 + 1):
                    o, on = base + z * plane, inn & (z < nz)
                    qn_in = read(qb_in, o + plane, on & (z + 1 < nz))
                    qy_in = read(qb_in, o + nx, on & yn)
                    qx_in = read(qb_in, o + 1, on & xn & (np.arange(cols)[None, :] % 4 == 3))
                    d = [read(xi_in, c * N + o, on) for c in range(3)]
                    qv, pv = read(q_in, o, on), read(p, o, on)
                    d = dual(par["sigma"][0], alpha, d, qn_in - qc if z + 1 < nz else zero, np.where(yn, qy_in - qc, 0.0),
                             np.where(xn, right(qc, qx_in[:, 3::4]) - qc, 0.0))
                    qnew, qb = primal(0, z, qv, pv, d[0], pz1, d[1], above(d[1], zero[:1]), d[2])
                    sqb[z & 1] = qb
                    e = d1
                    if z > zs:
                        so = sqb[(z - 1) & 1]
                        qy = np.concatenate([so[1:], zero[:1]])
                        nxt = np.concatenate([so[:, 4::4], zero[:, :1]], 1)
                        e = dual(par["sigma"][1], alpha, d1, qb - qb1 if z < nz else zero, np.where(yn, qy - qb1, 0.0),
                                 np.where(xn, right(qb1, nxt) - qb1, 0.0))
                    store = own if z - 1 >= z0 else np.zeros_like(own)
                    if store.any():
                        q2, qb2 = primal(1, z - 1, q1, p1, e[0], pz2, e[1], above(e[1], undefined[:1]), e[2])
                        w = (o - plane)[store]
                        out["q"][w], out["qb"][w] = q2[store], qb2[store]
                        for c in range(3):
                            out["xi"][c * N + w] = e[c][store]
                        written[w] += 1
                    pz1, pz2, d1, q1, qb1, p1, qc = d[0], e[0], d, qnew, qb, pv, qn_in
    assert (written == 1).all(), np.unique(written, return_counts=True)
    return out


@pytest.mark.parametrize("shape,B", [((8, 8, 8), 1), ((16, 32, 8), 2), ((32, 32, 32), 1), ((8, 16, 256), 2),
                                     ((64, 8, 16), 1), ((8, 32, 128), 1), ((16, 16, 64), 3)])
def test_pairs_match_the_oracle_prox(shape, B, oracle_mod):
    from oracle import solver
    nz, ny, nx = shape
    n = nz * ny * nx
    P = np.random.default_rng(3).standard_normal((B,) + shape) * 0.5 + 0.2
    p = P.ravel().copy()
    q = np.maximum(0.0, p)
    qb, xi = q.copy(), np.zeros(3 * B * n)
    alpha, iters = 0.2, 6
    tau = 1.0 / math.sqrt(12.0)
    sigma = 1.0 / (tau * 12.0)
    # the kernel's plan, and one with runs of three planes, so that every z halo occurs
    own = plan(nz, ny, nx, B)
    for k in range(iters // 2):
        par = {"sigma": [], "tau": [], "theta": []}
        for _ in range(2):
            theta = 1.0 / math.sqrt(1.0 + 2.0 * tau)
            par["sigma"].append(sigma)
            par["tau"].append(tau)
            par["theta"].append(theta)
            tau, sigma = theta * tau, sigma / theta
        r = launch(qb, xi, q, p, alpha, par, shape, B, own if k != 1 else own[:5] + (3, (nz + 2) // 3))
        qb, xi, q = r["qb"], r["xi"], r["q"]
    for b in range(B):
        ref = solver.tv_prox(P[b], alpha, iters)
        got = q[b * n:(b + 1) * n].reshape(shape)
        assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
