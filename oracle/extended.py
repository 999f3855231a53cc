"""The singular self rule of Thm 1 (Sec. 2.2) in extended precision (`numpy.longdouble`, 64 bits of mantissa on
x86), for the rounding errors of FP64 implementations (oracle; test infrastructure only).

The same discrete sum as `layer.SelfQuadrature`, with nodes, weights, Legendre functions and rotations formed
anew in extended precision.  The rotated expansions come from the values at the rotated grid points and the
exact discrete analysis of Sec. 2.1, not from Wigner matrices.
"""
from __future__ import annotations

import numpy as np

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def gauss(n: int):
    """Gauss-Legendre nodes (ascending) and weights: Newton steps from the FP64 nodes."""
    def poly(t):
        p0, p1 = np.ones_like(t), t.copy()
        for k in range(2, n + 1):
            p0, p1 = p1, ((2 * k - 1) * t * p1 - (k - 1) * p0) / LD(k)
        return p1, n * (t * p1 - p0) / (t * t - 1)

    t = np.polynomial.legendre.leggauss(n)[0].astype(LD)
    for _ in range(4):
        p, dp = poly(t)
        t = t - p / dp
    dp = poly(t)[1]
    return t, 2 / ((1 - t * t) * dp * dp)


def legendre(p: int, ct: np.ndarray, st: np.ndarray) -> np.ndarray:
    """Normalised P~_n^m (App. A, Condon-Shortley phase), [n][m][points], n, m <= p + 1."""
    P = np.zeros((p + 2, p + 2) + ct.shape, dtype=LD)
    P[0, 0] = np.sqrt(1 / (4 * PI))
    for m in range(p + 1):
        P[m + 1, m + 1] = -np.sqrt(1 + LD(1) / (2 * (m + 1))) * st * P[m, m]
        P[m + 1, m] = np.sqrt(LD(2 * m + 3)) * ct * P[m, m]
        for n in range(m + 2, p + 2):
            a = np.sqrt((4 * LD(n) * n - 1) / (LD(n) * n - LD(m) * m))
            b = np.sqrt(((LD(n) - 1) ** 2 - LD(m) * m) / (4 * (LD(n) - 1) ** 2 - 1))
            P[n, m] = a * (ct * P[n - 1, m] - b * P[n - 2, m])
    return P


def self_rule(xcoef: np.ndarray, p: int, pq: int, densities, lats) -> np.ndarray:
    """Raw rule for 'S' and 'D' (as `layer.SelfQuadrature.apply`) at the targets of some latitudes, for every
    density (FP64 coefficients [3][(p+1)^2]): extended-precision [S, D][density][3][lat][b]."""
    idx = [(n, m) for n in range(p + 1) for m in range(n + 1)]
    N, M = (np.array(v) for v in zip(*idx))
    tri = lambda T: np.stack([T[n, m] for n, m in idx])
    fac = np.where(M == 0, LD(1), LD(2))
    fields = [np.asarray(c, dtype=np.float64).reshape(3, -1) for c in [xcoef, *densities]]
    re = np.concatenate([c[:, N * (N + 1) + M] for c in fields]).astype(LD)
    im = np.concatenate([np.where(M > 0, c[:, N * (N + 1) - M], 0.0) for c in fields]).astype(LD)
    t, w = gauss(p + 1)
    tq, wq = gauss(pq + 1)
    st, sq = np.sqrt(1 - t * t), np.sqrt(1 - tq * tq)
    phi, phq = PI * np.arange(2 * p + 2).astype(LD) / (p + 1), PI * np.arange(2 * pq + 2).astype(LD) / (pq + 1)
    Pg, Tq = tri(legendre(p, t, st)), legendre(p, tq, sq)
    Pq = tri(Tq)
    dPq = np.stack([np.sqrt(LD((n - m) * (n + m + 1))) * Tq[n, m + 1] + m * tq / sq * Tq[n, m] for n, m in idx])
    cg, sg = np.cos(np.outer(M.astype(LD), phi)), np.sin(np.outer(M.astype(LD), phi))
    pole = np.where(M == 0, np.sqrt((2 * N.astype(LD) + 1) / (4 * PI)), LD(0))
    # singular weights (Thm 1)
    s, p0, p1 = 1 + tq, np.ones_like(tq), tq.copy()
    for k in range(2, pq + 1):
        p0, p1 = p1, ((2 * k - 1) * tq * p1 - (k - 1) * p0) / LD(k)
        s = s + p1
    wt = (PI / (pq + 1) * wq * 2 * np.sqrt((1 - tq) / 2) * s / sq)[:, None]

    def synth(T, dphi, r, i):
        out = np.zeros((len(r), pq + 1, 2 * pq + 2), dtype=LD)
        for m in range(p + 1):
            q = M == m
            hr, hi = (r[:, q] * fac[q]) @ T[q], (i[:, q] * fac[q]) @ T[q]
            c, sn = np.cos(m * phq), np.sin(m * phq)
            out += m * (-hr[:, :, None] * sn - hi[:, :, None] * c) if dphi else hr[:, :, None] * c - hi[:, :, None] * sn
        return out

    out = np.zeros((2, len(fields) - 1, 3, len(lats), 2 * p + 2), dtype=LD)
    vx, vy = st[:, None] * np.cos(phi), st[:, None] * np.sin(phi)
    vz = np.broadcast_to(t[:, None], vx.shape)
    for la, a in enumerate(lats):
        y0, y2 = t[a] * vx + st[a] * vz, -st[a] * vx + t[a] * vz
        for b in range(2 * p + 2):
            z0, z1 = np.cos(phi[b]) * y0 - np.sin(phi[b]) * vy, np.sin(phi[b]) * y0 + np.cos(phi[b]) * vy
            B = fac[:, None] * tri(legendre(p, y2.ravel(), np.sqrt(z0 * z0 + z1 * z1).ravel()))
            ang = np.outer(M.astype(LD), np.arctan2(z1, z0).ravel())
            val = (re @ (B * np.cos(ang)) - im @ (B * np.sin(ang))).reshape(-1, p + 1, 2 * p + 2)
            val = val * (PI / (p + 1)) * w[None, :, None]
            gr = np.stack([np.sum((val[:, :, :] @ cg[i]) * Pg[i], axis=1) for i in range(len(idx))], axis=1)
            gi = -np.stack([np.sum((val[:, :, :] @ sg[i]) * Pg[i], axis=1) for i in range(len(idx))], axis=1)
            X, Xt, Xp = synth(Pq, 0, gr[:3], gi[:3]), synth(dPq, 0, gr[:3], gi[:3]), synth(Pq, 1, gr[:3], gi[:3])
            n = np.stack([Xt[1] * Xp[2] - Xt[2] * Xp[1], Xt[2] * Xp[0] - Xt[0] * Xp[2], Xt[0] * Xp[1] - Xt[1] * Xp[0]])
            W = np.sqrt(np.sum(n * n, axis=0))
            xh = (gr[:3] @ pole)[:, None, None] - X
            r = np.sqrt(np.sum(xh * xh, axis=0))
            for d in range(len(fields) - 1):
                rho = synth(Pq, 0, gr[3 + 3 * d: 6 + 3 * d], gi[3 + 3 * d: 6 + 3 * d])
                xr = np.sum(xh * rho, axis=0)
                out[0, d, :, la, b] = np.sum((rho / r + xh * (xr / r ** 3)) * (wt * W), axis=(1, 2))
                out[1, d, :, la, b] = np.sum(-6 * xh * (xr * np.sum(xh * n, axis=0) / r ** 5) * wt, axis=(1, 2))
    return out
