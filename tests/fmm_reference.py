"""The uniform-grid fast multipole sum with the library's lists, order and truncation in numpy's long
double (64 bits of significand or more), so that what a plan's results differ by is its rounding and
nothing else.  For small grids."""
import math

import numpy as np

from paper_1610_04398_gb300 import api

LD, CLD = np.longdouble, np.clongdouble
C0 = LD(math.pi) / 4 - LD(1.5) - np.log(LD(2)) / 2


def _binom(n, k):
    return LD(math.comb(n, k)) if 0 <= k <= n else LD(0)


def multipoles(q, order):
    """Per level l: [4^l, order + 1], M_k = sum q w^k / k (entry 0: sum q) about each box's centre."""
    n = q.shape[0]
    k = np.arange(order + 1)
    out = []
    for level in range(int(np.log2(n // 8)) + 1):
        side, m = 2 ** level, n >> level
        c = (np.arange(m).astype(LD) + LD(0.5)) / m - LD(0.5)
        w = (c[None, :] + CLD(1j) * c[:, None]).ravel()
        pw = np.empty((m * m, order + 1), CLD)
        pw[:, 0] = 1
        for j in range(1, order + 1):
            pw[:, j] = pw[:, j - 1] * w
        qb = q.astype(LD).reshape(side, m, side, m).transpose(0, 2, 1, 3).reshape(side * side, m * m)
        out.append(qb.astype(CLD) @ (pw / np.maximum(k, 1)))
    return out


def locals_(M, h, n, order, theta):
    """Per level: [4^l, order + 1], complete locals b_l s^l for 2 pi P (entry 0: the constant, real)."""
    L = len(M) - 1
    k = np.arange(1, order + 1)
    R = np.array([[_binom(l + j - 1, j - 1) for j in k] for l in range(1, order + 1)])
    shift = np.array([[_binom(j, l) for j in range(order + 1)] for l in range(order + 1)])
    out = [np.zeros_like(m) for m in M]
    for level in range(2, L + 1):
        side = 2 ** level
        lns = np.log(LD(h)) + np.log(LD(n >> level))
        for c in range(4):
            ent = api.pp_m2l_entries(theta, c)
            for by in range(c >> 1, side, 2):
                for bx in range(c & 1, side, 2):
                    acc = np.zeros(order + 1, CLD)
                    for dx, dy, kind in ent:
                        if kind == 0:
                            sx, sy, ss, src = bx + dx, by + dy, side, M[level]
                            tau, rho = CLD(complex(dx, dy)), LD(1)
                        else:
                            sx, sy, ss, src = (bx >> 1) + dx, (by >> 1) + dy, side >> 1, M[level - 1]
                            tau, rho = CLD(complex(2 * dx + 0.5 - (c & 1), 2 * dy + 0.5 - (c >> 1))), LD(2)
                        if not (0 <= sx < ss and 0 <= sy < ss):
                            continue
                        m = src[sy * ss + sx]
                        it = 1 / tau
                        x = -m[1:] * np.cumprod(np.full(order, -rho * it))
                        acc[0] += m[0].real * (np.log(np.abs(tau)) + lns) + x.sum().real
                        acc[1:] += np.cumprod(np.full(order, it)) * (R.astype(CLD) @ x - m[0] / k)
                    out[level][by * side + bx] = acc
        if level > 2:  # the parent's complete locals
            for b in range(side * side):
                bx, by = b % side, b // side
                z = CLD(complex((bx & 1) - 0.5, (by & 1) - 0.5)) / 2
                p = out[level - 1][(by >> 1) * (side >> 1) + (bx >> 1)]
                pw = np.concatenate([[CLD(1)], np.cumprod(np.full(order, z))])
                sh = np.array([(p * shift[l] * np.concatenate([np.zeros(l, CLD), pw[:order + 1 - l]])).sum()
                               / LD(2) ** l for l in range(order + 1)])
                sh[0] = sh[0].real
                out[level][b] += sh
    return out


def near(q, h, theta):
    """2 pi P of the near leaves, [n, n]."""
    n = q.shape[0]
    nL = n // 8
    leaf = q.astype(LD).reshape(nL, 8, nL, 8).transpose(0, 2, 1, 3).reshape(nL, nL, 64)
    out = np.zeros((nL, nL, 64), LD)
    i = np.arange(64)
    for ox, oy in api.pp_near_offsets(theta):
        dx = (8 * ox + (i % 8)[None, :] - (i % 8)[:, None]).astype(LD)
        dy = (8 * oy + (i // 8)[None, :] - (i // 8)[:, None]).astype(LD)
        r2 = dx * dx + dy * dy
        K = np.where(r2 == 0, C0, np.log(np.where(r2 == 0, LD(1), r2)) / 2) + np.log(LD(h))
        ty, tx = np.mgrid[max(0, -oy):min(nL, nL - oy), max(0, -ox):min(nL, nL - ox)]
        out[ty, tx] += leaf[ty + oy, tx + ox] @ K.T
    return out.reshape(nL, nL, 8, 8).transpose(0, 2, 1, 3).reshape(n, n)


def far(Lo, n):
    """2 pi P of the leaf level's locals, [n, n]."""
    nL = n // 8
    i = np.arange(64)
    w = ((i % 8).astype(LD) - LD(3.5)) / 8 + CLD(1j) * (((i // 8).astype(LD) - LD(3.5)) / 8)
    pw = np.empty((64, Lo.shape[1]), CLD)
    pw[:, 0] = 1
    for j in range(1, Lo.shape[1]):
        pw[:, j] = pw[:, j - 1] * w
    return (Lo @ pw.T).real.reshape(nL, nL, 8, 8).transpose(0, 2, 1, 3).reshape(n, n)
