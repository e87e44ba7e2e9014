"""How far a double-float apply is from the exact values, with tasks of several directions, as batches run them.  The exact
values are the recurrences in extended precision (numpy's long double, 64 bits or more); the error is measured in units of
that of the same recurrences in plain numpy FP64.

Bound, from the recurrences emulated in double-float arithmetic over these instances: 17.8 in the Legendre basis, 18.5 with
scaled modes, 25.0 in the eigenbasis of the cell matrices, so 21.5."""
import math

import numpy as np
import pytest

from gpu_common import lib, spec2d, split, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

N, RX, POLAR, AZIM = 40, 4, 4, 16


def _apply(z, ss, st, T):
    """z - sum_j omega_j (D_j + Sigma_t)^{-1} Sigma_s z on the unit square in the arithmetic T"""
    zx, wz = np.polynomial.legendre.leggauss(POLAR)
    dirs = []
    for j2 in range(POLAR // 2):
        for j1 in range(AZIM):
            th, s = (2 * j1 + 1) * math.pi / AZIM, math.sqrt(1 - zx[j2] ** 2)
            dirs.append((math.cos(th) * s, math.sin(th) * s, wz[j2] / AZIM))
    h, i = T(1) / T(N), np.arange(N) // (N // RX)
    reg = i[:, None] * RX + i[None]
    s3, eye = np.sqrt(T(3)), np.eye(2, dtype=T)
    K = np.array([[T(1), s3], [-s3, T(3)]], dtype=T)
    src, total = z.astype(T) * ss.astype(T)[reg][..., None], np.zeros((N, N, 4), T)
    for q in range(4):
        fx, fy = (1, -1)[q & 1], (1, -1)[q >> 1]
        d = [x for x in dirs if (x[0] <= 0) + 2 * (x[1] <= 0) == q]
        sgn = np.array([1, fx, fy, fx * fy], T)
        S, R = src[::fy, ::fx] * sgn, reg[::fy, ::fx]
        al, be = (np.array([abs(x[k]) for x in d], T) / h for k in (0, 1))
        w = np.array([x[2] for x in d], T)[:, None, None]
        A = (np.kron(eye, K) * al[:, None, None, None] + np.kron(K, eye) * be[:, None, None, None] +
             np.eye(4, dtype=T) * st.astype(T)[None, :, None, None])
        M = np.concatenate([A, np.broadcast_to(np.eye(4, dtype=T), A.shape)], -1)
        for c in range(4):
            M[..., c, :] /= M[..., c, c][..., None].copy()
            for r in range(4):
                if r != c:
                    M[..., r, :] -= M[..., r, c][..., None].copy() * M[..., c, :]
        M = M[..., 4:]
        X, Y, phi = np.zeros((len(d), N, 2), T), np.zeros((len(d), N, 2), T), np.zeros((N, N, 4), T)
        a, b = al[:, None], be[:, None]
        for g in range(2 * N - 1):
            iy = np.arange(max(0, g - N + 1), min(N, g + 1))
            ix = g - iy
            x, y, s = X[:, iy], Y[:, ix], S[iy, ix][None]
            r = np.stack([s[..., 0] + a * x[..., 0] + b * y[..., 0], s[..., 1] - s3 * a * x[..., 0] + b * y[..., 1],
                          s[..., 2] + a * x[..., 1] - s3 * b * y[..., 0], s[..., 3] - s3 * (a * x[..., 1] + b * y[..., 1])], -1)
            p = (M[:, R[iy, ix]] * r[..., None, :]).sum(-1)
            X[:, iy] = np.stack([p[..., 0] + s3 * p[..., 1], p[..., 2] + s3 * p[..., 3]], -1)
            Y[:, ix] = np.stack([p[..., 0] + s3 * p[..., 2], p[..., 1] + s3 * p[..., 3]], -1)
            phi[iy, ix] = (w * p).sum(0)
        total += (phi * sgn)[::fy, ::fx]
    return z.astype(T) - total


def test_error_of_double_float_applies():
    torch = torch_cuda()
    B = lib()
    n = 8
    ss, sa, z = [], [], []
    x = (np.arange(N) + 0.5) / N
    C = np.cos(math.pi * np.arange(4)[:, None] * x)
    for seed in range(n):
        rs = np.random.RandomState(seed)
        ss.append(np.exp(rs.uniform(0.0, math.log(1e3), RX * RX)))
        sa.append(rs.uniform(0.0, 0.5, RX * RX))
        v, a = 0.3 * rs.standard_normal((N, N, 4)), rs.standard_normal((4, 4))
        v[..., 0] += np.einsum("ij,iy,jx->yx", a, C, C)
        z.append(v)
    gp = B.Problem(spec2d([N] * n, [N] * n, n_polar=POLAR, n_azim=AZIM, rx=RX, ry=RX), np.array(ss), np.array(sa))
    gp.set_sweep_variant(1, 4)
    dz = to_dev(np.concatenate([v.reshape(-1) for v in z]))
    wdf = torch.empty_like(dz)
    gp.apply_op(dz, wdf, double_float=True)
    hdf = split(wdf.cpu().numpy(), gp.offsets)
    e = np.zeros(2)
    for b in range(n):
        st = ss[b] + sa[b]
        exact = _apply(z[b], ss[b], st, np.longdouble).reshape(-1)
        plain = _apply(z[b], ss[b], st, np.float64).reshape(-1)
        e += [float(((v - exact) ** 2).sum()) for v in (plain, hdf[b])]
    plain, df = np.sqrt(e)
    assert df < 21.5 * plain
