"""The translation search and the volume pose at the sizes where their kernels
change path: box edges of every FFT radix (odd ones too), planes that fit in
shared memory and planes that do not, grid windows on both sides of the points a
column takes per pass, against plain NumPy transforms; poses that reach outside
the box, non-finite shifts."""
import numpy as np
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def freqs(N):
    k = np.arange(N)
    return np.where(k < (N + 1) // 2, k, k - N)


def grid(X, t):
    """N^-3 Re sum_k X(k) e^{2 pi i k.t/N} on the product of the axes' points t = (x, y, z)."""
    N = X.shape[0]
    e = [np.exp(2j * np.pi * np.outer(freqs(N), a) / N) for a in t]
    return np.einsum("zyx,xi,yj,zk->kji", X, e[0], e[1], e[2], optimize=True).real / N ** 3


@pytest.mark.parametrize("N,shift,up,prec", [
    (24, 2, 1, m.FP64), (45, 4, 10, m.FP64), (30, 9, 24, m.FP32), (80, 3, 4, m.FP64),
    (120, 2, 10, m.FP32), (27, 8, 2, m.FP32), (50, 1, 7, m.FP32), (72, 5, 10, m.FP32)])
def test_shift_search_against_numpy(N, shift, up, prec):
    B = 3
    rng = np.random.default_rng(N)
    ax = np.arange(N) - N / 2
    z, y, x = np.meshgrid(ax, ax, ax, indexing="ij")
    f, u = [], []
    for b in range(B):
        t = rng.uniform(-0.8 * shift, 0.8 * shift, 3)
        o = rng.uniform(-N / 6, N / 6, (6, 3))
        f.append(sum(np.exp(-((x - q[0] - t[0]) ** 2 + (y - q[1] - t[1]) ** 2 + (z - q[2] - t[2]) ** 2) / 8) for q in o))
        u.append(sum(np.exp(-((x - q[0]) ** 2 + (y - q[1]) ** 2 + (z - q[2]) ** 2) / 8) for q in o))
    f = (np.stack(f) + 0.1 * rng.standard_normal((B, N, N, N))).astype(np.float32)
    u = np.stack(u).astype(np.float32)
    plan = m.Plan(box_n=N, n_shells=2, L0=2, K=1, P=1, M_iter=1, L_sched=(2,), precision=prec)
    o = m.matcha_shift_search(plan, torch.from_numpy(f).cuda(), torch.from_numpy(u).cuda(), shift, up)
    torch.cuda.synchronize()
    # FP64: rounding of two transforms; FP32: sqrt(N^3) terms of relative 2^-24, bounded generously
    tol = 1e-11 if prec == m.FP64 else 2e-5
    h = int(np.floor(0.75 * up))
    for b in range(B):
        X = np.fft.fftn(f[b].astype(np.float64)) * np.conj(np.fft.fftn(u[b].astype(np.float64)))
        w = np.arange(-shift, shift + 1)
        c0 = grid(X, (w, w, w))
        i0 = np.unravel_index(np.argmax(c0), c0.shape)[::-1]
        t0 = np.array([w[q] for q in i0], float)
        fine = [t0[a] + np.arange(-h, h + 1) / up for a in range(3)]
        c1 = grid(X, fine)
        i1 = np.unravel_index(np.argmax(c1), c1.shape)[::-1]
        got = o["t"][b].cpu().numpy()
        at = [np.argmin(np.abs(fine[a] - got[a])) for a in range(3)]
        assert np.allclose([fine[a][at[a]] for a in range(3)], got, atol=1e-12)
        scale = np.abs(c1).max()
        # the returned point's value: the maximum up to rounding, and reported as such
        assert c1[at[2], at[1], at[0]] >= c1.max() - tol * scale
        assert abs(o["cc"][b].item() - c1[at[2], at[1], at[0]]) <= tol * scale
        if prec == m.FP64:
            assert at == list(i1)
    plan.close()


@pytest.mark.parametrize("N", [4, 17, 33])
@pytest.mark.parametrize("prec", [m.FP64, m.FP32])
def test_pose_against_numpy(N, prec):
    rng = np.random.default_rng(N)
    B = 3
    v = rng.standard_normal((B, N, N, N)).astype(np.float32)
    q, _ = np.linalg.qr(rng.standard_normal((B, 3, 3)))
    s = rng.uniform(-N, N, (B, 3))
    s[0] = 0.25
    s[2] = (1e12, 0, 0)  # far outside
    out = m.matcha_transform_volumes(torch.from_numpy(v).cuda(), torch.from_numpy(q).cuda(),
                                     torch.from_numpy(s).cuda(), precision=prec).cpu().numpy()
    ax = np.arange(N) - N / 2
    z, y, x = np.meshgrid(ax, ax, ax, indexing="ij")
    for b in range(B):
        p = np.stack([x, y, z], -1).reshape(-1, 3) @ q[b] + N / 2 - s[b]
        i0 = np.floor(p)
        fr = p - i0
        want = np.zeros(N ** 3)
        for d in np.ndindex(2, 2, 2):
            i = i0 + np.array(d)
            ok = ((i >= 0) & (i < N)).all(1)
            w = np.prod(np.where(d, fr, 1 - fr), 1)
            k = np.where(ok[:, None], i, 0).astype(int)
            want += np.where(ok, w * v[b][k[:, 2], k[:, 1], k[:, 0]], 0.0)
        # FP32 coordinates carry an error of a few 2^-24 N; a corner value changes by O(1)
        tol = 1e-6 if prec == m.FP64 else 3e-5 * N
        assert np.abs(out[b].reshape(-1) - want).max() <= tol, b
    nan = torch.full((B, 3), float("nan"), dtype=torch.float64, device="cuda")
    out = m.matcha_transform_volumes(torch.from_numpy(v).cuda(), None, nan, precision=prec)
    assert torch.isnan(out).all()
