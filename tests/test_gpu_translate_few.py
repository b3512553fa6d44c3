"""GPU tests of the partial inverse transforms and the poses where their work is
split otherwise: few volumes (each group of four grid points on CTAs of its own)
and FP64 (no padded points, columns packed over the rows, voxels of a plane in
runs), at grids of 1, 4n - 1, 4n and 4n + 1 points and boxes that fill no warp."""
import numpy as np
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def _search(N, B, shift, up, prec, f, u):
    plan = m.Plan(box_n=N, n_shells=2, L0=2, K=1, P=1, M_iter=1, L_sched=(2,), precision=prec)
    o = m.matcha_shift_search(plan, f, u, shift, up)
    torch.cuda.synchronize()
    plan.close()
    return o


def _volumes(N, B, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.randn(B, N, N, N, generator=g, device="cuda")
    u = torch.roll(f, (1, -1, 0), (1, 2, 3)) + 0.3 * torch.randn(B, N, N, N, generator=g, device="cuda")
    return f, u.contiguous()


@pytest.mark.parametrize("prec", [m.FP32, m.FP64])
@pytest.mark.parametrize("N,shift,up", [(9, 0, 1), (20, 1, 2), (27, 2, 4), (45, 3, 5), (48, 10, 3), (64, 20, 30)])
def test_few_volumes_give_the_bits_of_many(N, shift, up, prec):
    """One volume per call against the same volumes among as many as fill the chip."""
    B = 2 + 152 * 256 // (N * N)
    f, u = _volumes(N, B, N)
    many = _search(N, B, shift, up, prec, f, u)
    for b in (0, B // 2, B - 1):
        one = _search(N, 1, shift, up, prec, f[b:b + 1].contiguous(), u[b:b + 1].contiguous())
        for k in ("t", "cc", "flags"):
            assert torch.equal(one[k][0], many[k][b]), (k, b)


@pytest.mark.parametrize("N,shift,up", [(9, 0, 1), (27, 2, 4), (45, 3, 5), (60, 6, 7)])
def test_fp64_values_against_numpy(N, shift, up):
    f, u = _volumes(N, 2, 100 + N)
    o = _search(N, 2, shift, up, m.FP64, f, u)
    k = np.fft.fftfreq(N, 1.0 / N)
    for b in range(2):
        X = np.fft.fftn(f[b].double().cpu().numpy()) * np.conj(np.fft.fftn(u[b].double().cpu().numpy()))
        t = o["t"][b].cpu().numpy()
        e = [np.exp(2j * np.pi / N * k * t[a]) for a in range(3)]
        cc = np.einsum("zyx,z,y,x->", X, e[2], e[1], e[0]).real / N ** 3
        scale = np.abs(X).sum() / N ** 3
        # FP64: rounding of the transforms and the three sums of N terms
        assert abs(o["cc"][b].item() - cc) <= 1e-13 * scale


@pytest.mark.parametrize("prec", [m.FP32, m.FP64])
@pytest.mark.parametrize("N", [4, 15, 16, 24, 45])
def test_pose_of_few_and_of_many_volumes(N, prec):
    """One volume per call (two or one voxels per thread) against many (eight or four)."""
    B = 2 + 40 * 16 ** 3 * 152 // max(N, 16) ** 3
    g = torch.Generator(device="cuda").manual_seed(N)
    v = torch.randn(1, N, N, N, generator=g, device="cuda")
    R = torch.from_numpy(np.linalg.qr(np.random.default_rng(N).standard_normal((B, 3, 3)))[0]).cuda()
    s = N * (torch.rand(B, 3, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    for b, x in enumerate((float("inf"), -float("inf"), float("nan"), 1e300, -1e300, 3e9, -3e9)):
        s[b, b % 3] = x
    many = m.matcha_transform_volumes(v, R, s, B=B, precision=prec)
    for b in (0, 1, 2, 3, 4, 5, 6, 7, 8, B - 1):
        one = m.matcha_transform_volumes(v, R[b:b + 1].contiguous(), s[b:b + 1].contiguous(), precision=prec)
        assert torch.equal(one[0].view(torch.int32), many[b].view(torch.int32)), b
    assert torch.isnan(many[:3]).all()            # positions that are no numbers
    far = many[3:7] if prec == m.FP64 else many[5:7]  # (1e300 is an infinity in FP32)
    assert (far == 0).all()
