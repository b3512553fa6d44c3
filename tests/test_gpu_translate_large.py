"""GPU tests of the translation search at box edges whose planes are
transformed a direction at a time (k_fft_axis) and whose columns are as many as
shared memory holds beside the twiddles: FP64 takes eight columns per CTA from
N = 450 on, sixteen below."""
import math

import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def _on_grid(X, axes):
    """CC on a grid of shifts, axes = (x, y, z) points: N^-3 Re sum_k X(k) e^{2 pi i k.t/N}."""
    N = X.shape[0]
    k = torch.fft.fftfreq(N, d=1.0 / N, dtype=torch.float64, device=X.device)
    e = [torch.exp(2j * math.pi / N * k[:, None] * t[None, :]) for t in axes]
    Y = torch.einsum("zyx,za->ayx", X, e[2])
    Y = torch.einsum("ayx,yb->abx", Y, e[1])
    return torch.einsum("abx,xc->abc", Y, e[0]).real / N ** 3


def _blobs(N, centres):
    ax = torch.arange(N, dtype=torch.float64, device="cuda") - N / 2
    v = torch.zeros(N, N, N, dtype=torch.float64, device="cuda")
    for c in centres:
        g = [torch.exp(-(ax - c[a]) ** 2 / 18) for a in range(3)]
        v += g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
    return v


@pytest.mark.parametrize("N", [432, 450, 512])
def test_large_boxes_in_fp64(N):
    up, edge = 4, 2
    gen = torch.Generator(device="cuda").manual_seed(N)
    centres = (torch.rand(6, 3, generator=gen, device="cuda", dtype=torch.float64) - 0.5) * N / 3
    shift = torch.tensor([0.75, -1.25, 1.0], dtype=torch.float64, device="cuda")
    u = _blobs(N, centres).float()
    f = _blobs(N, centres + shift)
    f = (f + 0.05 * torch.randn(f.shape, generator=gen, device="cuda", dtype=torch.float64)).float()
    plan = m.Plan(box_n=N, n_shells=2, L0=2, K=1, P=1, M_iter=1, L_sched=(2,), precision=m.FP64)
    o = m.matcha_shift_search(plan, f[None].contiguous(), u[None].contiguous(), edge, up)
    torch.cuda.synchronize()
    plan.close()
    X = torch.fft.fftn(f.double()) * torch.fft.fftn(u.double()).conj()
    w = torch.arange(-edge, edge + 1, dtype=torch.float64, device="cuda")
    c0 = _on_grid(X, (w, w, w))
    q = int(c0.argmax())
    t0 = [w[q % 5], w[q // 5 % 5], w[q // 25]]
    h = int(math.floor(0.75 * up))
    off = torch.arange(-h, h + 1, dtype=torch.float64, device="cuda") / up
    fine = [t + off for t in t0]
    c1 = _on_grid(X, fine)
    got = o["t"][0]
    at = [int((fine[a] - got[a]).abs().argmin()) for a in range(3)]
    assert all(abs(float(fine[a][at[a]] - got[a])) < 1e-12 for a in range(3))
    # FP64: rounding of two transforms, as for the small boxes
    scale = float(c1.abs().max())
    value = float(c1[at[2], at[1], at[0]])
    assert value >= float(c1.max()) - 1e-11 * scale
    assert abs(float(o["cc"][0]) - value) <= 1e-11 * scale
    assert torch.allclose(got, shift, atol=0.5)
