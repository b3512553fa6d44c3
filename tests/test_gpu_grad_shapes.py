"""Template gradient at the sizes where its kernels change shape: one shell and
many per CTA, shell counts that leave a partial tile, odd and even bandwidths up
to the largest whose state fits in shared memory, batches with and without a
partial block of the reduction, records that are not 16-byte aligned; random
coefficients at random rotations against the oracle's adjoint."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2603_15285_gb300 as m
from gpu_helpers import coef_to_complex

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,S,L,B,prec", [
    (10, 3, 4, 1, m.FP64), (16, 5, 7, 3, m.FP64), (20, 9, 12, 70, m.FP32), (16, 6, 9, 150, m.FP32),
    (24, 7, 33, 2, m.FP32), (16, 3, 58, 2, m.FP64), (16, 2, 64, 1, m.FP32)])
def test_gradient_against_the_oracle(N, S, L, B, prec):
    R = 0.45 * N
    plan = m.Plan(box_n=N, n_shells=S, L0=min(4, L), K=1, P=4, M_iter=1,
                  L_sched=sorted({min(4, L), L}), r_max=R, precision=prec)
    rng = np.random.default_rng(L * B)
    deg = np.concatenate([np.full(l + 1, l) for l in range(L + 1)])
    order = np.concatenate([np.arange(l + 1) for l in range(L + 1)])
    amp = np.exp(-0.1 * deg)

    def coefs(*lead):
        v = amp * (rng.normal(size=lead + (S, len(deg))) + 1j * rng.normal(size=lead + (S, len(deg))))
        return np.where(order == 0, v.real, v)

    def device(v):
        return torch.view_as_real(torch.as_tensor(v, device="cuda")).to(plan.real_dtype).contiguous()

    f, h = device(coefs(B)), device(coefs(1))
    c = m.matcha_correlate_coeffs(plan, f, h, 0)
    eu = rng.uniform(0.2, 2.9, (B, 3))
    w = rng.uniform(0.5, 1.5, B)
    eud, wd = torch.as_tensor(eu, device="cuda"), torch.as_tensor(w, device="cuda")
    out = m.matcha_template_grad(plan, f, c, eud, weight=wd)
    each = m.matcha_template_grad(plan, f, c, eud, template_batch_stride=1)
    odd = torch.empty(c.numel() + 1, dtype=c.dtype, device="cuda")[1:].view(c.shape).copy_(c)
    moved = m.matcha_template_grad(plan, f, odd, eud, weight=wd)
    torch.cuda.synchronize()
    fo, ho = coef_to_complex(f), coef_to_complex(h[0])
    G, v4, flags = O.template_grad_batch(fo, ho, eu, S=S, r_max=R, L_sched=[L], N=N)
    assert not flags.any() and not out["flags"].cpu().numpy().any()
    # H v = grad: the error of the values is amplified by H's condition number.
    # Values: the recurrences lose a few times L ulps.
    plan64 = m.Plan(box_n=N, n_shells=S, L0=min(4, L), K=1, P=4, M_iter=1,
                    L_sched=sorted({min(4, L), L}), r_max=R, precision=m.FP64)
    c64 = m.matcha_correlate_coeffs(plan64, f.double(), h.double(), 0)
    o10 = m.matcha_objective(plan64, c64, eud[:, None].contiguous()).cpu().numpy().reshape(B, -1)
    H = o10[:, [4, 5, 6, 5, 7, 8, 6, 8, 9]].reshape(B, 3, 3)
    eps = np.finfo(np.float64 if prec == m.FP64 else np.float32).eps
    tol = 4 * L * eps * (10 + np.linalg.cond(H))
    np.testing.assert_allclose(out["shift"].cpu().numpy()[:, 3], v4[:, 3], rtol=0,
                               atol=4 * L * eps * np.abs(v4[:, 3]).max() * 10)
    for b in range(B):
        e = np.abs(coef_to_complex(each["coef_grad"][b]) - G[b]).max() / np.abs(G[b]).max()
        assert e < tol[b], (b, e, tol[b])
    total = (G * w[:, None, None]).sum(0)
    size = np.abs(G).max(axis=(1, 2)) * w
    bound = (tol * size).sum()
    assert np.abs(coef_to_complex(out["coef_grad"][0]) - total).max() < bound
    vox = O.analysis_adjoint(total, N, S, R, L)
    # the adjoint of the sampling, held against its own input's error
    slack = bound / np.abs(total).max() * 10
    assert np.abs(out["vox_grad"][0].cpu().numpy() - vox).max() < slack * np.abs(vox).max()
    for k in ("coef_grad", "shift"):
        assert torch.equal(moved[k], out[k])
    assert plan.device_status() == 0
    plan.close()
    plan64.close()
