"""GPU tests of the contraction on the CUDA cores on both sides of the choice
between its kernels: an output whose address is no multiple of 16 takes the
direct kernel, so each plan and batch is computed by both where the records are
chosen, bit for bit (bandwidths and shell counts around the residency rule, small
plans around the batch rule, one and several sweeps, the ball-harmonic basis)."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def _contract(plan, f, h, stride, off):
    n = f.shape[0] * plan.info.corr_entries * 4
    buf = torch.full((n + 4,), float("nan"), dtype=plan.real_dtype, device="cuda")
    c = buf[off:off + n]
    st = torch.cuda.current_stream().cuda_stream
    assert m.lib().matcha_correlate_coeffs(plan.handle, f.data_ptr(), h.data_ptr(), f.shape[0], stride,
                                           c.data_ptr(), st) == 0
    torch.cuda.synchronize()
    return c.clone()


@pytest.mark.parametrize("S,LJ,ball", [(1, 3, 0), (12, 14, 0), (24, 24, 0), (24, 25, 0), (32, 32, 0), (39, 47, 0),
                                       (40, 50, 0), (24, 64, 0), (24, 66, 0), (24, 67, 0), (100, 60, 0),
                                       (128, 40, 0), (16, 20, 18.0), (16, 30, 18.0)])
@pytest.mark.parametrize("stride", [0, 1])
def test_both_kernels_give_the_same_bits(S, LJ, ball, stride):
    plan = m.Plan(box_n=48, n_shells=S, L0=2, K=1, P=1, M_iter=1, L_sched=(2, LJ), precision=m.FP32, ball_lambda=ball)
    per = LJ // 2 + 1
    for B in sorted({1, 608 // per, 608 // per + 1}):
        g = torch.Generator(device="cuda").manual_seed(B)
        f, h = (torch.randn(B, S, plan.info.n_lm, 2, generator=g, device="cuda") for _ in range(2))
        a, d = _contract(plan, f, h, stride, 0), _contract(plan, f, h, stride, 1)
        assert torch.equal(a.view(torch.int32), d.view(torch.int32)), B
        assert not torch.isnan(a).any()
    plan.close()
