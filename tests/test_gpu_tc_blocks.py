"""GPU test of the tensor-core contraction against one template at batches around
the one where blocks of particles take over, and with blocks of every size."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,S,LJ", [(m.TF32, 8, 14), (m.TF32, 16, 24), (m.TF32, 24, 33), (m.TF32, 32, 48),
                                       (m.BF16, 16, 24), (m.BF16, 24, 33), (m.BF16, 48, 60)])
def test_tensor_core_kernels_give_the_same_bits(prec, S, LJ):
    """One template for all (blocks of particles where they win) against the same
    template per particle, around the batch where the choice changes and at blocks of
    every size."""
    plan = m.Plan(box_n=32, n_shells=S, L0=2, K=1, P=1, M_iter=1, L_sched=(2, LJ), precision=prec)
    edge = 304 // (LJ // 2 + 1)
    for B in (1, edge, edge + 1, 2 * edge + 3, 64, 131, 300):
        g = torch.Generator(device="cuda").manual_seed(B)
        f = torch.randn(B, S, plan.info.n_lm, 2, generator=g, device="cuda")
        h = torch.randn(1, S, plan.info.n_lm, 2, generator=g, device="cuda")
        one = m.matcha_correlate_coeffs(plan, f, h, 0)
        own = m.matcha_correlate_coeffs(plan, f, h.expand(B, -1, -1, -1).contiguous(), 1)
        assert plan.device_status() == 0
        assert torch.equal(one.view(torch.int32), own.view(torch.int32)), B
    plan.close()
