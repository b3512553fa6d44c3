"""GPU tests of the template gradient where its shells are split over CTAs: the
part counts follow the batch and what fits, and change no bit of a particle's
coefficients (odd shell counts, parts of one and of several tiles, shells that do
not fit one CTA, batches around one and two CTAs per SM)."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,S,LJ", [(m.FP32, 1, 9), (m.FP32, 7, 16), (m.FP32, 32, 20), (m.FP32, 40, 64),
                                       (m.FP64, 3, 9), (m.FP64, 12, 16), (m.FP64, 24, 32), (m.FP64, 41, 50)])
def test_parts_give_the_same_bits(prec, S, LJ):
    plan = m.Plan(box_n=16, n_shells=S, L0=4, K=1, P=2, M_iter=1, L_sched=(4, LJ), precision=prec)
    Bs = [1, 19, 38, 76, 77, 152, 153, 305]
    g = torch.Generator(device="cuda").manual_seed(S)
    f = torch.randn(Bs[-1], S, plan.info.n_lm, 2, generator=g, device="cuda", dtype=plan.real_dtype)
    c = torch.randn(Bs[-1], plan.info.corr_entries, 2, 2, generator=g, device="cuda", dtype=plan.real_dtype)
    e = 0.1 + torch.rand(Bs[-1], 3, generator=g, device="cuda", dtype=torch.float64)
    want = None
    for B in reversed(Bs):
        o = m.matcha_template_grad(plan, f[:B].contiguous(), c[:B].contiguous(), e[:B].contiguous(),
                                   template_batch_stride=1, voxels=False)
        if want is None:
            want = o
        assert torch.equal(o["coef_grad"], want["coef_grad"][:B]), B
        assert torch.equal(o["shift"], want["shift"][:B]), B
    plan.close()
