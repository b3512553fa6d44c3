"""The tensor-core contraction against one shared template: the kernel that stages
the template's operand once for a block of particles and stacks particles in a
tile gives the same bits as the template repeated for every particle.  Sizes:
four, two and one particles per tile, shell counts that are not multiples of
four and more items than a thread loads ahead, blocks with a partial tile,
batches of one block and of many."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def setup(S, L, B, prec):
    plan = m.Plan(box_n=32, n_shells=S, L0=min(L, 6), K=1, P=4, M_iter=1,
                  L_sched=sorted({min(L, 6), L}), precision=prec)
    g = torch.Generator(device="cuda").manual_seed(S * L + B)
    f = torch.randn((B, S, (L + 1) * (L + 2) // 2, 2), device="cuda", generator=g)
    h = torch.randn((1, S, (L + 1) * (L + 2) // 2, 2), device="cuda", generator=g)
    return plan, f, h


@pytest.mark.parametrize("S,L,B,prec", [
    (5, 3, 1, m.TF32), (7, 14, 37, m.TF32), (32, 29, 5, m.BF16), (32, 30, 9, m.TF32),
    (30, 48, 401, m.TF32), (32, 62, 3, m.TF32), (32, 62, 70, m.BF16), (100, 30, 6, m.BF16),
    (64, 21, 11, m.TF32)])
def test_shared_template_equals_repeated(S, L, B, prec):
    plan, f, h = setup(S, L, B, prec)
    shared = m.matcha_correlate_coeffs(plan, f, h, 0)
    own = m.matcha_correlate_coeffs(plan, f, h.expand(B, -1, -1, -1).contiguous(), 1)
    torch.cuda.synchronize()
    assert plan.device_status() == 0
    assert torch.equal(shared, own)
    plan.close()


def test_shared_template_wait_limit():
    plan, f, h = setup(16, 20, 50, m.TF32)
    good = m.matcha_correlate_coeffs(plan, f, h, 0)
    plan.set_wait_limit(0)
    m.matcha_correlate_coeffs(plan, f, h, 0)
    torch.cuda.synchronize()
    assert plan.device_status() == 1
    plan.set_wait_limit(-1)
    again = m.matcha_correlate_coeffs(plan, f, h, 0)
    torch.cuda.synchronize()
    assert plan.device_status() == 0
    assert torch.equal(again, good)
    plan.close()
