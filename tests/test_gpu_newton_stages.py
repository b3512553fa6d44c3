"""The refinement spread over a cluster stages a group of up to 24 degrees at a
time (STAGE_ENTRIES): bandwidths whose longest group is one short of a piece, one
piece, one more, and the same around two and three pieces (FP32 above 64 rescaled),
against the persistent queue, whose kernel stages nothing that way.  Bit for bit:
the order of every sum is the same.  FP64 refinements are spread at every batch,
FP32 ones at few particles."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,P,prec", [((5, 22), 16, m.FP32), ((5, 23), 5, m.FP32), ((5, 23, 24), 16, m.FP32),
                                           ((6, 46, 47), 7, m.FP32), ((6, 47, 48), 16, m.FP32),
                                           ((6, 70, 71), 3, m.FP32), ((6, 72), 16, m.FP32),
                                           ((5, 22, 23), 8, m.FP64), ((5, 24), 3, m.FP64),
                                           ((6, 46, 47), 5, m.FP64), ((6, 47, 48), 16, m.FP64)])
def test_pieces_against_the_queue(levels, P, prec):
    plan = m.Plan(box_n=20, n_shells=3, L0=levels[0], K=1, P=P, M_iter=2, L_sched=levels, precision=prec)
    g = torch.Generator(device="cuda").manual_seed(sum(levels) + P)
    h = torch.randn(20, 20, 20, generator=g, device="cuda").unsqueeze(0)
    f = h + 0.5 * torch.randn(160, 20, 20, 20, generator=g, device="cuda")
    for B in (2, 160):
        outs = []
        for k in (1, 2):
            plan.set_tiles(newton_sched=k)
            outs.append(m.matcha_align(plan, f[:B].contiguous(), h))
            torch.cuda.synchronize()
        assert torch.isfinite(outs[0]["score"]).all()
        for key in ("euler", "R", "score", "best_p", "flags"):
            torch.testing.assert_close(outs[0][key], outs[1][key], rtol=0, atol=0, equal_nan=True)
    assert plan.device_status() == 0
    plan.close()
