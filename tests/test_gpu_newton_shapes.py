"""The refinement's launch shapes: a particle on one CTA or spread over a
cluster (the shape follows the batch) gives the same bits, so a batch aligned
particle by particle, in small batches and whole agrees with itself; the
objective likewise.  Sizes: bandwidths around the staging buffer's length (16
degrees), candidate counts on both sides of 16 lanes, the rescaled recurrence
above L_J = 64, plans with fewer sub-slots than eight warps hold."""
import numpy as np
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu

CASES = [((5,), 4, m.FP32, 2), ((4, 15), 16, m.FP32, 3), ((6, 16, 17), 17, m.FP32, 3),
         ((8, 33), 5, m.FP64, 2), ((8, 20), 32, m.FP64, 1), ((10, 64, 70), 16, m.FP32, 1),
         ((12, 48), 10, m.FP64, 1), ((30, 100), 7, m.FP32, 2)]


@pytest.mark.parametrize("levels,P,prec,M", CASES)
def test_batches_of_any_size_agree(levels, P, prec, M):
    plan = m.Plan(box_n=16, n_shells=2, L0=levels[0], K=1, P=P, M_iter=M, L_sched=levels, precision=prec)
    B = 340
    g = torch.Generator(device="cuda").manual_seed(sum(levels) + P)
    # a decaying spectrum, so that the start points climb to nearby maxima
    lay = torch.as_tensor(m.corr_layout(levels[-1])[:, 2], device="cuda")
    amp = torch.exp(-0.15 * lay.double())
    c = torch.randn((9, plan.info.corr_entries, 2, 2), dtype=torch.float64, device="cuda", generator=g)
    c = (c * amp.repeat_interleave(4).view(1, -1, 2, 2)).to(plan.real_dtype)
    c = c[torch.arange(B, device="cuda") % 9].contiguous()
    q = torch.rand((9, P, 3), dtype=torch.float64, device="cuda", generator=g)
    q = q * torch.tensor([6.28, 2.9, 6.28], dtype=torch.float64, device="cuda") + 0.1
    euler = q[torch.arange(B, device="cuda") % 9].contiguous()
    n_cand = (torch.arange(B, dtype=torch.int32, device="cuda") % 9) * P // 8
    n_cand = torch.clamp(n_cand, max=P).to(torch.int32)

    def march(sel):
        work = torch.zeros((len(sel), 2), dtype=torch.int64, device="cuda")
        o = m.matcha_newton_march(plan, c[sel].contiguous(), n_cand[sel].contiguous(),
                                  euler[sel].contiguous(), work=work)
        obj = m.matcha_objective(plan, c[sel].contiguous(), euler[sel].contiguous())
        torch.cuda.synchronize()
        return {k: o[k].cpu().numpy() for k in ("euler", "score", "flags", "work")} | {"obj": obj.cpu().numpy()}

    whole = march(list(range(B)))
    assert plan.device_status() == 0
    assert np.isfinite(whole["obj"]).all()
    for n in (1, 3, 9, 40, 100, 200):
        part = march(list(range(n)))
        for k in whole:
            assert np.array_equal(part[k], whole[k][:n], equal_nan=k == "score"), (k, n)
    # the nine distinct particles repeat through the batch
    for k in whole:
        assert np.array_equal(whole[k][9:18], whole[k][:9], equal_nan=k == "score"), k
    assert plan.device_status() == 0
    plan.close()
