"""The search of a small batch spreads a particle's beta slices over a cluster
of CTAs: the same candidates, in the same order, as the chunked kernel, for
batches on both sides of each choice; maxima on the slices where two CTAs meet
(every slice has some over this many particles), equal values (a flat grid, a
grid constant in alpha), no candidates wanted, fewer maxima than wanted."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 2, 16, 17, 101, 102])
def test_split_search_equals_the_chunked_kernel(B):
    plan = m.Plan(box_n=16, n_shells=2, L0=8, K=2, P=32, M_iter=1, L_sched=[8, 11], precision=m.FP32)
    lay = m.corr_layout(11)
    g = torch.Generator(device="cuda").manual_seed(B)
    c = torch.randn((B, plan.info.corr_entries, 2, 2), device="cuda", generator=g)
    if B > 1:
        c[0] = 0.0                       # flat
        keep = torch.as_tensor(lay[:, 0] == 0, device="cuda")
        c[1][~keep] = 0.0                # constant in alpha
    want = torch.arange(B, dtype=torch.int32, device="cuda") % 33 if B > 2 else None
    outs = []
    for k in (1, 3):
        plan.set_tiles(soft_kernel=k)
        outs.append(m.matcha_soft_search(plan, c, P_per=want))
    torch.cuda.synchronize()
    for key in ("grid", "idx", "score", "euler", "n_cand"):
        torch.testing.assert_close(outs[0][key], outs[1][key], rtol=0, atol=0, equal_nan=True)
    plan.close()


@pytest.mark.parametrize("L0,K,prec", [(8, 2, m.FP64), (4, 1, m.FP64), (9, 1, m.FP32), (5, 3, m.FP32)])
def test_chunked_search_of_any_batch(L0, K, prec):
    """Also the chunked kernel splits small batches: a batch too large to split
    agrees with its parts."""
    plan = m.Plan(box_n=16, n_shells=2, L0=L0, K=K, P=20, M_iter=1, L_sched=[L0, L0 + 3], precision=prec)
    plan.set_tiles(soft_kernel=1)
    B = 700
    g = torch.Generator(device="cuda").manual_seed(L0)
    c = torch.randn((13, plan.info.corr_entries, 2, 2), dtype=plan.real_dtype, device="cuda", generator=g)
    c[3] = 0.0
    c = c[torch.arange(B, device="cuda") % 13].contiguous()
    want = torch.arange(B, dtype=torch.int32, device="cuda") % 13 + 8
    whole = m.matcha_soft_search(plan, c, P_per=want)
    for n in (1, 2, 7, 40, 76, 130, 290):
        part = m.matcha_soft_search(plan, c[:n].contiguous(), P_per=want[:n].contiguous())
        torch.cuda.synchronize()
        for key in ("grid", "idx", "score", "euler", "n_cand"):
            torch.testing.assert_close(part[key], whole[key][:n], rtol=0, atol=0, equal_nan=True)
    plan.close()
