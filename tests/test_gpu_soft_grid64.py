"""GPU test of the FP64 search through memory against the streaming search, bit for
bit, at odd and even numbers of order rows and points per angle."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L0,K", [(9, 2), (10, 2), (12, 2), (6, 3), (5, 5), (4, 7)])
def test_fp64_grids_through_memory(L0, K):
    """The slab kernel's FP64 items against the streaming kernel (no grid given)."""
    plan = m.Plan(box_n=16, n_shells=4, L0=L0, K=K, P=16, M_iter=1, L_sched=(L0, L0 + 1), precision=m.FP64)
    g = torch.Generator(device="cuda").manual_seed(L0)
    f, h = (torch.randn(3, 4, plan.info.n_lm, 2, generator=g, device="cuda", dtype=torch.float64) for _ in range(2))
    c = m.matcha_correlate_coeffs(plan, f, h, 1)
    s = m.matcha_soft_search(plan, c)
    B, P = 3, 16
    i32, f64 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.float64, device="cuda")
    n = m.matcha_soft_search_noalloc(plan, c, torch.empty(B, P, **i32), torch.empty(B, P, 3, **f64),
                                     torch.empty(B, P, **f64), torch.empty(B, **i32))
    for k in ("idx", "euler", "n_cand"):
        assert torch.equal(s[k], n[k]), k
    assert torch.equal(torch.nan_to_num(s["score"]), torch.nan_to_num(n["score"]))
    plan.close()
