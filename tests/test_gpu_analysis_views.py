"""GPU test of alignments whose particles and templates together need more texture
views than one launch carries (192^3: a view per volume), against smaller batches
that share a launch."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [m.FP32, m.FP64])
def test_more_views_than_a_launch(prec):
    N, B = 192, 150
    plan = m.Plan(box_n=N, n_shells=2, L0=3, K=1, P=3, M_iter=1, L_sched=(3, 5), precision=prec)
    g = torch.Generator(device="cuda").manual_seed(0)
    v = torch.randn(B, N, N, N, generator=g, device="cuda")
    h = torch.randn(B, N, N, N, generator=g, device="cuda")
    whole = m.matcha_align(plan, v, h)
    for b0 in (0, B // 2):
        part = m.matcha_align(plan, v[b0:b0 + B // 2], h[b0:b0 + B // 2])
        for k in ("euler", "score", "best_p", "flags"):
            assert torch.equal(part[k], whole[k][b0:b0 + B // 2]), (k, b0)
    # and the coefficients of either batch alone
    f = m.matcha_analyze(plan, v)
    for b in (0, B - 1):
        assert torch.equal(m.matcha_analyze(plan, v[b:b + 1])[0], f[b])
    plan.close()
