"""GPU test of the autotuner on the tensor-core contraction: CTAs per SM are timed
where they are a choice (a template per particle, small batches) and not where
blocks of particles share one template."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,own,timed", [(300, False, False), (300, True, True), (3, False, True)])
def test_contraction_choice(B, own, timed):
    plan = m.Plan(box_n=16, n_shells=8, L0=4, K=1, P=2, M_iter=1, L_sched=(4, 14), precision=m.TF32)
    g = torch.Generator(device="cuda").manual_seed(B)
    v = torch.randn(B, 16, 16, 16, generator=g, device="cuda")
    h = torch.randn(B if own else 1, 16, 16, 16, generator=g, device="cuda")
    rep = plan.autotune(v, h)
    if timed:
        assert rep["tc_ctas_per_sm"] in (1, 2) and min(rep["tc_ms"]) > 0
    else:
        assert rep["tc_ctas_per_sm"] == 0 and rep["tc_ms"] == [-1.0, -1.0]
    plan.set_tiles(**{k: rep[k] for k in ("analyze_shells", "tc_ctas_per_sm", "soft_kernel", "newton_sched")})
    plan.close()
