"""GPU tests of the sum of the template gradient over the particles of one
template: as accurate as FP64 additions of the particles' FP32 terms, also where
large terms cancel and small ones remain."""
import numpy as np
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def _weights(kind, B):
    """Particles of equal terms up to the weight, so the weights set the sum's course."""
    w = np.empty(B)
    if kind == "half an ulp":     # a large term, then ones just below half an ulp of it
        w[:] = np.float32(2.0 ** -24 * (1 - 2.0 ** -10))
        w[0::16] = 1.0
    elif kind == "cancelling":    # large terms that cancel at the end of each 16
        w[:] = 2.0 ** -25 * (1 + np.arange(B) / B)
        w[0::16], w[15::16] = 1.0, -1.0
    else:                          # terms of all sizes and both signs
        rng = np.random.default_rng(3)
        w[:] = rng.choice([-1.0, 1.0], B) * 2.0 ** rng.uniform(-40, 0, B)
    return w


@pytest.mark.parametrize("B", [16, 33, 512])
@pytest.mark.parametrize("kind", ["half an ulp", "cancelling", "mixed"])
def test_sum_over_particles(kind, B):
    LJ = 10
    plan = m.Plan(box_n=16, n_shells=4, L0=4, K=1, P=2, M_iter=1, L_sched=(4, LJ), precision=m.FP32)
    gen = torch.Generator(device="cuda").manual_seed(5)
    one = torch.randn(1, 4, plan.info.n_lm, 2, generator=gen, device="cuda")
    h = torch.randn(1, 4, plan.info.n_lm, 2, generator=gen, device="cuda")
    f = one.expand(B, -1, -1, -1).contiguous()
    c = m.matcha_correlate_coeffs(plan, f, h, 0)
    e = torch.tensor([[0.4, 1.1, 2.0]], dtype=torch.float64, device="cuda").expand(B, -1).contiguous()
    w = torch.from_numpy(_weights(kind, B)).cuda()
    # the particles' own terms, from a template each; then their sum for a shared one
    own = m.matcha_template_grad(plan, f, c, e, weight=w, template_batch_stride=1, voxels=False)["coef_grad"]
    tot = m.matcha_template_grad(plan, f, c, e, weight=w, template_batch_stride=0, voxels=False)["coef_grad"]
    x = own.cpu().numpy().astype(np.longdouble)
    want, size = x.sum(axis=0), np.abs(x).sum(axis=0)
    got = tot[0].cpu().numpy().astype(np.longdouble)
    plan.close()
    # FP64 additions lose at most 2^-53 of the partial sums each, and the result is
    # rounded to FP32 once
    bound = B * 2.0 ** -53 * size + 2.0 ** -24 * np.abs(want)
    assert (np.abs(got - want) <= bound).all(), float((np.abs(got - want) / np.maximum(bound, 1e-300)).max())
