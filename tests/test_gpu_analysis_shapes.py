"""The analysis gives the same bits whatever shape its launch takes: shells per
CTA pinned or chosen (small and large boxes, bandwidths at which four CTAs of
two shells do or do not fit an SM, batches of one wave and of several), and
particles and templates in one launch or in two (texture views for both, for
neither, or for one of them)."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,S,L,B,prec", [
    (32, 12, 16, 1, m.FP32), (64, 8, 40, 160, m.FP32), (48, 6, 39, 3, m.FP32), (128, 10, 20, 2, m.FP32),
    (136, 6, 48, 3, m.FP32), (131, 4, 12, 2, m.FP32), (48, 6, 20, 5, m.FP64), (128, 4, 10, 1, m.FP64)])
def test_shells_per_cta(N, S, L, B, prec):
    plan = m.Plan(box_n=N, n_shells=S, L0=4, K=1, P=4, M_iter=1, L_sched=[4, L], precision=prec)
    g = torch.Generator(device="cuda").manual_seed(N + L)
    v = torch.randn((B, N, N, N), device="cuda", generator=g)
    auto = m.matcha_analyze(plan, v)
    for G in (1, 2):
        plan.set_tiles(analyze_shells=G)
        assert torch.equal(m.matcha_analyze(plan, v), auto)
    plan.close()


@pytest.mark.parametrize("N,stride,shift", [(32, 0, 0), (32, 1, 0), (32, 1, 4), (30, 1, 0), (32, 0, 4)])
def test_particles_and_templates_in_one_launch(N, stride, shift):
    plan = m.Plan(box_n=N, n_shells=8, L0=6, K=1, P=6, M_iter=2, L_sched=[6, 11], precision=m.FP32)
    B = 5
    g = torch.Generator(device="cuda").manual_seed(N + stride)
    buf = torch.randn(B * N ** 3 + shift, device="cuda", generator=g)
    parts = buf[shift:].view(B, N, N, N)   # shifted: no texture view
    temps = torch.randn((B if stride else 1, N, N, N), device="cuda", generator=g)
    out = m.matcha_align(plan, parts, temps)
    f, h = m.matcha_analyze(plan, parts), m.matcha_analyze(plan, temps)
    ref = m.align_from_coefs(plan, f, h, stride)
    torch.cuda.synchronize()
    for k in ("euler", "R", "score", "best_p", "flags"):
        assert torch.equal(out[k], ref[k]), k
    plan.close()
