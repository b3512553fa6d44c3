"""GPU tests of searches and refinements at batches around the numbers of clusters
that run at once (the choice of CTAs per particle changes there, and with it the
kernel): every particle's results are those of the particle alone, bit for bit, and
those of a call whose parts run on several streams."""
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu

EDGES = (15, 16, 36, 37, 46, 47, 76, 77, 97, 98, 153)


def _coeffs(plan, B, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    f, h = (torch.randn(B, plan.n_shells, plan.info.n_lm, 2, generator=g, device="cuda", dtype=plan.real_dtype)
            for _ in range(2))
    return m.matcha_correlate_coeffs(plan, f, h, 1)


def _same(a, b, keys):
    for k in keys:
        x, y = (t.view(torch.int64) if t.dtype == torch.float64 else t for t in (a[k], b[k]))
        assert torch.equal(x, y), k


@pytest.mark.parametrize("prec,L0,K", [(m.FP32, 8, 2), (m.FP32, 6, 2), (m.FP32, 6, 3), (m.FP32, 11, 2),
                                       (m.FP64, 4, 2), (m.FP64, 8, 2)])
def test_search(prec, L0, K):
    plan = m.Plan(box_n=16, n_shells=4, L0=L0, K=K, P=9, M_iter=1, L_sched=(L0, L0 + 1), precision=prec)
    c = _coeffs(plan, EDGES[-1], L0)
    ref = None
    for B in reversed(EDGES):
        s = m.matcha_soft_search(plan, c[:B].contiguous())
        ref = ref or s
        _same(s, {k: v[:B] for k, v in ref.items()}, ("idx", "euler", "score", "n_cand", "grid"))
    plan.close()


@pytest.mark.parametrize("prec,LJ,P", [(m.FP32, 16, 16), (m.FP32, 40, 16), (m.FP32, 32, 8), (m.FP32, 24, 24),
                                       (m.FP32, 70, 10), (m.FP64, 16, 16), (m.FP64, 20, 32)])
def test_refinement(prec, LJ, P):
    plan = m.Plan(box_n=16, n_shells=4, L0=4, K=1, P=P, M_iter=2, L_sched=(4, LJ), precision=prec)
    c = _coeffs(plan, EDGES[-1], LJ)
    s = m.matcha_soft_search(plan, c)
    ref = obj = None
    for B in reversed(EDGES):
        cb, e = c[:B].contiguous(), s["euler"][:B].contiguous()
        r = m.matcha_newton_march(plan, cb, s["n_cand"][:B].contiguous(), e.clone())
        o = m.matcha_objective(plan, cb, e)
        ref, obj = (ref or r), (o if obj is None else obj)
        _same(r, {k: v[:B] for k, v in ref.items() if v is not None}, ("euler", "score", "flags"))
        # (missing candidates have beta = 0, where no derivative exists)
        assert torch.equal(torch.isnan(o), torch.isnan(obj[:B]))
        assert torch.equal(torch.nan_to_num(o), torch.nan_to_num(obj[:B]))
    plan.close()


@pytest.mark.parametrize("prec", [m.FP32, m.FP64])
def test_parts_of_one_alignment(prec):
    plan = m.Plan(box_n=16, n_shells=5, L0=6, K=2, P=8, M_iter=2, L_sched=(6, 12), precision=prec)
    B = 300
    g = torch.Generator(device="cuda").manual_seed(1)
    v, h = (torch.randn(B, 16, 16, 16, generator=g, device="cuda") for _ in range(2))
    v, h = (torch.nn.functional.avg_pool3d(x[:, None], 3, 1, 1)[:, 0].contiguous() for x in (v, h))
    a = m.matcha_align(plan, v, h)
    for b0, b1 in ((0, 40), (40, 90), (255, 300)):
        b = m.matcha_align(plan, v[b0:b1].contiguous(), h[b0:b1].contiguous())
        _same(b, {k: x[b0:b1] for k, x in a.items()}, ("euler", "R", "score", "best_p", "flags"))
    plan.close()
