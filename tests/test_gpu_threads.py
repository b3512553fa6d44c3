"""GPU tests of calls from several host threads at once, each on its own stream,
whose launches of one kernel ask for different amounts of shared memory: the
limit of a kernel is one value for all of them, so a call may never lower it
below what another's launch is about to ask for.  Every call succeeds and gives
the bits it gives alone."""
import threading

import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu

CALLS = 2500


def _plan(prec, LJ, S=8, P=16, K=2, L0=8):
    return m.Plan(box_n=16, n_shells=S, L0=L0, K=K, P=P, M_iter=1, L_sched=(L0, LJ) if LJ > L0 else (L0,),
                  precision=prec)


def _c(plan, B, gen):
    return torch.randn(B, plan.info.corr_entries, 2, 2, generator=gen, device="cuda", dtype=plan.real_dtype)


def _angles(B, Q, gen):
    a = torch.rand(B, Q, 3, generator=gen, device="cuda", dtype=torch.float64)
    return a * torch.tensor([6.28, 3.14, 6.28], dtype=torch.float64, device="cuda")


def _objective(plan, B, gen):
    c, e = _c(plan, B, gen), _angles(B, plan.P, gen)
    out = torch.empty(B, plan.P, 10, dtype=torch.float64, device="cuda")
    args = (plan.handle, c.data_ptr(), B, plan.L_final, plan.P, e.data_ptr(), out.data_ptr())
    return m.lib().matcha_objective, args, (out,), (c, e)


def _march(plan, B, gen):
    c, e = _c(plan, B, gen), _angles(B, plan.P, gen)
    n = torch.zeros(B, dtype=torch.int32, device="cuda")  # no candidates: the launch is what counts
    s = torch.zeros(B, plan.P, dtype=torch.float64, device="cuda")
    fl = torch.ones(B, plan.P, dtype=torch.int32, device="cuda")
    args = (plan.handle, c.data_ptr(), B, n.data_ptr(), e.data_ptr(), s.data_ptr(), fl.data_ptr(), None)
    return m.lib().matcha_newton_march, args, (e, s, fl), (c, n)


def _correlate(plan, B, gen):
    f, h = (torch.randn(B, plan.n_shells, plan.info.n_lm, 2, generator=gen, device="cuda",
                        dtype=plan.real_dtype) for _ in range(2))
    c = torch.empty(B, plan.info.corr_entries, 2, 2, dtype=plan.real_dtype, device="cuda")
    args = (plan.handle, f.data_ptr(), h.data_ptr(), B, 1, c.data_ptr())
    return m.lib().matcha_correlate_coeffs, args, (c,), (f, h)


def _search(plan, B, gen):
    c = _c(plan, B, gen)
    n = plan.info.soft_n
    grid = torch.empty(B, n, n, n, dtype=plan.real_dtype, device="cuda")
    idx = torch.empty(B, plan.P, dtype=torch.int32, device="cuda")
    e = torch.empty(B, plan.P, 3, dtype=torch.float64, device="cuda")
    s = torch.empty(B, plan.P, dtype=torch.float64, device="cuda")
    k = torch.empty(B, dtype=torch.int32, device="cuda")
    args = (plan.handle, c.data_ptr(), B, None, grid.data_ptr(), idx.data_ptr(), e.data_ptr(), s.data_ptr(),
            k.data_ptr())
    return m.lib().matcha_soft_search, args, (grid, idx, e, k), (c, s)


def _gradient(plan, B, gen):
    f = torch.randn(B, plan.n_shells, plan.info.n_lm, 2, generator=gen, device="cuda", dtype=plan.real_dtype)
    c, e = _c(plan, B, gen), _angles(B, 1, gen)
    g = torch.empty(1, plan.n_shells, plan.info.n_lm, 2, dtype=plan.real_dtype, device="cuda")
    sh = torch.empty(B, 4, dtype=torch.float64, device="cuda")
    size = m.ctypes.c_size_t()
    assert m.lib().matcha_template_grad_workspace_size(plan.handle, B, 0, m.ctypes.byref(size)) == 0
    ws = torch.empty(size.value, dtype=torch.uint8, device="cuda")
    args = (plan.handle, f.data_ptr(), c.data_ptr(), B, 0, e.data_ptr(), None, g.data_ptr(), None, sh.data_ptr(),
            None, ws.data_ptr(), size.value)
    return m.lib().matcha_template_grad, args, (g, sh), (f, c, e, ws)


# (call, plans of the two threads (None: the first one's), batches): in each the two
# launches of a kernel ask for different amounts
CASES = {
    "objective, two batches of a plan": (_objective, [dict(prec=m.FP64, LJ=16), None], (4, 160)),
    "refinement, two batches of a plan": (_march, [dict(prec=m.FP64, LJ=16), None], (4, 160)),
    "gradient, two batches of a plan": (_gradient, [dict(prec=m.FP32, LJ=32, S=32), None], (1, 310)),
    "refinement, two plans": (_march, [dict(prec=m.FP32, LJ=16), dict(prec=m.FP32, LJ=40)], (160, 160)),
    "contraction, two plans": (_correlate, [dict(prec=m.FP32, LJ=32, S=64), dict(prec=m.FP32, LJ=32, S=128)], (2, 2)),
    "search, two plans": (_search, [dict(prec=m.FP32, LJ=0, L0=12, K=3), dict(prec=m.FP32, LJ=0, L0=16, K=3)], (2, 2)),
}


@pytest.mark.parametrize("name", CASES)
def test_shared_memory_limits_of_concurrent_calls(name):
    call, plans, batches = CASES[name]
    gen = torch.Generator(device="cuda").manual_seed(7)
    plans = [_plan(**p) if p else None for p in plans]
    work = [call(p or plans[0], B, gen) for p, B in zip(plans, batches)]
    alone = []
    for fn, args, outs, _ in work:
        assert fn(*args, torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        alone.append([o.clone() for o in outs])
    streams = [torch.cuda.Stream() for _ in work]
    start = threading.Barrier(len(work))
    bad = [None] * len(work)

    def loop(i):
        fn, args, _, _ = work[i]
        st = streams[i].cuda_stream
        torch.cuda.set_device(0)
        start.wait()
        bad[i] = sum(fn(*args, st) != 0 for _ in range(CALLS))

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for p in plans:
        if p:
            p.close()
    assert bad == [0] * len(work)
    for (_, _, outs, _), want in zip(work, alone):
        for o, w in zip(outs, want):
            assert torch.equal(o, w)
