"""The SOFFT search through memory (soft_grid.cu) against the slice-streaming
kernel, which the allocation-free entry point runs on the same plans: the same
candidates, bit for bit, at grid sizes around the kernels' tiles (8 x 8 and 4 x
4 blocks, runs of 30 gammas, several beta slices per CTA), on plateaus, with
NaN and infinite coefficients and per-particle candidate counts; and the grid's
own local maxima by brute force."""
import numpy as np
import pytest
import torch

import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def plan(L0, K, P, prec):
    return m.Plan(box_n=16, n_shells=2, L0=L0, K=K, P=P, M_iter=1, L_sched=(L0, L0 + 3), precision=prec)


def both(p, c, P_per=None):
    a = m.matcha_soft_search(p, c, P_per=P_per)
    B, P = c.shape[0], p.P
    b = dict(idx=torch.empty((B, P), dtype=torch.int32, device="cuda"),
             euler=torch.empty((B, P, 3), dtype=torch.float64, device="cuda"),
             score=torch.empty((B, P), dtype=torch.float64, device="cuda"),
             n_cand=torch.empty((B,), dtype=torch.int32, device="cuda"))
    m.matcha_soft_search_noalloc(p, c, b["idx"], b["euler"], b["score"], b["n_cand"], P_per=P_per)
    torch.cuda.synchronize()
    for k in b:
        x, y = a[k].cpu().numpy(), b[k].cpu().numpy()
        assert np.array_equal(x, y, equal_nan=k == "score"), k
    return a


def random_c(p, B, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = torch.randn((B, p.info.corr_entries, 2, 2), dtype=torch.float64, device="cuda", generator=g)
    return c.to(p.real_dtype).contiguous()


def brute(grid, P):
    """Indices of the P strongest local maxima of one [i][k][j] grid."""
    n = grid.shape[0]
    idx = np.arange(n ** 3).reshape(n, n, n)
    ok = ~np.isnan(grid)
    for di in (-1, 0, 1):
        for dk in (-1, 0, 1):
            for dj in (-1, 0, 1):
                if not (di or dk or dj):
                    continue
                v = np.roll(grid, (-di, -dj), (0, 2))
                q = np.roll(idx, (-di, -dj), (0, 2))
                lo, hi = max(0, -dk), n - max(0, dk)
                a, b = grid[:, lo:hi], v[:, lo + dk:hi + dk]
                ok[:, lo:hi] &= (a > b) | ((a == b) & (idx[:, lo:hi] < q[:, lo + dk:hi + dk]))
    p = np.flatnonzero(ok)
    return p[np.lexsort((p, -grid.reshape(-1)[p]))][:P]


@pytest.mark.parametrize("L0,K,prec", [(8, 4, m.FP32), (10, 3, m.FP32), (14, 2, m.FP32), (6, 5, m.FP32),
                                       (11, 2, m.FP64), (8, 3, m.FP64), (29, 1, m.FP32)])
@pytest.mark.parametrize("B,P", [(1, 32), (3, 5)])
def test_candidates_match_the_streaming_kernel(L0, K, prec, B, P):
    p = plan(L0, K, P, prec)
    c = random_c(p, B, L0 * 100 + K)
    per = torch.arange(B, dtype=torch.int32, device="cuda") * 3
    both(p, c, P_per=per)
    a = both(p, c)
    grid = a["grid"].cpu().numpy()
    for b in range(B):
        want = brute(grid[b], P)
        got = a["idx"][b].cpu().numpy()
        assert a["n_cand"][b].item() == len(want) and np.array_equal(got[:len(want)], want)
    p.close()


@pytest.mark.parametrize("prec", [m.FP32, m.FP64])
def test_plateaus_and_non_finite_values(prec):
    p = plan(11, 3, 8, prec)
    c = random_c(p, 5, 7)
    c[0] = 0                      # one plateau over the whole grid
    c[1] = float("nan")
    c[2, 0, 0, 0] = float("inf")
    c[3] = 0
    c[3, 0, 0, 0] = -1.0          # a negative constant
    a = both(p, c)
    assert a["n_cand"][1].item() == 0
    p.close()


@pytest.mark.parametrize("prec", [m.FP32, m.FP64])
def test_unaligned_grid(prec):
    """A grid that starts off a 16-byte boundary takes element stores."""
    p = plan(11, 3, 8, prec)
    c, n = random_c(p, 2, 3), p.info.soft_n
    a = m.matcha_soft_search(p, c)
    room = torch.empty(2 * n ** 3 + 1, dtype=p.real_dtype, device="cuda")
    g = room[1:].view(2, n, n, n)
    b = m.matcha_soft_search(p, c, grid=g)
    assert torch.equal(a["grid"], b["grid"]) and torch.equal(a["idx"], b["idx"])
    p.close()
