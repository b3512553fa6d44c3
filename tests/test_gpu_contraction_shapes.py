"""The contraction at the sizes where its launch changes: one sweep of blocks per
CTA and several, bandwidths whose products pass through shared memory and ones
that are stored directly, orders that do not fill a block, one shell and many,
few CTAs and many, an output that is not 16-byte aligned; against the sums in
FP64, with the rounding bound of a sum of S products."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2603_15285_gb300 as m

pytestmark = pytest.mark.gpu


def reference(f, h, w, L):
    """(c_mn, c_nm) per layout entry, and the sums of the products' magnitudes."""
    lay = np.asarray(m.corr_layout(L))
    M, N, l = lay[:, 0], lay[:, 1], lay[:, 2]

    def at(v, order):
        k = np.abs(order)
        z = v[:, :, l * (l + 1) // 2 + np.minimum(k, l)]
        return np.where(order < 0, (-1.0) ** k * z.conj(), z)

    fm, fn = at(f, M), at(f, N)
    hm, hn = at(h, M), at(h, N)
    ww = w[None, :, None]
    z = np.stack([(ww * fm * hn.conj()).sum(1), (ww * fn * hm.conj()).sum(1)], -1)
    mag = np.stack([(ww * abs(fm) * abs(hn)).sum(1), (ww * abs(fn) * abs(hm)).sum(1)], -1)
    empty = N > M
    z[:, empty] = 0
    mag[:, empty] = 0
    return z, mag


@pytest.mark.parametrize("S,L,B,stride,prec", [
    (1, 1, 1, 0, m.FP32), (3, 2, 2, 1, m.FP64), (5, 7, 300, 0, m.FP32), (32, 16, 3, 1, m.FP32),
    (31, 33, 20, 1, m.FP32), (12, 48, 2, 0, m.FP32), (4, 70, 1, 0, m.FP32), (128, 12, 2, 1, m.FP64),
    (9, 33, 3, 0, m.FP64), (3, 52, 1, 1, m.FP64)])
def test_contraction_against_sums(S, L, B, stride, prec):
    plan = m.Plan(box_n=16, n_shells=S, L0=min(L, 4), K=1, P=4, M_iter=1,
                  L_sched=sorted({min(L, 4), L}), precision=prec, r_max=6.0)
    g = torch.Generator(device="cuda").manual_seed(S * L + B)
    nlm = (L + 1) * (L + 2) // 2
    order0 = torch.as_tensor([l * (l + 1) // 2 for l in range(L + 1)], device="cuda")

    def coefs(n):
        v = torch.randn((n, S, nlm, 2), dtype=torch.float64, device="cuda", generator=g)
        v[:, :, order0, 1] = 0.0
        return v.to(plan.real_dtype)

    f, h = coefs(B), coefs(B if stride else 1)
    c = m.matcha_correlate_coeffs(plan, f, h, stride)
    torch.cuda.synchronize()
    w = O.radial_nodes(S, 6.0)[1]  # weights with r^2 (NumPy's rule loses digits from S = 100 on)
    fz, hz = [torch.view_as_complex(v.double().contiguous()).cpu().numpy() for v in (f, h)]
    z, mag = reference(fz, np.broadcast_to(hz, fz.shape) if not stride else hz, w, L)
    got = m.corr_pairs(c.double().cpu().numpy())
    got = got[..., 0] + 1j * got[..., 1]
    eps = np.finfo(np.float64 if prec == m.FP64 else np.float32).eps
    # each part sums 2S products of rounded weights and operands
    assert np.all(abs(got - z) <= (2 * S + 8) * eps * mag + 1e-300)
    plan.close()
