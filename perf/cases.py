"""Timed cases of the alignment library: what a subtomogram pipeline has it do.

Each case is one call through the public entry points (one call per pass) on
inputs made from a seed: Gaussian-blob templates, particles that are the same
blobs at a random pose plus noise and a missing wedge.  ``listed`` names twelve
of them, ``draw`` makes more over the same ranges.
"""
import math

import numpy as np
import torch

import paper_2603_15285_gb300 as m

PRECISIONS = {"fp64": m.FP64, "fp32": m.FP32, "tf32": m.TF32, "bf16": m.BF16}


# ---------------------------------------------------------------- the cases

def _case(kind, precision, batch, box, shells, levels, L0=None, K=2, P=16, M=3, **more):
    levels = [int(L) for L in levels]
    c = dict(kind=kind, precision=precision, batch=batch, box=box, shells=shells,
             levels=",".join(map(str, levels)), K=K, P=P, M=M, snr=0.1, shared=False,
             vary_P=False)
    c.update(more)
    return c


def listed():
    cases = []

    def add(name, *a, **kw):
        cases.append(dict(_case(*a, **kw), name=name))

    # One small particle, as picked in a viewer or on the fly at the microscope: latency.
    add("align_one_32", "align", "fp32", 1, 32, 12, (8, 12, 16), P=8, snr=0.5)
    # A production batch of subtomograms, each against its own template (the
    # throughput workload of the benchmark).
    add("align_batch_64", "align", "fp32", 1024, 64, 32, (8, 16, 24, 32))
    # The FP64 plan on a validation subset of the same data.
    add("align_fp64_64", "align", "fp64", 40, 64, 32, (8, 16, 24, 32))
    # Rotation and translation of roughly centred particles: three alternations.
    add("align6d_64", "align6d", "fp32", 96, 64, 32, (8, 16, 24, 32), rounds=3, max_shift=5,
        upsample=10, shift=3.0)
    # Encoding full-size volumes once, before they are compared with many others.
    add("analyze_200", "analyze", "fp32", 24, 200, 40, (30, 40), snr=1.0)
    # Comparing encoded particles with one encoded reference on the tensor cores.
    add("correlate_tf32", "correlate", "tf32", 768, 64, 32, (8, 16, 24, 32, 40, 48), shared=True)
    # The exhaustive first search at the published setting: 124 points per angle.
    add("search_paper", "search", "fp32", 32, 96, 40, (30, 40), P=10, M=1, snr=1.0)
    # A denser first search at low bandwidth, odd batch.
    add("search_dense", "search", "fp32", 121, 64, 32, (8, 16, 24, 32), K=4)
    # Refinement only, from known candidates, five steps per band to L = 45.
    add("refine_sta", "refine", "fp32", 200, 64, 40, (30, 40, 45), P=10, M=5, snr=1.0)
    # Refinement to the largest bandwidth, one step per band.
    add("refine_wide", "refine", "fp32", 36, 64, 32, (30, 40, 60, 100), P=10, M=1, snr=1.0)
    # Scoring given orientations with derivatives in double precision.
    add("score_fp64", "score", "fp64", 75, 64, 32, (8, 16, 24, 32))
    # The backward pass of a template optimisation over one batch of particles.
    add("template_grad_64", "template_grad", "fp32", 512, 64, 32, (8, 16, 24, 32), shared=True,
        snr=0.2)
    return cases


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _one_draw(rng):
    kind = rng.choice(["align", "align", "align6d", "analyze", "correlate", "search", "refine",
                       "score", "template_grad"])
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64", "tf32", "bf16"])
    if kind in ("analyze", "score", "template_grad", "search", "refine") and prec in ("tf32", "bf16"):
        prec = "fp32"
    box = _log_int(rng, 24, 200) if kind == "analyze" else _log_int(rng, 24, 96)
    if kind == "align6d":
        box = rng.choice([24, 30, 32, 36, 40, 48, 50, 54, 60, 64, 72])
    K = 2
    if kind in ("search", "refine") and rng.random() < 0.5:  # the large first bands
        L0 = rng.randint(12, 30)
    else:
        L0 = rng.choice([6, 8, 8, 8, 8, 9, 10, 11, 12])
        if kind == "search":
            K = rng.randint(2, 5)
    top = {"fp64": 40, "tf32": 48, "bf16": 48}.get(prec, 48)
    if kind == "refine" and prec == "fp32":
        top = rng.choice([48, 48, 100])
    LJ = max(L0 + 2, _log_int(rng, 14, top))
    step = rng.choice([4, 8, 8, 10, 20])
    levels = sorted(set(list(range(L0, LJ, step))[:15] + [LJ]))
    shells = max(8, min(48, LJ + rng.randint(-6, 3), box // 2))
    big = {"align": 900, "align6d": 96, "analyze": 600, "correlate": 1000, "search": 400,
           "refine": 600, "score": 300, "template_grad": 512}[kind]
    batch = _log_int(rng, 1, big)
    P = rng.choice([5, 8, 10, 16] if LJ > 64 else [5, 8, 10, 16, 16, 24, 32])
    c = _case(kind, prec, batch, box, shells, levels, K=K, P=P, M=rng.choice([1, 2, 3, 3, 5]),
              snr=round(rng.uniform(0.05, 1.0), 3), shared=rng.random() < 0.3,
              vary_P=kind in ("align", "search") and rng.random() < 0.3)
    if kind == "align6d":
        c.update(rounds=rng.randint(1, 3), max_shift=rng.randint(2, 6),
                 upsample=rng.choice([1, 4, 10]), shift=2.0)
    return c


def _cost(case):
    w = work(case)
    rate = 0.6e12 if case["precision"] == "fp64" else 2e13
    return w["bytes"] / 4e12 + w["flops"] / rate


def draw(rng):
    most = max(_cost(c) for c in listed())
    byte = max(work(c)["bytes"] for c in listed())
    while True:
        c = _one_draw(rng)
        if _cost(c) <= most and work(c)["bytes"] <= byte:
            return c


# ------------------------------------------------------------------- inputs

def _levels(case):
    return [int(x) for x in case["levels"].split(",")]


def _plan(case):
    L = _levels(case)
    return m.Plan(box_n=case["box"], n_shells=case["shells"], L0=L[0], K=case["K"], P=case["P"],
                  M_iter=case["M"], L_sched=L, precision=PRECISIONS[case["precision"]])


def _rotations(rng, B):
    q = rng.standard_normal((B, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                    axis=1).reshape(B, 3, 3)


def _in_ball(rng, shape, radius):
    d = rng.standard_normal(shape + (3,))
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    return d * (radius * rng.random(shape + (1,)) ** (1 / 3))


def _render(centres, amps, N, sigma, out):
    """Sums of isotropic Gaussians at (x, y, z) offsets from N/2, float32 [b][z][y][x]."""
    grid = torch.arange(N, dtype=torch.float32, device="cuda") - N / 2
    step = max(1, (1 << 28) // (centres.shape[1] * N * N))
    for b in range(0, centres.shape[0], step):
        o = torch.as_tensor(centres[b:b + step], dtype=torch.float32, device="cuda")
        a = torch.as_tensor(amps[b:b + step], dtype=torch.float32, device="cuda")
        g = torch.exp((grid - o[..., None]) ** 2 * (-0.5 / sigma ** 2))    # [b][n][xyz][N]
        yx = (g[:, :, 1, :, None] * g[:, :, 0, None, :]).flatten(2)
        z = (g[:, :, 2] * a[..., None]).transpose(1, 2)
        out[b:b + step] = torch.bmm(z, yx).view(-1, N, N, N)


def _volumes(case, seed):
    """Templates (one, or one per particle) and particles at random poses."""
    rng = np.random.default_rng([int(seed), 2603])
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    B, N = case["batch"], case["box"]
    Bt = 1 if case["shared"] else B
    n = max(12, min(160, int(0.75 * N)))
    sigma = 1.5 if N < 44 else 2.0 if N < 128 else 3.0
    off, amp = _in_ball(rng, (Bt, n), 0.37 * N), rng.uniform(0.5, 1.0, (Bt, n))
    R = _rotations(rng, B)
    tau = _in_ball(rng, (B, 1), case.get("shift", 0.0))
    templates = torch.empty((Bt, N, N, N), dtype=torch.float32, device="cuda")
    particles = torch.empty((B, N, N, N), dtype=torch.float32, device="cuda")
    _render(off, amp, N, sigma, templates)
    off, amp = np.broadcast_to(off, (B, n, 3)), np.broadcast_to(amp, (B, n))
    _render(np.einsum("bij,bnj->bni", R, off + tau), amp, N, sigma, particles)
    k = torch.fft.fftfreq(N, device="cuda")
    kx = torch.fft.rfftfreq(N, device="cuda")
    wedge = k[:, None, None].abs() <= math.tan(math.radians(60)) * kx.abs() + 1e-6
    wedge = wedge.expand(N, N, N // 2 + 1)
    step = max(1, (1 << 27) // N ** 3)
    for b in range(0, B, step):
        v = particles[b:b + step]
        var = (v * v).mean(dim=(1, 2, 3), keepdim=True) / case["snr"]
        noise = torch.empty_like(v).normal_(generator=gen)
        v += var.sqrt() * noise
        if N >= 44:  # tilt range +-60 degrees about y
            v.copy_(torch.fft.irfftn(torch.fft.rfftn(v, dim=(1, 2, 3)) * wedge, s=(N, N, N),
                                     dim=(1, 2, 3)))
    return templates, particles, R, rng


def prepare(case, seed):
    templates, particles, _, rng = _volumes(case, seed)
    plan = _plan(case)
    s = dict(case=case, plan=plan)
    B, kind = case["batch"], case["kind"]
    s["P_per"] = None
    if case["vary_P"]:
        s["P_per"] = torch.as_tensor(rng.integers(1, case["P"] + 1, B), dtype=torch.int32,
                                     device="cuda")
    if kind == "align":
        s.update(particles=particles, templates=templates, ws=m.alloc_workspace(plan, B))
        return s
    if kind == "align6d":
        stride = 0 if case["shared"] and B != 1 else 1
        s.update(particles=particles, templates=templates,
                 ws=m.alloc_workspace6d(plan, B, stride, case["max_shift"], case["upsample"]))
        return s
    if kind == "analyze":
        s.update(particles=particles)
        return s
    f, h = m.matcha_analyze(plan, particles), m.matcha_analyze(plan, templates)
    stride = 0 if case["shared"] else 1
    if kind == "correlate":
        s.update(f=f, h=h, stride=stride)
        return s
    c = m.matcha_correlate_coeffs(plan, f, h, stride)
    s["c"] = c
    if kind == "search":
        n = plan.info.soft_n
        s["grid"] = torch.empty((B, n, n, n), dtype=plan.real_dtype, device="cuda")
        return s
    # starting points near the particles' true rotations and at random, as a
    # search or an earlier iteration leaves them
    q = rng.uniform(size=(B, case["P"], 3)) * np.array([2 * np.pi, np.pi - 0.2, 2 * np.pi])
    q[..., 1] += 0.1
    s["euler"] = torch.as_tensor(q, dtype=torch.float64, device="cuda")
    if kind == "refine":
        found = m.matcha_soft_search(plan, c)
        s.update(euler=found["euler"], n_cand=found["n_cand"])
    elif kind == "template_grad":
        found = m.align_from_coefs(plan, f, h, stride)
        w = torch.as_tensor(rng.uniform(0.5, 1.5, B), dtype=torch.float64, device="cuda")
        s.update(f=f, stride=stride, euler=found["euler"], weight=w)
    torch.cuda.synchronize()
    return s


def run(s):
    case, plan = s["case"], s["plan"]
    kind = case["kind"]
    if kind == "align":
        return m.matcha_align(plan, s["particles"], s["templates"], P_per=s["P_per"], ws=s["ws"])
    if kind == "align6d":
        return m.matcha_align6d(plan, s["particles"], s["templates"], case["rounds"],
                                case["max_shift"], case["upsample"], ws=s["ws"])
    if kind == "analyze":
        return m.matcha_analyze(plan, s["particles"])
    if kind == "correlate":
        return m.matcha_correlate_coeffs(plan, s["f"], s["h"], s["stride"])
    if kind == "search":
        return m.matcha_soft_search(plan, s["c"], P_per=s["P_per"], grid=s["grid"])
    if kind == "refine":  # in place, so each pass starts from a copy
        out = m.matcha_newton_march(plan, s["c"], s["n_cand"], s["euler"].clone())
        return dict(euler=out["euler"], score=out["score"], flags=out["flags"])
    if kind == "score":
        return m.matcha_objective(plan, s["c"], s["euler"])
    return m.matcha_template_grad(plan, s["f"], s["c"], s["euler"], weight=s["weight"],
                                  template_batch_stride=s["stride"])


# --------------------------------------------------------------------- work

def _terms(L):
    """Wigner terms up to degree L: sum (2l+1)^2."""
    return (L + 1) * (2 * L + 1) * (2 * L + 3) // 3


def _steps(L):
    """Recurrence steps of one evaluation: order pairs m >= |n| times their degrees."""
    return sum((2 * k + 1) * (L - k + 1) for k in range(L + 1))


def work(case):
    """Bytes and operations of one pass: inputs once, outputs once, and the
    arithmetic of the path with its symmetries used."""
    L, B, N, S, P, K = (_levels(case), case["batch"], case["box"], case["shells"], case["P"],
                        case["K"])
    LJ, r = L[-1], 8 if case["precision"] == "fp64" else 4
    Bt = 1 if case["shared"] else B
    nlm, n = (LJ + 1) * (LJ + 2) // 2, 2 * K * (L[0] + 1)
    coef = S * nlm * 2 * r                                   # bytes per volume
    corr = 8 * r * (LJ + 1) * (LJ + 2) * (LJ + 3) // 6       # bytes per pair
    vol = 4 * N ** 3
    nphi = 2 * LJ + 2
    analyze = S * ((LJ + 1) * nphi * (14 + 2.5 * math.log2(nphi)) + 2 * nlm * (LJ + 1))
    correlate = 4 * S * _terms(LJ)
    search = n * (4 * _terms(L[0]) + 2.5 * n * n * math.log2(n * n)) + 26 * n ** 3
    refine = P * sum(_steps(x) * (36 * case["M"] + 13) for x in L)
    align = analyze + correlate + search + refine
    kind = case["kind"]
    if kind == "align":
        return dict(bytes=(B + Bt) * vol + 120 * B, flops=B * align + Bt * analyze)
    if kind == "align6d":
        fft = 2 * 5 * N ** 3 * math.log2(N ** 3)             # both volumes, complex pair
        return dict(bytes=(B + Bt) * vol + 200 * B,
                    flops=case["rounds"] * (B * (align + analyze) + B * (fft + 60 * N ** 3)))
    if kind == "analyze":
        return dict(bytes=B * (vol + coef), flops=B * analyze)
    if kind == "correlate":
        return dict(bytes=(B + Bt) * coef + B * corr, flops=B * correlate)
    if kind == "search":
        c0 = 8 * r * (L[0] + 1) * (L[0] + 2) * (L[0] + 3) // 6
        return dict(bytes=B * (c0 + r * n ** 3 + 36 * P), flops=B * search)
    if kind == "refine":
        return dict(bytes=B * (corr + 60 * P), flops=B * refine)
    if kind == "score":
        return dict(bytes=B * (corr + 104 * P), flops=B * P * 36 * _steps(LJ))
    grad = 8 * S * sum((l + 1) * (2 * l + 1) for l in range(LJ + 1)) + 36 * _steps(LJ)
    return dict(bytes=B * (coef + corr) + Bt * (coef + 2 * vol), flops=B * grad + Bt * analyze)


# ------------------------------------------------- the same in 64 bits, plainly

def _legendre(L, x):
    """Orthonormal Pbar_lm(x), m >= 0 (Condon-Shortley phase), [lm][len(x)]."""
    out = np.zeros(((L + 1) * (L + 2) // 2, len(x)))
    s = np.sqrt(1 - x * x)
    pmm = np.full_like(x, math.sqrt(1 / (4 * math.pi)))
    for mm in range(L + 1):
        if mm:
            pmm = -math.sqrt((2 * mm + 1) / (2 * mm)) * s * pmm
        prev, cur = np.zeros_like(x), pmm
        for l in range(mm, L + 1):
            out[l * (l + 1) // 2 + mm] = cur
            a = math.sqrt((4 * (l + 1) ** 2 - 1) / ((l + 1) ** 2 - mm * mm))
            b = math.sqrt((l * l - mm * mm) / (4 * l * l - 1)) if l > mm else 0.0
            prev, cur = cur, a * (x * cur - b * prev)
    return out


def _radial(case):
    x, w = np.polynomial.legendre.leggauss(case["shells"])
    R = case["box"] / 2 - 1.0
    r = R / 2 * (x + 1)
    return r, R / 2 * w * r * r


def _analysis(case, vols):
    """Shell samples (trilinear) and their spherical-harmonic coefficients:
    complex [b][s][lm] of float64 volumes."""
    L, N, S = _levels(case)[-1], case["box"], case["shells"]
    r, _ = _radial(case)
    x, w = np.polynomial.legendre.leggauss(L + 1)
    nphi = 2 * L + 2
    phi = 2 * np.pi * np.arange(nphi) / nphi
    st = np.sqrt(1 - x * x)
    d = np.stack([st[:, None] * np.cos(phi), st[:, None] * np.sin(phi),
                  np.broadcast_to(x[:, None], (L + 1, nphi))], -1)
    p = torch.as_tensor(r[:, None, None, None] * d + N / 2, device="cuda")  # [s][j][k][xyz]
    i0 = torch.floor(p)
    fr = p - i0
    i0 = i0.long()
    flat = vols.reshape(vols.shape[0], -1)
    smp = 0
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                i, j, k = i0[..., 0] + dx, i0[..., 1] + dy, i0[..., 2] + dz
                ok = ((i >= 0) & (i < N) & (j >= 0) & (j < N) & (k >= 0) & (k < N))
                wt = ((fr[..., 0] if dx else 1 - fr[..., 0]) * (fr[..., 1] if dy else 1 - fr[..., 1])
                      * (fr[..., 2] if dz else 1 - fr[..., 2])) * ok
                lin = (k.clamp(0, N - 1) * N + j.clamp(0, N - 1)) * N + i.clamp(0, N - 1)
                smp = smp + flat[:, lin.reshape(-1)].reshape((-1,) + lin.shape) * wt
    F = torch.fft.fft(smp, dim=-1)[..., :L + 1]                               # [b][s][j][m]
    P = torch.as_tensor(_legendre(L, x) * w * 2 * np.pi / nphi, device="cuda")
    lm_m = torch.as_tensor([mm for l in range(L + 1) for mm in range(l + 1)], device="cuda")
    out = torch.zeros(smp.shape[:2] + (len(lm_m),), dtype=torch.complex128, device="cuda")
    for j in range(L + 1):
        out = out + P[:, j] * F[:, :, j][..., lm_m]
    return out


def _degree(f, l):
    """[..][n = -l..l] of degree l from [..][lm], m >= 0, of real functions."""
    a = f[..., l * (l + 1) // 2:(l + 1) * (l + 2) // 2]
    sg = torch.as_tensor([(-1.0) ** k for k in range(l, 0, -1)], device=f.device)
    return torch.cat([a[..., 1:].flip(-1).conj() * sg, a], -1)


def _complex(t):
    return torch.view_as_complex(t.double().contiguous())


def _entries(L):
    """(l, m, n, entry, slot) of every stored order pair m >= |n|."""
    rows, e = [], 0
    for mm in range(L + 1):
        for j in range(mm + 1):
            for l in range(mm, L + 1):
                for slot in (0, 1):
                    if 2 * j - mm + slot <= mm:
                        rows.append((l, mm, 2 * j - mm + slot, e, slot))
                e += 1
    return np.array(rows), e


def _pack(mats, L, B):
    """Degree matrices c^l [b][m][n] in the library's grouped layout, float64."""
    rows, n = _entries(L)
    out = torch.zeros((B, n, 4, 2), dtype=torch.float64, device="cuda")
    for l in range(L + 1):
        q = torch.as_tensor(rows[rows[:, 0] == l], device="cuda")
        a, b, e, s = q[:, 1] + l, q[:, 2] + l, q[:, 3], q[:, 4]
        for k, v in enumerate((mats[l][:, a, b], mats[l][:, b, a])):
            out[:, e, 2 * k, s], out[:, e, 2 * k + 1, s] = v.real, v.imag
    return out.reshape(B, 2 * n, 2, 2)


def _unpack(c, L, upto):
    """Degree matrices [b][m][n], l <= upto, of a correlation buffer."""
    rows, n = _entries(L)
    g = c.reshape(c.shape[0], n, 4, 2).double()
    mats = []
    for l in range(upto + 1):
        q = torch.as_tensor(rows[rows[:, 0] == l], device="cuda")
        mm, nn, e, s = q[:, 1], q[:, 2], q[:, 3], q[:, 4]
        M = torch.zeros((c.shape[0], 2 * l + 1, 2 * l + 1), dtype=torch.complex128, device="cuda")
        sg = 1.0 - 2.0 * ((mm + nn) % 2)
        for k, (a, b) in enumerate(((mm, nn), (nn, mm))):
            v = torch.complex(g[:, e, 2 * k, s], g[:, e, 2 * k + 1, s])
            M[:, -a + l, -b + l] = sg * v.conj()
            M[:, a + l, b + l] = v
        mats.append(M)
    return mats


def _wigner(l, beta, order=0):
    """d^l(beta) (or its derivative of that order): [len(beta)][m][n], from the
    eigenvectors of J_y."""
    k = np.arange(-l, l)
    up = np.diag(np.sqrt(l * (l + 1) - k * (k + 1.0)), -1)         # <k+1|J_+|k>
    ev, V = np.linalg.eigh((up - up.T) / 2j)
    ev = np.round(ev)
    V, ev = torch.as_tensor(V, device="cuda"), torch.as_tensor(ev, device="cuda")
    ph = torch.exp(-1j * ev * beta.reshape(-1, 1).double()) * (-1j * ev) ** order
    return torch.einsum("ik,bk,jk->bij", V, ph, V.conj()).real


def _grid(case, c):
    L = _levels(case)
    L0, n, B = L[0], 2 * case["K"] * (L[0] + 1), c.shape[0]
    beta = torch.as_tensor(np.pi * (2 * np.arange(n) + 1) / (2 * n), device="cuda")
    mats = _unpack(c, L[-1], L0)
    ds = [_wigner(l, beta) for l in range(L0 + 1)]
    out = torch.empty((B, n, n, n), dtype=torch.float64, device="cuda")
    for b in range(B):
        S = torch.zeros((n, n, n), dtype=torch.complex128, device="cuda")   # [k][m][n]
        for l in range(L0 + 1):
            o = torch.arange(-l, l + 1, device="cuda") % n
            S[:, o[:, None], o[None, :]] += mats[l][b] * ds[l]
        out[b] = (torch.fft.ifft2(S).real * (n * n)).transpose(0, 1)
    return out


def _objective(case, c, euler):
    """C, its gradient and Hessian at [b][q][3] angles: [b][q][10]."""
    L = _levels(case)[-1]
    B, Q = euler.shape[:2]
    al, be, ga = euler.unbind(-1)
    out = torch.zeros((B, Q, 10), dtype=torch.float64, device="cuda")
    for l, M in enumerate(_unpack(c, L, L)):
        o = torch.arange(-l, l + 1, device="cuda", dtype=torch.float64)
        ea, eg = torch.exp(1j * al[..., None] * o), torch.exp(1j * ga[..., None] * o)
        for k in range(3):
            d = _wigner(l, be.reshape(-1), k).reshape(B, Q, 2 * l + 1, 2 * l + 1)
            T = M[:, None] * d

            def total(pa, pg):
                return torch.einsum("bqm,bqmn,bqn->bq", ea * (1j * o) ** pa, T,
                                    eg * (1j * o) ** pg).real
            if k == 0:
                for i, a, g in ((0, 0, 0), (1, 1, 0), (3, 0, 1), (4, 2, 0), (6, 1, 1), (9, 0, 2)):
                    out[..., i] += total(a, g)
            elif k == 1:
                for i, a, g in ((2, 0, 0), (5, 1, 0), (8, 0, 1)):
                    out[..., i] += total(a, g)
            else:
                out[..., 7] += total(0, 0)
    return out


def _template_grad(case, s):
    """Gradient of sum_b w_b C(theta_b) in the template's coefficients and
    voxels, with the implicit-function term through theta."""
    L, N, S = _levels(case)[-1], case["box"], case["shells"]
    f, eu, B = _complex(s["f"]), s["euler"], s["case"]["batch"]
    o10 = _objective(case, s["c"], eu[:, None])[:, 0]
    g = o10[:, 1:4]
    H = o10[:, [4, 5, 6, 5, 7, 8, 6, 8, 9]].reshape(B, 3, 3)
    v = torch.linalg.solve(H, g)
    wr = torch.as_tensor(_radial(case)[1], device="cuda")
    X = []
    for l in range(L + 1):
        o = torch.arange(-l, l + 1, device="cuda", dtype=torch.float64)
        ph = torch.exp(1j * (eu[:, 0, None, None] * o[:, None] + eu[:, 2, None, None] * o))
        lin = 1 - 1j * (v[:, 0, None, None] * o[:, None] + v[:, 2, None, None] * o)
        E = ph * (_wigner(l, eu[:, 1]) * lin - v[:, 1, None, None] * _wigner(l, eu[:, 1], 1))
        x = torch.einsum("b,s,bsm,bmn->bsn", s["weight"], wr.double(), _degree(f, l), E)
        sg = torch.as_tensor([(-1.0) ** k for k in range(1, l + 1)], device="cuda")
        q = x[..., l:].clone()
        q[..., 1:] += (x[..., :l].flip(-1) * sg).conj()
        X.append(q)
    G = torch.cat(X, -1)
    G = G if s["stride"] else G.sum(0, keepdim=True)
    vol = torch.zeros((G.shape[0], N, N, N), dtype=torch.float64, device="cuda", requires_grad=True)
    h = _analysis(case, vol)
    (h.real * G.real + h.imag * G.imag).sum().backward()
    return dict(coef_grad=torch.view_as_real(G), vox_grad=vol.grad, shift=torch.cat([v, o10[:, :1]], 1),
                flags=None)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("align", "align6d", "refine"):  # results of a search: no closed form
        return None
    s = prepare(case, seed)
    L = _levels(case)[-1]
    with torch.set_grad_enabled(kind == "template_grad"):
        if kind == "analyze":
            return torch.cat([torch.view_as_real(_analysis(case, v.double()))
                              for v in s["particles"].split(max(1, (1 << 26) // case["box"] ** 3))])
        if kind == "correlate":
            f, h = _complex(s["f"]), _complex(s["h"])
            w = torch.as_tensor(_radial(case)[1], device="cuda")
            mats = [torch.einsum("s,bsm,bsn->bmn", w.to(f.dtype), _degree(f, l),
                                 _degree(h, l).conj().expand(f.shape[0], -1, -1))
                    for l in range(L + 1)]
            return _pack(mats, L, f.shape[0])
        if kind == "search":
            return dict(grid=_grid(case, s["c"]), idx=None, euler=None, score=None, n_cand=None)
        if kind == "score":
            return _objective(case, s["c"], s["euler"])
        if case["batch"] > 1 and s["stride"] and case["batch"] * case["box"] ** 3 > 1 << 26:
            return None
        return _template_grad(case, s)
