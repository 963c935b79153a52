"""Workloads of the sparse correlation match, each through the package's public calls.

A case names the operation (``op``), the plan (crystal phases, grid step, shells, in-plane
bins, operand precision) and the batch (patterns and how their peak lists come about).  The
values are those of the repository's own configurations and tests, or lie between them:
plans of 0.5 to 6 degrees on 40 to 200 shells and 72 to 360 bins, scans of one pattern (a
live display) to 65,536 (a whole 256 x 256 scan), 5 to 80 peaks a pattern.

Operations:
  match     match(): the indexing of a batch (options: runner-up, per-phase scores, top-K
            rescoring), which is what a user of the library runs most
  refined   match() on a coarse plan with its runner-up, then refine(): continuous orientations
  score     kinematical_score() / kinematical_score_strain() forward and backward
  multi     match_multi(): overlapping patterns
  bounds    bounds(): the shell contraction alone
  spectra   polar_spectra(): the polar images' spectra alone
  plan      Plan(): building an orientation plan, and its spectra
"""

import math

import numpy as np
import torch

from paper_2111_00171_gb300 import acom

LAM, DELTA, QMAX, SIGMA = 0.01969, 0.08, 1.5, 0.02
PREC = {"fp32": acom.ACOM_PREC_FP32, "bf16": acom.ACOM_PREC_BF16, "fp16": acom.ACOM_PREC_FP16,
        "fp8": acom.ACOM_PREC_FP8}
OPERAND = {"fp32": 8, "bf16": 4, "fp16": 4, "fp8": 2}      # bytes of a complex plan value
# peak lists: mean number of peaks a pattern
PEAKS = {"uniform": 35, "poisson": 30, "threshold": 33, "overlap": 60}


def _case(name, op, step, patterns, precision="fp16", shells=150, dq=0.01, phi=360,
          peaks="uniform", **more):
    return {"name": name, "op": op, "phases": "Au", "step": step, "shells": shells, "dq": dq,
            "phi": phi, "precision": precision, "patterns": patterns, "peaks": peaks, **more}


def listed():
    return [
        # one pattern at a time under a live display: launches and latency
        _case("live_1", "match", 1.0, 1),
        # the paper's plain method: 100 independent patterns, 2-degree grid, FP32 operands
        _case("plain_100_fp32", "match", 2.0, 100, "fp32", 75, 0.02, 180, "threshold"),
        # a small scan, its size no multiple of a tile
        _case("scan_4095", "match", 1.0, 4095),
        # the whole 256 x 256 scan, in the chunks its tuner picks
        _case("scan_65536", "match", 1.0, 65536, chunk=32768),
        # a scan with FP32 operands, the binding's default precision
        _case("scan_8190_fp32", "match", 1.0, 8190, "fp32"),
        # the finest grid: 3,486 axes
        _case("halfdeg_16000", "match", 0.5, 16000, peaks="poisson"),
        # a sample of two phases: every phase's best score and the phase decision
        _case("phases_8192", "match", 2.0, 8192, "fp16", 75, 0.02, 180, "threshold",
              phases="Au+Mg", step2=1.0),
        # coarse match and continuous refinement from the match and its runner-up
        _case("refined_16384", "refined", 3.0, 16384, "bf16"),
        # score and gradient with respect to the orientation, for a caller's own optimiser
        _case("score_4000", "score", 3.0, 4000, "fp32", strain=False),
        # up to three orientations of overlapping grains
        _case("multi_2000", "multi", 1.0, 2000, peaks="overlap"),
        # the polar images' spectra for a caller's own correlation
        _case("spectra_1000", "spectra", 2.0, 1000, "fp32"),
        # the 1-degree plan of a crystal
        _case("plan_1deg", "plan", 1.0, 0),
    ]


# (shells, dq, bins): the configurations of the tests and workloads and sizes between them
GEOMETRIES = ((150, 0.01, 360), (150, 0.01, 360), (75, 0.02, 180), (40, 0.0375, 72),
              (200, 0.0075, 72), (100, 0.015, 240), (117, 0.0125, 300))


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("match",) * 6 + ("refined", "score", "multi", "bounds", "spectra", "plan"))
    shells, dq, phi = rng.choice(GEOMETRIES)
    precision = rng.choice(("fp16", "fp16", "fp16", "bf16", "fp32", "fp8"))
    if precision == "fp8" and op != "match":
        precision = "fp16"
    step = round(rng.uniform(0.8, 4.0), 2)
    c = {"op": op, "phases": "Au", "step": step, "shells": shells, "dq": dq, "phi": phi,
         "precision": precision, "patterns": 0,
         "peaks": rng.choice(("uniform", "poisson", "threshold"))}
    if op == "match":
        c["patterns"] = _between(rng, 1, 8000 if precision == "fp32" else 40000)
        if precision == "fp8":
            c["rescore_top"] = 8             # E4M3 bounds are used with top-8 rescoring
        elif c["patterns"] <= 6000 and rng.random() < 0.3:
            c.update(phases="Au+Mg", step2=round(rng.uniform(1.0, 3.0), 2), peaks="threshold")
    elif op == "refined":
        c.update(patterns=_between(rng, 16, 16000), step=round(rng.uniform(2.0, 4.0), 2))
    elif op == "score":
        c.update(patterns=_between(rng, 8, 30000), strain=rng.random() < 0.5)
    elif op == "multi":
        c.update(patterns=_between(rng, 8, 4000), peaks="overlap")
    elif op == "bounds":
        c["patterns"] = _between(rng, 8, 4000)
    elif op == "spectra":
        c["patterns"] = _between(rng, 8, 2000)
    return c


# ------------------------------------------------------------------------------- inputs


def _crystal(phase, seed=None):
    """The package's crystal; with a seed, one of a slightly other lattice (an alloy, a
    measured lattice constant)."""
    a = 1.0 if seed is None else 1.0 + 0.02 * (np.random.default_rng(seed).random() - 0.5)
    if phase == "Au":
        return acom.au_crystal(4.08 * a), acom.cubic_triangle()
    return acom.mg_crystal(3.21 * a, 5.21 * a), acom.hexagonal_triangle()


def _phases(case):
    out = [("Au", case["step"])]
    if case["phases"] == "Au+Mg":
        out.append(("Mg", case["step2"]))
    return out


def _make_plan(case, phase, step, seed=None):
    crystal, (tri, area) = _crystal(phase, seed)
    return acom.Plan(crystal, tri, area, step, case["shells"], case["dq"], case["phi"],
                     delta=DELTA, lam=LAM, q_max=QMAX, sigma_exc=SIGMA,
                     precision=PREC[case["precision"]])


def _reflections(crystal):
    """FP64 (g [G][3], |F| [G]) of every reflection 0 < |g| < q_max."""
    recip = np.linalg.inv(crystal.lattice).T
    n = [int(QMAX * np.linalg.norm(v)) for v in crystal.lattice]
    hkl = np.stack(np.meshgrid(*(np.arange(-k, k + 1) for k in n), indexing="ij"), -1).reshape(-1, 3)
    g = hkl @ recip
    q = np.linalg.norm(g, axis=1)
    keep = (q > 0) & (q < QMAX)
    hkl, g, q = hkl[keep], g[keep], q[keep]
    f = crystal.ff_A * np.exp(-crystal.ff_B * (q * q)[:, None])
    F = np.abs((f * np.exp(-2j * np.pi * (hkl @ crystal.frac_pos.T))).sum(1))
    on = F >= 1e-9 * F.max()
    return g[on], F[on]


def _rotations(gen, n):
    q = torch.randn(n, 4, generator=gen, device="cuda", dtype=torch.float64)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)],
                       1).reshape(n, 3, 3)


def _spots(phase, m):
    """Spots of the orientations m [n][3][3] (crystal = m sample), strongest first: x, y, I."""
    g, F = (torch.from_numpy(v).cuda() for v in _reflections(_crystal(phase)[0]))
    lab = torch.einsum("gi,nij->ngj", g, m)
    s = 1 / LAM - torch.sqrt(lab[..., 0] ** 2 + lab[..., 1] ** 2 + (lab[..., 2] - 1 / LAM) ** 2)
    I, order = torch.sort(F * F * torch.exp(-s * s / (2 * SIGMA ** 2)), dim=1, descending=True)
    return lab[..., 0].gather(1, order), lab[..., 1].gather(1, order), I


def _counts_by_threshold(I, most=40):
    return (I > 1e-3 * I[:, :1]).sum(1).clamp(max=most)


def _batch(case, seed):
    """Peak lists (row_ptr, qx, qy, I) on the GPU and the true orientations."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B = case["patterns"]
    if case["peaks"] in ("uniform", "poisson"):
        # a scan over a Voronoi map of grains: neighbouring patterns share an orientation, each
        # keeps its strongest peaks
        side = max(1, math.isqrt(B))
        grains = max(1, B // 328)
        at = torch.arange(B, device="cuda")
        pix = torch.stack([(at % side).double(), (at // side).double()], 1)
        centres = torch.rand(grains, 2, generator=gen, device="cuda", dtype=torch.float64) * \
            torch.tensor([side, B / side], device="cuda", dtype=torch.float64)
        lab = torch.cdist(pix, centres).argmin(1)
        R = _rotations(gen, grains)
        x, y, I = _spots("Au", R)
        if case["peaks"] == "uniform":
            n = torch.randint(10, 61, (B,), generator=gen, device="cuda")
        else:
            n = torch.poisson(torch.full((B,), 30.0, device="cuda"), generator=gen).long().clamp(5, 80)
        truth = R[lab]
    elif case["peaks"] == "threshold":
        # independent orientations, the peaks above a thousandth of the strongest
        truth = _rotations(gen, B)
        x, y, I = _spots("Au", truth)
        n = _counts_by_threshold(I)
        if case["phases"] == "Au+Mg":
            other = _spots("Mg", truth)
            wide = max(x.shape[1], other[0].shape[1])
            is_mg = torch.rand(B, generator=gen, device="cuda") < 0.5
            n = torch.where(is_mg, _counts_by_threshold(other[2]), n)
            x, y, I = (torch.where(is_mg[:, None], torch.nn.functional.pad(v, (0, wide - v.shape[1])),
                                   torch.nn.functional.pad(u, (0, wide - u.shape[1])))
                       for u, v in zip((x, y, I), other))
        lab = torch.arange(B, device="cuda")
    else:
        # two overlapping grains, the second weaker: 30 peaks of each
        truth = _rotations(gen, B)
        one, two = _spots("Au", truth), _spots("Au", _rotations(gen, B))
        x, y, I = (torch.cat([u[:, :30], v[:, :30]], 1) for u, v in zip(one, two))
        I[:, 30:] *= 0.6
        n = torch.full((B,), 60, device="cuda")
        lab = torch.arange(B, device="cuda")
    row_ptr = torch.zeros(B + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = n.cumsum(0)
    nnz = int(row_ptr[-1])
    pat = torch.repeat_interleave(torch.arange(B, device="cuda"), n)
    k = torch.arange(nnz, device="cuda") - row_ptr[pat]
    src = lab[pat] * x.shape[1] + k
    noise = torch.randn(3, nnz, generator=gen, device="cuda", dtype=torch.float64)
    qx = (x.reshape(-1)[src] + 0.005 * noise[0]).float()
    qy = (y.reshape(-1)[src] + 0.005 * noise[1]).float()
    inten = (I.reshape(-1)[src] * torch.exp(0.1 * noise[2])).float()
    return (row_ptr, qx, qy, inten), truth


def _score_inputs(case, seed, truth):
    """Starting orientations a degree or so from the truth, rotation vectors, strains and the
    weights of a caller's loss."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    B = case["patterns"]
    r = (0.02 * torch.randn(B, 3, generator=gen, device="cuda")).requires_grad_()
    e = (0.005 * torch.randn(B, 6, generator=gen, device="cuda")).requires_grad_() \
        if case["strain"] else None
    weight = torch.rand(B, generator=gen, device="cuda") + 0.5
    return truth.float().contiguous(), r, e, weight


def prepare(case, seed):
    s = {"case": case, "seed": seed}
    if case["op"] == "plan":
        return s
    plans = [_make_plan(case, phase, step) for phase, step in _phases(case)]
    s["plan"] = plans[0] if len(plans) == 1 else acom.Plan.concat(plans)
    s["peaks"], truth = _batch(case, seed)
    if case["op"] == "score":
        s["orient"], s["r"], s["e"], s["weight"] = _score_inputs(case, seed, truth)
    return s


def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "plan":
        plan = _make_plan(case, "Au", case["step"], s["seed"])
        out = {"spectra": plan.spectra(), "zone_axes": plan.zone_axes(),
               "reflections": plan.info["n_reflections"]}
        plan.close()
        return out
    plan, peaks = s["plan"], s["peaks"]
    if op == "match":
        return plan.match(*peaks, chunk=case.get("chunk", 0), rescore_top=case.get("rescore_top", 0),
                          phase_scores=case["phases"] == "Au+Mg")
    if op == "refined":
        found = plan.match(*peaks, runner=True)
        orient, score, start = plan.refine(*peaks, found["orient"].clone(),
                                           orient_alt=found["runner_orient"])
        return {"match": found, "orient": orient, "score": score, "start": start}
    if op == "score":
        r, e = s["r"], s["e"]
        r.grad = None
        if e is None:
            S = acom.kinematical_score(r, plan, peaks, s["orient"])
        else:
            e.grad = None
            S = acom.kinematical_score_strain(r, e, plan, peaks, s["orient"])
        (S * s["weight"]).sum().backward()
        return {"score": S.detach(), "grad_r": r.grad, "grad_e": None if e is None else e.grad}
    if op == "multi":
        return plan.match_multi(*peaks, n_matches=3)
    if op == "bounds":
        return plan.bounds(*peaks)
    return plan.polar_spectra(*peaks)


# -------------------------------------------------------------------- work and exact values


def _axes_count(case):
    z = 0
    for phase, step in _phases(case):
        area = _crystal(phase)[1][1]
        n = max(1, math.floor(math.sqrt(2 * area) / math.radians(step)))
        z += (n + 1) * (n + 2) // 2
    return z


def work(case):
    """Each input read once, each output written once; the contraction's 8 flops per (axis,
    shell, frequency), the transforms' 2.5 N log2 N per shell row."""
    B, S, N, F = case["patterns"], case["shells"], case["phi"], case["phi"] // 2 + 1
    Z = _axes_count(case)
    peaks = B * (8 + 12 * PEAKS[case["peaks"]])
    plan = Z * S * F * OPERAND[case["precision"]]
    raster = 2.5 * N * math.log2(N) * S
    contraction = 8.0 * Z * S * F
    op = case["op"]
    if op == "plan":
        return {"bytes": Z * S * F * 8, "flops": Z * raster}
    if op == "score":
        # 13 flops per (reflection near the Ewald sphere, peak) pair; 41 such reflections
        return {"bytes": peaks + B * (36 + 12 + 16 + (48 if case["strain"] else 0)),
                "flops": B * 41.0 * PEAKS[case["peaks"]] * 13}
    if op == "spectra":
        return {"bytes": peaks + B * (S * F * 8 + 4), "flops": B * raster}
    if op == "bounds":
        return {"bytes": peaks + plan + B * Z * 4, "flops": B * (raster + contraction)}
    times = 3 if op == "multi" else 1
    w = {"bytes": times * (plan + B * 57) + peaks, "flops": times * B * (raster + contraction)}
    if op == "refined":
        w["bytes"] += peaks + B * 41
        w["flops"] += B * 4 * 21 * 41.0 * PEAKS[case["peaks"]] * 13
    return w


def _grid64(tri, area, step):
    v = [np.array(p, float) / np.linalg.norm(p) for p in tri]

    def slerp(a, b, t):
        om = math.acos(max(-1.0, min(1.0, float(a @ b))))
        if om < 1e-15:
            return a
        return (math.sin((1 - t) * om) * a + math.sin(t * om) * b) / math.sin(om)

    n = max(1, math.floor(math.sqrt(2 * area) / math.radians(step)))
    pts = [v[0]]
    for i in range(1, n + 1):
        a, b = slerp(v[0], v[1], i / n), slerp(v[0], v[2], i / n)
        pts += [slerp(a, b, j / i) for j in range(i + 1)]
    pts = np.array(pts)
    return pts / np.linalg.norm(pts, axis=1, keepdims=True)


def _images64(case, r, gam, w, e2, item, items, shell_power):
    """Sum of tents per item: [items][S][N] from the peaks of each item (sorted by item)."""
    S, N = case["shells"], case["phi"]
    q = (torch.arange(S, device="cuda", dtype=torch.float64) + 1) * case["dq"]
    phi = 2 * math.pi * torch.arange(N, device="cuda", dtype=torch.float64) / N
    out = torch.zeros(items, S, N, device="cuda", dtype=torch.float64)
    rows = q if shell_power else torch.ones_like(q)
    for a in range(0, len(r), 1024):
        d = phi[None] - gam[a:a + 1024, None]
        d = torch.remainder(d + math.pi, 2 * math.pi) - math.pi
        radial = (r[a:a + 1024, None] - q) ** 2 + e2[a:a + 1024, None]
        t = 1 - torch.sqrt(radial[:, :, None] + d[:, None] ** 2 * (q * q)[None, :, None]) / DELTA
        out.index_add_(0, item[a:a + 1024], t.clamp_(min=0) * w[a:a + 1024, None, None])
    return out * rows[None, :, None]


def _plan64(case, seed=None):
    """(spectra [Z][S][F] complex128 of the normalised plan, zone axes of all phases)."""
    spectra, axes = [], []
    for phase, step in _phases(case):
        crystal, (tri, area) = _crystal(phase, seed)
        g, F = (torch.from_numpy(v).cuda() for v in _reflections(crystal))
        za = torch.from_numpy(_grid64(tri, area, step)).cuda()
        for a in range(0, len(za), 256):
            z = za[a:a + 256]
            th, ph = torch.acos(z[:, 2].clamp(-1, 1)), torch.atan2(-z[:, 0], z[:, 1])
            c1, s1, c2, s2, o = ph.cos(), ph.sin(), th.cos(), th.sin(), torch.zeros_like(th)
            R = torch.stack([c1, -s1 * c2, -s1 * s2, s1, c1 * c2, c1 * s2, o, -s2, c2], 1).reshape(-1, 3, 3)
            p = torch.einsum("gi,zij->zgj", g, R)
            kz = -1 / LAM
            s = -(p[..., 0] ** 2 + p[..., 1] ** 2 + p[..., 2] * (2 * kz + p[..., 2])) / \
                (2 * torch.sqrt(p[..., 0] ** 2 + p[..., 1] ** 2 + (kz + p[..., 2]) ** 2))
            near = s.abs() < DELTA
            item = near.nonzero()[:, 0]
            P = _images64(case, p[..., :2].norm(dim=2)[near], torch.atan2(p[..., 1], p[..., 0])[near],
                          F.expand(len(z), -1)[near], (s * s)[near], item, len(z), True)
            norm = P.flatten(1).norm(dim=1)
            P *= torch.where(norm > 0, 1 / norm, torch.zeros_like(norm))[:, None, None]
            spectra.append(torch.fft.rfft(P))
        axes.append(za)
    return torch.cat(spectra), torch.cat(axes)


def _patterns64(case, peaks, a, b):
    """Spectra [n][S][F] and norms of the polar images of patterns a .. b - 1."""
    row_ptr, qx, qy, I = peaks
    lo, hi = int(row_ptr[a]), int(row_ptr[b])
    x, y, i = qx[lo:hi].double(), qy[lo:hi].double(), I[lo:hi].double()
    item = torch.repeat_interleave(torch.arange(b - a, device="cuda"), row_ptr[a + 1:b + 1] - row_ptr[a:b])
    r = torch.sqrt(x * x + y * y)
    X = _images64(case, r, torch.atan2(y, x), r * i.clamp(min=0).sqrt(), torch.zeros_like(r), item,
                  b - a, False)
    return torch.fft.rfft(X), X.flatten(1).norm(dim=1)


def _correlations64(case, peaks, bound):
    """Per pattern and phase the best correlation, or per axis the spectral bound, and ||X||."""
    P, _ = _plan64(case)
    N, F = case["phi"], case["phi"] // 2 + 1
    sizes = [len(_grid64(*_crystal(phase)[1], step)) for phase, step in _phases(case)]
    w = torch.full((F, 1, 1), 2.0 / N, device="cuda", dtype=torch.float64)
    w[0] = w[-1] = 1.0 / N
    Pf = P.permute(2, 0, 1).conj().resolve_conj().contiguous()
    del P
    best, norms = [], []
    n = max(1, min(128, (1 << 27) // (Pf.shape[1] * N)))
    for a in range(0, case["patterns"], n):
        X, norm = _patterns64(case, peaks, a, min(a + n, case["patterns"]))
        Xf = X.permute(2, 1, 0).contiguous()
        c, m = Pf @ Xf, Pf @ Xf.conj()
        norms.append(norm)
        if bound:
            best.append((w * torch.maximum(c.abs(), m.abs())).sum(0).T.contiguous())
        else:
            top = torch.maximum(*(torch.fft.irfft(v, n=N, dim=0).amax(0) for v in (c, m)))
            best.append(torch.stack([t.amax(0) for t in top.split(sizes)], 1))
    return torch.cat(best), torch.cat(norms)


def _scores64(case, peaks, orient, r, e):
    """Kinematical score at Exp(r) m^T, strained by e, from its definition (rho = 0.03)."""
    row_ptr, qx, qy, I = peaks
    g, F = (torch.from_numpy(v).cuda() for v in _reflections(_crystal("Au")[0]))
    amp = g.norm(dim=1) * F
    S = []
    for a in range(0, case["patterns"], 256):
        b = min(a + 256, case["patterns"])
        cnt = row_ptr[a + 1:b + 1] - row_ptr[a:b]
        k = torch.arange(int(cnt.max()), device="cuda")
        on = k < cnt[:, None]
        at = (row_ptr[a:b, None] + k).clamp(max=len(qx) - 1)
        x, y = qx[at].double(), qy[at].double()
        pw = torch.where(on, torch.sqrt(x * x + y * y) * I[at].double().clamp(min=0).sqrt(), 0.0)
        v = r[a:b]
        o = torch.zeros_like(v[:, 0])
        K = torch.stack([o, -v[:, 2], v[:, 1], v[:, 2], o, -v[:, 0], -v[:, 1], v[:, 0], o], 1).reshape(-1, 3, 3)
        R = torch.linalg.matrix_exp(K) @ orient[a:b].transpose(1, 2)
        gs = g.expand(b - a, -1, -1)
        if e is not None:
            t = e[a:b]
            E = torch.stack([t[:, 0], t[:, 1], t[:, 2], t[:, 1], t[:, 3], t[:, 4], t[:, 2], t[:, 4],
                             t[:, 5]], 1).reshape(-1, 3, 3)
            gs = gs + gs @ E
        lab = gs @ R.transpose(1, 2)
        kz = lab[..., 2] - 1 / LAM
        nk = torch.sqrt(lab[..., 0] ** 2 + lab[..., 1] ** 2 + kz ** 2)
        s = -((lab ** 2).sum(2) - 2 * lab[..., 2] / LAM) / (2 * nk)
        bg = amp * torch.exp(-s * s / (4 * SIGMA ** 2))
        d2 = (x[:, :, None] - lab[:, None, :, 0]) ** 2 + (y[:, :, None] - lab[:, None, :, 1]) ** 2
        C = (pw[:, :, None] * bg[:, None] * torch.exp(-d2 / (2 * 0.03 ** 2))).sum((1, 2))
        S.append(C / bg.norm(dim=1))
    return torch.cat(S)


def exact(case, seed):
    op = case["op"]
    if op == "plan":
        P, za = _plan64(case, seed)
        return {"spectra": torch.view_as_real(P), "zone_axes": za, "reflections": None}
    peaks, truth = _batch(case, seed)
    if op == "score":
        orient, r, e, weight = _score_inputs(case, seed, truth)
        r = r.detach().double().requires_grad_()
        e = None if e is None else e.detach().double().requires_grad_()
        S = _scores64(case, peaks, orient.double(), r, e)
        (S * weight.double()).sum().backward()
        return {"score": S.detach(), "grad_r": r.grad, "grad_e": None if e is None else e.grad}
    if op == "spectra":
        X, norm = _patterns64(case, peaks, 0, case["patterns"])
        return torch.view_as_real(X), norm
    if 16.0 * _axes_count(case) * case["shells"] * case["phi"] / 2 * case["patterns"] > 4e12:
        return None                              # about ten seconds of FP64 products
    best, norm = _correlations64(case, peaks, op == "bounds")
    if op == "bounds":
        return best
    score = best.amax(1)
    out = {"score": score, "score_cos": torch.where(norm > 0, score / norm, torch.zeros_like(score))}
    if case["phases"] == "Au+Mg" and case.get("rescore_top", 0) == 0:
        out["phase_score"] = best
    if op == "refined":
        return {"match": out}
    return [out] if op == "multi" else out
