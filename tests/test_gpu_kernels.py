"""Kernels at the sizes where their tilings and splits can go wrong (edges of tiles,
remainders, one pattern, batches that leave SMs idle), against FP64 values of the same
spectra."""

import math

import numpy as np
import pytest

import synth
from gpu_common import LAM, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()


def au_plan(step, shells, dq, n_phi, precision=0):
    from paper_2111_00171_gb300 import acom
    tri, area = acom.cubic_triangle()
    return acom.Plan(acom.au_crystal(), tri, area, step, shells, dq, n_phi, lam=LAM,
                     precision=precision)


def bounds64(plan, peaks):
    """FP64 spectral bounds of the plan's and the patterns' FP32 spectra, and the sum
    (1/N) sum_f w_f max_z ||P_zf|| ||X_bf|| that scales their rounding."""
    import torch
    P = torch.view_as_complex(plan.spectra()).to(torch.complex128)           # [Z][S][F]
    X = torch.view_as_complex(plan.polar_spectra(*peaks)[0]).to(torch.complex128)
    N, F = plan.info["n_phi"], plan.info["n_freq"]
    w = torch.full((F,), 2.0 / N, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 1.0 / N
    c = torch.einsum("zsf,bsf->bzf", P.conj(), X).abs()
    m = torch.einsum("zsf,bsf->bzf", P.conj(), X.conj()).abs()
    scale = (w * P.norm(dim=1).amax(0) * X.norm(dim=1)).sum(1)               # [B]
    return (torch.maximum(c, m) * w).sum(2), scale


# one pattern; a tile's edge and one past it; more tiles than the GPU holds CTAs of
# (on the tensor cores: one K tile, two, a second one not full; else on the CUDA cores)
@pytest.mark.parametrize("geometry", [(3.0, 75, 0.02, 180), (3.0, 150, 0.01, 360),
                                      (4.0, 117, 0.0125, 300), (6.0, 200, 0.0075, 72),
                                      (2.0, 33, 0.045, 84)], ids=str)
@pytest.mark.parametrize("patterns", [1, 63, 65, 1300])
def test_fp32_bounds_at_tile_edges(geometry, patterns):
    plan = au_plan(*geometry)
    peaks = to_dev(synth.random_patterns(31 + patterns, n_patterns=patterns))
    got = plan.bounds(*peaks).double()
    want, scale = bounds64(plan, peaks)
    # dot products of the shells, four products, root and the sum over frequencies
    S, F = math.ceil(geometry[1] / 32) * 32, geometry[3] // 2 + 1
    tol = (3 * (S + 2) + 2 * F) * 2.0 ** -24 * scale
    assert ((got - want).abs() <= tol[:, None]).all()
    plan.close()


# one pattern and the edges of 64- and 128-pattern tiles; one to three K stages; a last
# wave split over the frequencies (20,000 patterns: 157 tiles), and a batch of few tiles
@pytest.mark.parametrize("geometry,patterns", [
    ((3.0, 150, 0.01, 360), 1), ((3.0, 150, 0.01, 360), 64), ((2.0, 75, 0.02, 180), 65),
    ((2.0, 75, 0.02, 180), 128), ((6.0, 200, 0.0075, 72), 129), ((6.0, 400, 0.00375, 72), 193),
    ((6.0, 40, 0.0375, 72), 20000)], ids=str)
def test_tensor_core_bounds_at_tile_edges(geometry, patterns):
    plan = au_plan(*geometry, precision=1)
    peaks = to_dev(synth.random_patterns(77, n_patterns=patterns))
    got = plan.bounds(*peaks).double()
    want, scale = bounds64(plan, peaks)
    # BF16 operands: 2^-7 a product, sqrt(2) a side; FP32 accumulation charged 8-fold
    S, F = math.ceil(geometry[1] / 32) * 32, geometry[3] // 2 + 1
    tol = (2.0 ** -6 + (3 * (S + 2) + 2 * F) * 2.0 ** -21) * scale
    assert ((got - want).abs() <= tol[:, None]).all()
    plan.close()


def test_search_with_more_pending_axes_than_the_sorted_list():
    """E4M3 bounds leave about a third of 3,486 axes pending after the first batch, more
    than the search sorts at a time: the certified winners are the FP32 plan's."""
    import torch
    peaks = to_dev(synth.random_patterns(905, n_patterns=24))
    got = {}
    for precision in (0, 3):
        plan = au_plan(0.5, 150, 0.01, 360, precision=precision)
        r = plan.match(*peaks)
        got[precision] = r["score"].cpu().numpy()
        evaluated = plan.get_info()["last_evaluated"] / 24
        plan.close()
    assert evaluated > 512          # or the sorted list was never exceeded
    # the same axis scored in batches of another size: another split of the shell sums
    np.testing.assert_allclose(got[3], got[0], rtol=2e-6)


def test_refined_axis_with_more_neighbours_than_are_handed_on():
    """A grid whose step is so coarse against its region that an axis has more than 32
    neighbours takes the summed hand-off: the orientation is the oracle's refinement."""
    from oracle import acom_oracle as O
    from gpu_common import au_refl
    from paper_2111_00171_gb300 import acom
    # a narrow triangle about [001] whose stated area gives it many axes within 1.5 steps
    tri = [[0, 0, 1], [0, 0.1, 1], [0.1, 0.1, 1]]
    area = 4.0 * (14 * math.radians(2.0)) ** 2 / 8.0           # n = 14 rows at 2 degrees
    scan = synth.random_patterns(8, n_patterns=12)
    plan = acom.Plan(acom.au_crystal(), tri, area, 2.0, 40, 0.0375, 72, lam=LAM)
    za = O.zone_axis_grid(*tri, 2.0, area)
    assert (za @ za[60] >= math.cos(math.radians(3.0))).sum() > 32
    oplan = O.orientation_plan(au_refl(), za, O.PlanParams(40, 0.0375, 72, 0.08, lam=LAM))
    r = plan.match(*to_dev(scan))
    m = r["orient"].cpu().numpy()
    for b in range(scan.n_patterns):
        mt = O.match_pattern(oplan, *scan.pattern(b))
        if (int(r["za_idx"][b]), int(r["phi3_bin"][b]), int(r["mirror"][b])) != (mt.za, mt.k, mt.mirror):
            continue                                            # a tie resolved the other way
        # FP32 scores weight the mean: 1e-5 relative, over a neighbourhood of 3 degrees
        np.testing.assert_allclose(m[b], O.refine(mt, za, 2.0).m, atol=1e-4)
    plan.close()


def test_orientation_from_more_neighbours_than_are_handed_on():
    """Patterns along axes of such a grid, whose winners' neighbours are counted: at least
    half of them have the oracle's winner (a tie may be resolved the other way), each with
    more than 32 neighbours, and then its orientation."""
    from oracle import acom_oracle as O
    from gpu_common import au_refl
    from paper_2111_00171_gb300 import acom
    tri = [[0, 0, 1], [0, 0.1, 1], [0.1, 0.1, 1]]
    area = 4.0 * (14 * math.radians(2.0)) ** 2 / 8.0
    plan = acom.Plan(acom.au_crystal(), tri, area, 2.0, 40, 0.0375, 72, lam=LAM)
    za = O.zone_axis_grid(*tri, 2.0, area)
    oplan = O.orientation_plan(au_refl(), za, O.PlanParams(40, 0.0375, 72, 0.08, lam=LAM))
    rng = np.random.default_rng(16)
    spec = synth.au_fcc()
    g, F2 = synth.reflection_table(spec, 1.5)
    lists, truth = [], []
    for i in rng.choice(len(za), 12, replace=False):
        m = np.linalg.qr(np.column_stack([za[i], rng.normal(size=(3, 2))]))[0]
        m = m[:, [1, 2, 0]] * np.sign(m[:, 0] @ za[i])        # the beam along the axis
        m[:, 0] *= np.sign(np.linalg.det(m))
        lists.append(synth._sorted_list(g, F2, m, LAM, 0.02))
        truth.append(m)
    scan = synth.Scan(*synth._assemble(lists, np.full(12, 30), rng, 0.005, 0.1), np.array(truth),
                      np.zeros(12, np.int32), (spec,), "axes of a narrow grid")
    r = plan.match(*to_dev(scan))
    m = r["orient"].cpu().numpy()
    same = 0
    for b in range(scan.n_patterns):
        mt = O.match_pattern(oplan, *scan.pattern(b))
        if (int(r["za_idx"][b]), int(r["phi3_bin"][b]), int(r["mirror"][b])) != (mt.za, mt.k, mt.mirror):
            continue
        same += 1
        assert (za @ za[mt.za] >= math.cos(math.radians(3.0))).sum() > 32
        # FP32 scores weight the mean: 1e-5 relative, over a neighbourhood of 3 degrees
        np.testing.assert_allclose(m[b], O.refine(mt, za, 2.0).m, atol=1e-4)
    assert same >= 6
    plan.close()


@pytest.mark.parametrize("precision", [0, 2], ids=["fp32", "fp16"])
def test_bins_with_a_prime_factor_above_five(precision):
    """84 = 4 * 3 * 7 bins take the direct transform: the certified match finds the
    oracle's score (the exact evaluation reads the shells that the raster records)."""
    from oracle import acom_oracle as O
    from gpu_common import au_refl
    v0, v1, v2, area = O.cubic_triangle()
    za = O.zone_axis_grid(v0, v1, v2, 4.0, area)
    oplan = O.orientation_plan(au_refl(), za, O.PlanParams(33, 0.045, 84, 0.08, lam=LAM))
    plan = au_plan(4.0, 33, 0.045, 84, precision=precision)
    scan = synth.random_patterns(84, n_patterns=40)
    r = plan.match(*to_dev(scan))
    for b in range(scan.n_patterns):
        assert math.isclose(float(r["score"][b]), O.match_pattern(oplan, *scan.pattern(b)).score,
                            rel_tol=1e-4), b
    plan.close()


@pytest.mark.parametrize("geometry", [(6.0, 200, 0.0075, 72), (3.0, 150, 0.01, 360),
                                      (4.0, 33, 0.045, 84), (3.0, 117, 0.0125, 300)], ids=str)
@pytest.mark.parametrize("precision", [0, 1, 2, 3], ids=["fp32", "bf16", "fp16", "fp8"])
def test_plan_layouts(geometry, precision):
    """The plan's spectra are normalised slices (Parseval over shells and bins), and the
    polar spectra's norms agree with their sums, at frequency and shell counts that are
    no multiples of the tiles."""
    import torch
    plan = au_plan(*geometry, precision=precision)
    F, N = plan.info["n_freq"], plan.info["n_phi"]
    w = torch.full((F,), 2.0 / N, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 1.0 / N
    norm = lambda x: (x.double().square().sum((1, 3)) * w).sum(1)
    # FP32 sums of F terms and the rounding of the scale
    assert ((norm(plan.spectra()) - 1).abs() < 2 * F * 2.0 ** -24).all()
    peaks = to_dev(synth.random_patterns(6, n_patterns=37))
    X, xn = plan.polar_spectra(*peaks)
    assert ((norm(X).sqrt() - xn).abs() < 2 * F * 2.0 ** -24 * xn).all()
    plan.close()


@pytest.mark.parametrize("geometry", [(3.0, 75, 0.02, 180), (3.0, 150, 0.01, 360),
                                      (4.0, 117, 0.0125, 300)], ids=str)
def test_fp16_pairs_are_no_less_accurate_than_fp32(geometry):
    """The FP32 contraction on the tensor cores (FP16 pairs, bounds()) is no further from
    FP64 than the one on the CUDA cores (bounds_static())."""
    import torch
    plan = au_plan(*geometry)
    peaks = to_dev(synth.random_patterns(123, n_patterns=200))
    want, _ = bounds64(plan, peaks)
    pairs = plan.bounds(*peaks)
    cores = plan.bounds_static(*peaks, out=torch.empty_like(pairs))
    off = lambda u: float((u.double() - want).norm())
    assert off(pairs) <= off(cores)
    plan.close()


# one tile, cut into a group per frequency or two; 168 tiles, the last 16 in groups of 21
# frequencies and the others whole, each in four sums
@pytest.mark.parametrize("geometry,patterns", [
    ((4.0, 75, 0.02, 180), 8), ((4.0, 75, 0.02, 180), 120), ((4.0, 100, 0.015, 240), 120),
    ((4.0, 117, 0.0125, 300), 120), ((1.0, 150, 0.01, 360), 2600)], ids=str)
def test_fp16_pairs_in_few_and_in_many_tiles(geometry, patterns):
    """However the batch cuts the frequencies into groups, the FP16 pairs' bounds are no
    further from FP64 than those of the CUDA cores, which add all frequencies in turn."""
    import torch
    plan = au_plan(*geometry)
    scan = synth.random_patterns(145, n_patterns=patterns)
    peaks = to_dev(scan)
    pairs = plan.bounds(*peaks)
    cores = plan.bounds_static(*peaks, out=torch.empty_like(pairs))
    # patterns of the first and of the last tiles
    idx = np.r_[0:min(patterns, 128), max(128, patterns - 168):patterns]
    want, _ = bounds64(plan, to_dev(scan.subset(idx)))
    for part in (slice(0, 128), slice(128, None)):
        off = lambda u: float((u[torch.from_numpy(idx).cuda()].double() - want)[part].norm())
        assert off(pairs) <= off(cores)
    plan.close()


@pytest.mark.parametrize("geometry", [(3.0, 33, 0.045, 180), (3.0, 60, 0.025, 180),
                                      (3.0, 75, 0.02, 180)], ids=str)
def test_margin_of_the_fp16_pairs(geometry):
    """The search's rounding margin covers what the FP16 pairs can be off by: 220 + 2 F units
    of 2^-24 (operands 17, accumulation 194, magnitude 6; the sum over frequencies).  An
    axis that was not evaluated reports its bound plus the margin."""
    import torch
    plan = au_plan(*geometry)
    peaks = to_dev(synth.random_patterns(14, n_patterns=40))
    U = plan.bounds(*peaks).double()
    top = plan.match(*peaks, za_scores=True, refine=False)["za_scores"].double()
    margin = top - U * (1.0 + 1e-5)
    margin[margin <= 0] = float("nan")                # evaluated: the exact score
    got = margin.nanmedian(dim=1).values              # (sums in FP32 round by 1 % of it)
    _, scale = bounds64(plan, peaks)
    need = (220 + 2 * plan.info["n_freq"]) * 2.0 ** -24 * scale
    assert (got >= 0.99 * need).all()
    plan.close()


def test_fp16_pairs_of_values_far_below_the_largest():
    """A peak that no axis' rows reach but 10^6 times as heavy as the others takes the scale
    of the pairs, so that the others' low halves are FP16 subnormals: their bounds are off
    by no more than those halves' spacing allows, and the match finds the winners that the
    patterns have without that peak."""
    import torch
    plan = au_plan(3.0, 150, 0.01, 360)
    scan = synth.random_patterns(15, n_patterns=24)
    n = np.diff(scan.row_ptr)
    at = scan.row_ptr[:-1]                            # the heavy peak before each pattern's own
    heavy = synth.Scan(scan.row_ptr + np.arange(25), np.insert(scan.qx, at, 0.1).astype(np.float32),
                       np.insert(scan.qy, at, 0.0).astype(np.float32),
                       np.insert(scan.I, at, scan.I.max() * 1e12).astype(np.float32),
                       scan.truth, scan.phase, scan.crystals, "a heavy peak")
    assert (np.diff(heavy.row_ptr) == n + 1).all() and plan.info["k0"] * 0.01 > 0.1 + 0.08
    peaks = to_dev(heavy)
    want, _ = bounds64(plan, peaks)
    P = torch.view_as_complex(plan.spectra()).to(torch.complex128)[:, plan.info["k0"]:]
    N, F = plan.info["n_phi"], plan.info["n_freq"]
    w = torch.full((F,), 2.0 / N, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 1.0 / N
    # 2^-25 of a scaled value: the scale is above 2^13 / B, B the sum of the peaks' weights
    # times the bins that their tents cover, all 360 of them at most
    q = np.hypot(heavy.qx.astype(float), heavy.qy)
    B = np.add.reduceat(q * np.sqrt(heavy.I.astype(float)) * 360, heavy.row_ptr[:-1])
    off = torch.from_numpy(B).cuda() * 2.0 ** -38
    # four real products, 118 shells
    tol = 4 * math.sqrt(118.0) * off[:, None] * (w * P.norm(dim=1)).sum(1)[None]
    tol = tol + 2.0 ** -17 * want
    assert ((plan.bounds(*peaks).double() - want).abs() <= tol).all()
    got, alone = plan.match(*peaks), plan.match(*to_dev(scan))
    assert ((got["score"] - alone["score"]).abs() <= 2e-6 * alone["score"]).all()
    plan.close()


@pytest.mark.parametrize("precision", [0, 2], ids=["fp32", "fp16"])
def test_weights_near_the_top_of_fp32(precision):
    """Peak weights up to 1e36 (omega 2, so a weight is its intensity times q): the FP16
    scale covers FP32's range, and the winners and scores are those of the same pattern
    with weights near 1, but for the scale."""
    import torch
    from paper_2111_00171_gb300 import acom
    tri, area = acom.cubic_triangle()
    plan = acom.Plan(acom.au_crystal(), tri, area, 3.0, 75, 0.02, 180, lam=LAM, omega=2.0,
                     precision=precision)
    rp, qx, qy, I = to_dev(synth.random_patterns(12, n_patterns=20))
    I = I / I.max()
    want = plan.match(rp, qx, qy, I)["score"].double()
    up = 2.0 ** 119                                   # exact
    got = plan.match(rp, qx, qy, I * up)["score"].double() / up
    # the same axis scored in batches of another size: another split of the shell sums
    assert ((got - want).abs() <= 2e-6 * want).all()
    plan.close()


@pytest.mark.parametrize("geometry", [(6.0, 150, 0.01, 360), (6.0, 40, 0.0375, 72),
                                      (6.0, 33, 0.045, 84)], ids=str)
def test_spectra_into_an_array_that_is_not_8_byte_aligned(geometry):
    """The C calls write spectra to any float address: the same values one float further
    on, and nothing on either side of them."""
    import ctypes as C
    import torch
    from paper_2111_00171_gb300 import acom
    lib = acom.load_library()
    plan = au_plan(*geometry)
    scan = to_dev(synth.random_patterns(13, n_patterns=5))
    pk = plan._csr(*scan)
    stream = torch.cuda.current_stream().cuda_stream

    def polar(ptr):
        assert lib.acom_polar_spectra(plan.handle, C.byref(pk), C.c_void_p(ptr), None,
                                      C.c_void_p(stream)) == 0

    def spectra(ptr):
        assert lib.acom_plan_get_spectra(plan.handle, C.c_void_p(ptr), C.c_void_p(stream)) == 0

    for call, want in ((polar, plan.polar_spectra(*scan)[0]), (spectra, plan.spectra())):
        buf = torch.full((want.numel() + 3,), -7.0, device="cuda")
        assert buf.data_ptr() % 8 == 0
        call(buf.data_ptr() + 4)
        torch.cuda.synchronize()
        assert torch.equal(buf[1:-2], want.reshape(-1))
        assert float(buf[0]) == -7.0 and bool((buf[-2:] == -7.0).all())
    plan.close()


@pytest.mark.parametrize("geometry", [(6.0, 150, 0.01, 360), (6.0, 75, 0.02, 180)], ids=str)
@pytest.mark.parametrize("precision", [1, 2], ids=["bf16", "fp16"])
def test_sixteen_bit_copies_with_one_and_two_staging_buffers(geometry, precision):
    """Patterns of few and of many peaks in turn in the same CTAs (a second staging
    buffer fits behind 178 peaks at 360 bins, 478 at 180): each pattern's bounds are
    those it has among patterns of its kind."""
    import torch
    rng = np.random.default_rng(5)
    counts = np.array([20, 600, 178, 179, 478, 479, 0, 1000, 3] * 120)
    rp = np.zeros(len(counts) + 1, np.int64)
    np.cumsum(counts, out=rp[1:])
    r, t = rng.uniform(0.1, 1.45, rp[-1]), rng.uniform(-np.pi, np.pi, rp[-1])
    scan = synth.Scan(rp, (r * np.cos(t)).astype(np.float32), (r * np.sin(t)).astype(np.float32),
                      rng.lognormal(0.0, 1.0, rp[-1]).astype(np.float32),
                      np.tile(np.eye(3), (len(counts), 1, 1)), np.zeros(len(counts), np.int32),
                      (synth.au_fcc(),), "few and many peaks")
    plan = au_plan(*geometry, precision=precision)
    peaks = to_dev(scan)
    want, scale = bounds64(plan, peaks)
    S, F = math.ceil(geometry[1] / 32) * 32, geometry[3] // 2 + 1
    tol = (2.0 ** -6 + (3 * (S + 2) + 2 * F) * 2.0 ** -21) * scale
    got = plan.bounds(*peaks)
    assert ((got.double() - want).abs() <= tol[:, None]).all()
    # the same terms whichever buffers the pattern's neighbours used; a batch of another
    # size may sum the frequencies in other groups, F terms in FP32
    few = np.nonzero(counts <= 178)[0]
    alone = plan.bounds(*to_dev(scan.subset(few)))
    assert ((got[torch.from_numpy(few).cuda()] - alone).abs() <= F * 2.0 ** -23 * alone).all()
    plan.close()


@pytest.mark.parametrize("sigma", [1e-6, 0.02, 0.3])
def test_kinematical_score_reflection_list(sigma):
    """The reflections that contribute are found in two steps (a bound, then the cut):
    scores and gradients at shape factors from far narrower than the rounding of an
    excitation error to wider than all reflections, for a last block that is not full,
    against FP64 autograd of the definition."""
    import torch
    from paper_2111_00171_gb300 import acom
    from oracle import acom_oracle as O
    from gpu_common import au_refl
    tri, area = acom.cubic_triangle()
    plan = acom.Plan(acom.au_crystal(), tri, area, 6.0, 40, 0.0375, 72, lam=LAM, sigma_exc=sigma)
    scan = synth.random_patterns(21, n_patterns=13)
    m = torch.from_numpy(scan.truth.astype(np.float32)).cuda()
    s, g, _ = plan.kinematical_score(*to_dev(scan), m, rho=0.05)
    refl = au_refl()
    for b in range(scan.n_patterns):
        want = O.kinematical_score(scan.truth[b].astype(np.float32).astype(np.float64).T,
                                   *scan.pattern(b), refl, LAM, sigma, 0.05)
        if sigma < 1e-3:
            # at such a width FP32 excitation errors decide at random; finite and no larger
            # than the peaks' weights allow
            assert math.isfinite(float(s[b])) and torch.isfinite(g[b]).all()
            continue
        assert float(s[b]) == pytest.approx(want.S, rel=1e-4), b
        np.testing.assert_allclose(g[b].cpu().numpy(), want.grad, rtol=0,
                                   atol=1e-3 * np.abs(want.grad).max(), err_msg=str(b))
    plan.close()


@pytest.mark.parametrize("step", [45.0, 9.0, 2.0])
def test_grid_neighbours(step):
    """Neighbour lists of grids with fewer axes than a warp's lanes, some more, and several
    hundred: the refined orientation, a mean over the listed axes, is the oracle's."""
    from oracle import acom_oracle as O
    from gpu_common import au_refl
    v0, v1, v2, area = O.cubic_triangle()
    za = O.zone_axis_grid(v0, v1, v2, step, area)
    oplan = O.orientation_plan(au_refl(), za, O.PlanParams(40, 0.0375, 72, 0.08, lam=LAM))
    plan = au_plan(step, 40, 0.0375, 72)
    scan = synth.random_patterns(9, n_patterns=12)
    r = plan.match(*to_dev(scan))
    m = r["orient"].cpu().numpy()
    same = 0
    for b in range(scan.n_patterns):
        mt = O.match_pattern(oplan, *scan.pattern(b))
        if (int(r["za_idx"][b]), int(r["phi3_bin"][b]), int(r["mirror"][b])) != (mt.za, mt.k, mt.mirror):
            continue                                            # a tie resolved the other way
        same += 1
        # FP32 scores weight the mean: 1e-5 relative, over a neighbourhood below 1.2 radians
        np.testing.assert_allclose(m[b], O.refine(mt, za, step).m, atol=1e-4)
    assert same > 0
    plan.close()


@pytest.mark.parametrize("q_max", [0.5, 1.5, 3.1])
def test_reflections_of_small_and_large_boxes(q_max):
    """Index boxes of a part of a block, of several blocks, and of several rounds of the
    compaction: as many reflections as the oracle's, and their order and amplitudes through
    the plan's spectra (rows are normalised sums in that order)."""
    from oracle import acom_oracle as O
    from paper_2111_00171_gb300 import acom
    tri, area = acom.cubic_triangle()
    au = acom.au_crystal()
    refl = O.reflections(au.lattice, au.frac_pos, au.ff_A, au.ff_B, q_max)
    plan = acom.Plan(au, tri, area, 12.0, 40, 0.08, 72, lam=LAM, q_max=q_max)
    assert plan.info["n_reflections"] == len(refl.F)
    za = O.zone_axis_grid(*O.cubic_triangle()[:3], 12.0, O.cubic_triangle()[3])
    oplan = O.orientation_plan(refl, za, O.PlanParams(40, 0.08, 72, 0.08, lam=LAM))
    scan = synth.random_patterns(10, n_patterns=8)
    r = plan.match(*to_dev(scan))
    for b in range(scan.n_patterns):
        assert math.isclose(float(r["score"][b]), O.match_pattern(oplan, *scan.pattern(b)).score,
                            rel_tol=1e-4), b
    plan.close()


@pytest.mark.parametrize("call", ["match", "bounds", "polar_spectra", "refine", "kinematical_score"])
def test_rows_that_do_not_start_at_zero(call):
    """A batch whose rows start at the second peak (all in range) is refused by whichever
    kernel reads the first pattern, and the next good batch is accepted."""
    import torch
    from paper_2111_00171_gb300 import acom
    plan = au_plan(6.0, 40, 0.0375, 72)
    scan = synth.random_patterns(11, n_patterns=70)
    rp, qx, qy, I = to_dev(scan)
    bad = rp.clone()
    bad[0] = 1
    m = torch.from_numpy(scan.truth.astype(np.float32)).cuda()
    run = getattr(plan, call)
    more = {"refine": (m.clone(),), "kinematical_score": (m,)}.get(call, ())
    with pytest.raises(acom.AcomError, match="row_ptr"):
        run(bad, qx, qy, I, *more)
    run(rp, qx, qy, I, *more)
    plan.close()


@pytest.mark.parametrize("geometry", [(6.0, 117, 0.0125, 300), (6.0, 85, 0.0175, 120)], ids=str)
def test_e4m3_bounds_of_the_last_shells(geometry):
    """Plans whose first shell is an odd multiple of 16, so that E4M3's K steps of 32 end
    past the last shell: bounds of patterns with all peaks there against FP64.  Rounding a
    product of two E4M3 values costs 2^-3 + 2^-8 of it at most, both parts of a complex
    product sqrt 2 times that; 2^-6 more for values below the normal range."""
    import torch
    plan = au_plan(*geometry, precision=3)
    N, F = geometry[3], geometry[3] // 2 + 1
    assert plan.info["k0"] % 32 == 16
    P = torch.view_as_complex(plan.spectra()).to(torch.complex128)
    last = int((P.abs().amax((0, 2)) > 0).nonzero().max())     # the last shell that is not empty
    rng = np.random.default_rng(5)
    rp = np.concatenate([[0], np.cumsum(rng.integers(4, 12, 9))]).astype(np.int64)
    r, t = last * geometry[2] + 0.05, rng.uniform(-np.pi, np.pi, rp[-1])
    peaks = tuple(torch.from_numpy(x).cuda() for x in (
        rp, (r * np.cos(t)).astype(np.float32), (r * np.sin(t)).astype(np.float32),
        np.ones(rp[-1], np.float32)))
    X = torch.view_as_complex(plan.polar_spectra(*peaks)[0]).to(torch.complex128)
    w = torch.full((F,), 2.0 / N, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 1.0 / N
    want, _ = bounds64(plan, peaks)
    tol = (math.sqrt(2.0) * (2.0 ** -3 + 2.0 ** -8) + 2.0 ** -6) * (
        torch.einsum("zsf,bsf->bzf", P.abs(), X.abs()) * w).sum(2)
    assert ((plan.bounds(*peaks).double() - want).abs() <= tol).all()
    assert (want > 2.0 * tol).any()                            # a missing shell would show
    one, pair = (plan.match(*peaks, cta_pairs=c) for c in (0, 1))
    assert (one["za_idx"] == pair["za_idx"]).all() and (one["score"] == pair["score"]).all()
    plan.close()
