"""The fp16 digit products that carry the GEMM-class steps of the F64 and F32 modes, through the
path's own gather and GEMM, against extended-precision products and the CUDA-core GEMMs."""
import time

import numpy as np
import pytest

from paper_2103_11595_gb300 import ajf, workloads as W

# shapes (complex M, N, K): the smallest; 2 and 4 digits per 128-byte row (K = 16, 8); X tiles of 32,
# 64 and 128 rows; Y tiles with and without missing rows; one and several K chunks and strips; K splits
SHAPES = [(16, 16, 8), (16, 256, 16), (32, 128, 8), (64, 32, 32), (128, 256, 32), (16, 512, 64), (256, 16, 128),
          (64, 64, 512), (16, 32, 4096)]


def operands(M, N, K, dist, seed):
    r = np.random.default_rng(seed)
    A = r.standard_normal((M, K)) + 1j * r.standard_normal((M, K))
    B = r.standard_normal((N, K)) + 1j * r.standard_normal((N, K))
    if dist == "equal":  # every digit of every entry the same: the largest sums the tensor core can see
        A = np.full((M, K), 1.9999999999999998 * (1 + 1j))
        B = np.full((N, K), -1.9999999999999998 * (1 - 1j))
    elif dist == "graded":
        A = A * 10.0 ** r.uniform(-200, 0, (M, 1)) * 10.0 ** r.uniform(-3, 0, (M, K))
        B = B * 10.0 ** r.uniform(-3, 0, (N, K))
        A[1], B[2] = 0, 0
    return A, B


def exact(A, B):
    a, b, c, d = (x.astype(np.longdouble) for x in (A.real, A.imag, B.real, B.imag))
    return a @ c.T - b @ d.T, a @ d.T + b @ c.T


def bound(A, B, R, f32):
    """Element bound. Digits: 2^-56 (F64) or 2^-38 of the row maximum per factor, the dropped levels
    less than that again, over 2K products; the fixed-point sum: up to three roundings per chunk of
    64 columns in units of 2^-54 (chunks per sum) of the maxima's product; the result's own rounding."""
    K2 = 2 * A.shape[1]
    m = np.maximum(abs(A.real), abs(A.imag)).max(1)[:, None] * np.maximum(abs(B.real), abs(B.imag)).max(1)[None, :]
    chunks = max(1, K2 // 64)
    c = min(chunks, 32)
    per = K2 * 4 * (2.0 ** -38 if f32 else 2.0 ** -56) + 1.5 * chunks * c * 2.0 ** -54
    return 2.0 ** (-24 if f32 else -53) * 1.01 * np.maximum(abs(R[0]), abs(R[1])).astype(float) + m * per


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_digit_gemm_against_extended_precision(precision, shape):
    for dist in ("normal", "equal", "graded"):
        if precision == "f32" and dist == "graded":
            continue  # FP32 results would leave their range
        A, B = operands(*shape, dist, 7)
        R = exact(A, B)
        got = [ajf.ajf_selftest_digit_gemm(0, precision, A, B, order=o) for o in (0, 1, 2)]
        assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])  # any source bit order
        err = np.maximum(abs(got[0].real - R[0]), abs(got[0].imag - R[1])).astype(float)
        assert (err <= bound(A, B, R, precision == "f32")).all(), (dist, (err / bound(A, B, R, precision == "f32")).max())
        # and no further off than the CUDA-core GEMM it stands in for
        simt = ajf.ajf_selftest_digit_gemm(0, precision, A, B, digits=False)
        es = np.maximum(abs(simt.real - R[0]), abs(simt.imag - R[1])).astype(float)
        assert np.linalg.norm(err) <= np.linalg.norm(es) or dist == "equal"


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(16, 16, 8), (16, 32, 16), (32, 128, 64), (64, 64, 512), (16, 32, 4096)])
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_non_finite_rows_stay_non_finite(precision, shape):
    """A row with an infinity or a NaN anywhere gives NaN products, and no other row is touched."""
    M, N, K = shape
    A, B = operands(M, N, K, "normal", 3)
    clean = ajf.ajf_selftest_digit_gemm(0, precision, A, B)
    A, B = A.copy(), B.copy()
    A.real[1, K - 1] = np.inf
    A.imag[M - 1, 0] = np.nan
    B.imag[2, K // 2] = -np.inf
    B.real[N - 1, 1] = np.nan
    bad = np.zeros((M, N), bool)
    bad[[1, M - 1]] = True
    bad[:, [2, N - 1]] = True
    for order in (0, 1, 2):
        C = ajf.ajf_selftest_digit_gemm(0, precision, A, B, order=order)
        assert np.isnan(C.real[bad]).all() and np.isnan(C.imag[bad]).all()
        assert np.array_equal(C[~bad], clean[~bad])


@pytest.mark.gpu
def test_fixed_arena_takes_plans_that_only_digits_outgrow():
    """A plan over the 64 MiB of the no-allocation call because of its digit operands runs there with
    CUDA-core GEMMs, and the context's own program is unchanged."""
    inst = W.mid(0)
    with ajf.Context(0) as c:
        ajf.load_instance(c.handle, inst)
        info = ajf.ajf_plan(c.handle, 1, trials=8)
        assert info["n_tc_gemms"] > 0 and info["arena_bytes"] > 64 << 20
        r = ajf.ajf_fidelity_alg1(c.handle)
        n = ajf.ajf_fidelity_noalloc(c.handle, 1)
        again = ajf.ajf_fidelity_alg1(c.handle)
    assert abs(n["F"] - r["F"]) <= 1e-12 and again == r


@pytest.mark.gpu
@pytest.mark.parametrize("n,gates,noises,seed,own", [(14, 170, 8, 1, False), (14, 170, 8, 2, True)])
def test_fixed_arena_calls_only_enqueue_once_prepared(n, gates, noises, seed, own):
    """Plans that fit the fixed arena with CUDA-core GEMMs only, on their own path (no preparation needed:
    lowering takes a millisecond) and on one planned for it (ajf_prepare_noalloc): no call plans, which takes
    0.6 s here against milliseconds for the evaluation, and all agree."""
    inst = W.mid(seed, n=n, n_gates=gates, n_noises=noises)
    with ajf.Context(0) as c:
        ajf.load_instance(c.handle, W.tiny(0))  # loads the kernels of the path
        ajf.ajf_plan(c.handle, 2, trials=2)
        ajf.ajf_fidelity_noalloc(c.handle, 2)
        ajf.load_instance(c.handle, inst)
        info = ajf.ajf_plan(c.handle, 2, trials=8)
        assert info["arena_bytes"] > 64 << 20 and info["plan_seconds"] > 0.1
        r = ajf.ajf_fidelity_alg2(c.handle)
        if own:
            ajf.ajf_prepare_noalloc(c.handle)
        t = []
        for _ in range(3):
            t0 = time.perf_counter()
            got = ajf.ajf_fidelity_noalloc(c.handle, 2)
            t.append(time.perf_counter() - t0)
            assert abs(got["F"] - r["F"]) <= 1e-12
        assert t[0] < 3 * min(t) + 0.05
        ajf.ajf_prepare_noalloc(c.handle)  # nothing left to do
        ajf.load_instance(c.handle, W.mid(0))
        ajf.ajf_plan(c.handle, 2, trials=2)
        for call in (lambda: ajf.ajf_prepare_noalloc(c.handle), lambda: ajf.ajf_fidelity_noalloc(c.handle, 2)):
            with pytest.raises(ajf.AjfError) as e:
                call()
            assert e.value.status == ajf.AJF_E_NOMEM


def test_prepare_noalloc_needs_a_plan_and_a_device():
    with ajf.Context(-1) as c:
        ajf.load_instance(c.handle, W.tiny(0))
        for plan in (False, True):
            if plan:
                ajf.ajf_plan(c.handle, 2, trials=2)
            with pytest.raises(ajf.AjfError) as e:
                ajf.ajf_prepare_noalloc(c.handle)
            assert e.value.status == ajf.AJF_E_STATE


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_budget_between_the_two_gemms_keeps_the_plan(precision):
    """A memory budget that the CUDA-core GEMMs' plan meets is met, whatever the digit operands need."""
    inst = W.mid(0)
    with ajf.Context(-1) as c:
        ajf.load_instance(c.handle, inst)
        roomy = ajf.ajf_plan(c.handle, 2, precision=precision, trials=8)
        assert roomy["n_tc_gemms"] > 0
        ajf.ajf_check_plan(c.handle)
        tight = ajf.ajf_plan(c.handle, 2, precision=precision, trials=8, mem_budget_bytes=0.96 * roomy["arena_bytes"])
        ajf.ajf_check_plan(c.handle)
        assert tight["n_tc_gemms"] == 0 and tight["arena_bytes"] <= 0.96 * roomy["arena_bytes"]
        again = ajf.ajf_plan(c.handle, 2, precision=precision, trials=8)
        assert again["n_tc_gemms"] > 0 and again["arena_bytes"] == roomy["arena_bytes"]


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_plans_do_not_depend_on_the_budgets_before(precision):
    """In one context, plans for falling and rising budgets are those of fresh contexts: as small, or
    refused as over the budget with the smallest arena that any of the GEMMs and paths needs."""
    inst = W.mid(0)

    def plan(c, budget):
        try:
            i = ajf.ajf_plan(c.handle, 2, precision=precision, trials=8, mem_budget_bytes=budget)
            return i["arena_bytes"], i["n_tc_gemms"]
        except ajf.AjfError as e:
            assert e.status == ajf.AJF_E_BUDGET
            return "over budget", str(e).split("bytes")[0]

    with ajf.Context(-1) as c:
        ajf.load_instance(c.handle, inst)
        roomy = plan(c, 1e18)[0]
        for f in (0.96, 0.85, 0.8, 0.3, 0.8, 0.96, 0.2, 1.0):
            with ajf.Context(-1) as fresh:
                ajf.load_instance(fresh.handle, inst)
                want = plan(fresh, f * roomy)
            assert plan(c, f * roomy) == want, f
        over = [plan(c, 1.0)[1], plan(c, 0.3 * roomy)[1]]
        assert over[0] == over[1]  # the smallest, and kept: nothing is left to try
        smallest = float(over[0].split("needs")[1])
        assert plan(c, smallest)[0] == smallest and plan(c, smallest - 1)[0] == "over budget"


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_auto_slicing_leaves_plans_whole_that_fit_with_either_gemm(precision):
    """AJF_SLICE_AUTO slices nothing while some unsliced plan fits the budget (a sliced plan is refused by
    the single-run calls), and digit products' plans beyond that."""
    inst = W.mid(0)

    def plan(budget, **kw):
        with ajf.Context(-1) as c:
            ajf.load_instance(c.handle, inst)
            info = ajf.ajf_plan(c.handle, 2, precision=precision, trials=8, mem_budget_bytes=budget, **kw)
            ajf.ajf_check_plan(c.handle)
        return info

    roomy = plan(1e18)["arena_bytes"]
    with pytest.raises(ajf.AjfError) as e:
        plan(1.0)
    smallest = float(str(e.value).split("needs")[1].split("bytes")[0])
    assert smallest < roomy
    for budget in (roomy, roomy - 1, smallest):
        auto, plain = plan(budget, slice_bonds="auto"), plan(budget)
        assert auto["n_sliced_bonds"] == 0 and auto["arena_bytes"] == plain["arena_bytes"] <= budget
    tight = plan(smallest - 1, slice_bonds="auto")
    assert tight["n_sliced_bonds"] == 1 and tight["n_tc_gemms"] > 0 and tight["arena_bytes"] < smallest


def row_bound(A, B, R, f32):
    """Error bound of a digit product against row maxima m (per factor, real parts and imaginary ones), term
    by term. Operands: the last digit's rounding, 2^-56 m (2^-38 m with four digits), on either side.
    Dropped levels, 2^-14 q^2 = m^2 units of 2^(-9 l): 4 pairs of digits at l = 7, 3 at l = 4, and less than
    1% below. Tensor-core sums (64 columns, at most 2^16 per product, 16 products and the running sum to an
    addition, each truncated to a unit of the sum): with six digits exact up to 2^24, so one unit of 2 for
    each of 4 x 17 terms at level 4, where the sum can pass it; with four digits, where the last one has a
    fraction, one unit for each of 16 x 17 terms at level 3. Fixed point: three roundings per chunk in
    units of 2^-54 (chunks per sum). The result's own rounding."""
    K2 = 2 * A.shape[1]
    m = np.maximum(abs(A.real), abs(A.imag)).max(1)[:, None] * np.maximum(abs(B.real), abs(B.imag)).max(1)[None, :]
    chunks = max(1, K2 // 64)
    per = K2 * (2 * 2.0 ** -38 + 3.03 * 2.0 ** -34 if f32 else 2 * 2.0 ** -56 + 4.04 * 2.0 ** -61)
    per += chunks * (272 * 2.0 ** -41 if f32 else 136 * 2.0 ** -50) + 1.5 * chunks * min(chunks, 32) * 2.0 ** -54
    return 2.0 ** (-24 if f32 else -53) * 1.01 * np.maximum(abs(R[0]), abs(R[1])).astype(float) + m * per


@pytest.mark.gpu
@pytest.mark.parametrize("K", [8, 16, 64, 4096])  # four, two and one digits per 128-byte row; K splits
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_digit_gemm_with_the_largest_digits(precision, K):
    """Entries whose digits all are the largest that they can be (255 and -255; 256 and -256): the exact
    levels' sums come within 1% of the 2^24 that FP32 holds, and the fixed-point sums to their largest."""
    T = 4 if precision == "f32" else 6
    places = [2.0 ** (-9 * t) for t in range(T)]
    same = 255.0 * sum(places)                  # 255 in every place
    mixed = 256.0 - 256.0 * sum(places[1:])     # 256, then -256
    for a in (same, -same, mixed):
        for b in (same, mixed):
            for za, zb in ((1 - 1j, 1 + 1j), (1 + 1j, 1 + 1j)):  # all terms of Re, and of Im, of one sign
                A, B = np.full((32, K), a * za), np.full((32, K), b * zb)
                R = exact(A, B)
                C = ajf.ajf_selftest_digit_gemm(0, precision, A, B)
                err = np.maximum(abs(C.real - R[0]), abs(C.imag - R[1])).astype(float)
                assert (err <= row_bound(A, B, R, precision == "f32")).all(), (a, b, err.max())


@pytest.mark.gpu
@pytest.mark.parametrize("decades", [3, 6, 10, 12])
@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_digit_gemm_is_normwise_per_row(precision, decades):
    """Entries graded within their rows, at random and oppositely in the two operands: the error is bounded
    by the row maxima, not by sum |a||b| (the figure printed, with the CUDA-core GEMM's)."""
    r = np.random.default_rng(decades)
    M, N, K = 32, 32, 64
    A = r.standard_normal((M, K)) + 1j * r.standard_normal((M, K))
    B = r.standard_normal((N, K)) + 1j * r.standard_normal((N, K))
    grade = 10.0 ** -np.linspace(0, decades, K)
    for name, fa, fb in (("random", 10.0 ** r.uniform(-decades, 0, (M, K)), 10.0 ** r.uniform(-decades, 0, (N, K))),
                         ("opposed", grade, grade[::-1])):
        a, b = A * fa, B * fb
        R = exact(a, b)
        C = ajf.ajf_selftest_digit_gemm(0, precision, a, b)
        S = ajf.ajf_selftest_digit_gemm(0, precision, a, b, digits=False)
        e, es = (np.maximum(abs(X.real - R[0]), abs(X.imag - R[1])).astype(float) for X in (C, S))
        mag = abs(a) @ abs(b).T
        print(f"{precision} {name} 10^-{decades}: error / sum |a||b| {(e / mag).max():.1e} (CUDA cores {(es / mag).max():.1e})")
        assert (e <= row_bound(a, b, R, precision == "f32")).all()
