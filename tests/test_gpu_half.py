"""FP16 copies of TF32 operands: the operands are the same, so a contraction computed from copies is the product of the operands
rounded to 11 bits; a copy that cannot hold its matrix is not used."""
import numpy as np
import pytest

import gn_workloads as wl
from oracle import gn_oracle as orc
from test_gpu_parity import TOL, dev, make_ctx, relb

pytestmark = pytest.mark.gpu
HALF, PAIR = 9, 5                    # debug_gemm kinds: the CTA-pair kernel on copies, and on the FP32 matrices


def round11(a):
    """To nearest even, 11 significant bits: what TMA makes of a float on its way to TF32, and FP16 of a scaled one."""
    bits = a.view(np.uint32)
    return ((bits + 0xFFF + ((bits >> 13) & 1)) & 0xFFFFE000).astype(np.uint32).view(np.float32)


@pytest.fixture(scope="module")
def ctx():
    import paper_1802_00130_b200 as gn
    p = wl.make("tiny")
    c = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]), gn.GN_TF32)
    yield c
    c.close()


def operands(M, N, K, a_k, b_k, seed, scale=1.0):
    rng = np.random.Generator(np.random.PCG64(seed))
    A = scale * rng.standard_normal((M, K) if a_k else (K, M), dtype=np.float32)
    B = rng.standard_normal((N, K) if b_k else (K, N), dtype=np.float32)
    return A, B


# tile edges in M (256), N (tiles of 128, 192 and 256) and K (blocks of 64), K slices, several rounds of tiles
SHAPES = [(132, 128, 20), (256, 256, 64), (260, 132, 68), (512, 384, 1000), (640, 192, 520), (300, 520, 200), (260, 2000, 3000),
          (2000, 784, 3000), (12000, 2000, 196)]


@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
@pytest.mark.parametrize("shape", SHAPES)
def test_contraction_of_copies_is_the_product_of_the_rounded_operands(ctx, shape, a_k, b_k):
    M, N, K = shape
    A, B = operands(M, N, K, a_k, b_k, M + 3 * N + 5 * K)
    D = ctx.debug_gemm(HALF, dev(A), dev(B), a_kmajor=a_k, b_kmajor=b_k).cpu().numpy()
    ra, rb = round11(A).astype(np.float64), round11(B).astype(np.float64)
    ref = (ra if a_k else ra.T) @ (rb.T if b_k else rb)
    # the tensor core truncates each addition of 16 terms into its accumulator: at most 2^-23 of it a step, and the products are exact
    bound = (K / 16 + 1) * 2.0 ** -23
    assert np.linalg.norm(D - ref) <= bound * np.linalg.norm(ref)
    assert np.max(np.abs(D - ref)) <= 8 * bound * np.sqrt(K)


@pytest.mark.parametrize("scale", [1e-30, 1e-12, 1e12, 1e30])
def test_scales_of_whole_matrices_cost_nothing(ctx, scale):
    A, B = operands(300, 260, 500, True, True, 11, scale)
    D = ctx.debug_gemm(HALF, dev(A), dev(B)).cpu().numpy().astype(np.float64)
    ref = round11(A).astype(np.float64) @ round11(B).astype(np.float64).T
    assert np.linalg.norm(D - ref) <= 1e-5 * np.linalg.norm(ref)


def far_column(A):
    A[:, 3] *= 1e-11


def far_row(A):
    A[7] *= 1e-11


def infinity(A):
    A[5, 9] = np.inf


def not_a_number(A):
    A[5, 9] = np.nan


@pytest.mark.parametrize("spoil", [far_column, far_row, infinity, not_a_number])
@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, False)])
def test_a_copy_that_cannot_hold_its_matrix_is_not_used(ctx, spoil, a_k, b_k):
    A, B = operands(520, 392, 300, a_k, b_k, 13)
    spoil(A)
    got = ctx.debug_gemm(HALF, dev(A), dev(B), a_kmajor=a_k, b_kmajor=b_k).cpu().numpy()
    want = ctx.debug_gemm(PAIR, dev(A), dev(B), a_kmajor=a_k, b_kmajor=b_k).cpu().numpy()
    # (with TF32 operands the K slices are cut at other places: the order of sums may differ, nothing else)
    fin = np.isfinite(want)
    assert np.array_equal(fin, np.isfinite(got))
    assert np.linalg.norm(got[fin] - want[fin]) <= 1e-5 * np.linalg.norm(want[fin])
    if spoil in (far_column, far_row):          # the far row or column itself
        ref = round11(A).astype(np.float64)
        ref = (ref if a_k else ref.T) @ (round11(B).astype(np.float64).T if b_k else round11(B).astype(np.float64))
        rows = np.linalg.norm(got - ref, axis=1) <= 1e-5 * np.linalg.norm(ref, axis=1)
        assert rows.all()


def far_end_of_a_column(A):
    A[:-(A.shape[0] % 16 or 16), 3] = 0
    A[-(A.shape[0] % 16 or 16):, 3] *= 1e-11


def far_end_of_a_row(A):
    A[7, :-(A.shape[1] % 128)] = 0
    A[7, -(A.shape[1] % 128):] *= 1e-11


@pytest.mark.parametrize("spoil", [far_end_of_a_column, far_end_of_a_row])
@pytest.mark.parametrize("a_k", [True, False])
def test_runs_at_the_end_of_a_row_or_column_are_judged(ctx, spoil, a_k):
    """The only numbers of a row or column stand at its end, in fewer elements than a run has, far below the others."""
    A, B = operands(516, 392, 300, a_k, True, 13)
    spoil(A)
    got = ctx.debug_gemm(HALF, dev(A), dev(B), a_kmajor=a_k, b_kmajor=True).cpu().numpy()
    ref = round11(A).astype(np.float64)
    ref = (ref if a_k else ref.T) @ round11(B).astype(np.float64).T
    assert (np.linalg.norm(got - ref, axis=1) <= 1e-5 * np.linalg.norm(ref, axis=1)).all()


NETS = {
    "mid": lambda: wl.make("mid"),
    "wide_output": lambda: wl.make_custom([260, 392, 520, 260, 132], l=1500, nS=1100, C=15.0, seed=51, x="normal"),
    "ragged_tiles": lambda: wl.make_custom([300, 520, 392, 264, 10], l=2300, nS=1700, C=23.0, seed=53, x="sparse80"),
    "one_output": lambda: wl.make_custom([260, 392, 264, 1], l=1500, nS=1100, C=15.0, seed=61, x="normal"),
    "three_outputs": lambda: wl.make_custom([260, 392, 268, 3], l=1500, nS=1037, C=15.0, seed=63, x="normal"),
    "sixteen_outputs": lambda: wl.make_custom([260, 392, 132, 16], l=1500, nS=1100, C=15.0, seed=65, x="uniform"),
    "two_layers": lambda: wl.make_custom([784, 516, 7], l=1200, nS=900, C=12.0, seed=55, x="uniform"),
}


@pytest.mark.parametrize("v_scale", [1.0, 1e-15])
@pytest.mark.parametrize("name", sorted(NETS))
def test_passes_with_copies_against_the_checker(name, v_scale):
    """Products, block products, gradient and loss with copies wherever they can be made and with none: both within the mode's
    bound, the same from run to run, and no further from the checker with copies than without."""
    import torch
    p = NETS[name]()
    w, th, C = p["widths"], p["theta"], p["C"]
    XS, v = p["X"][p["idx"]], (v_scale * p["v"]).astype(np.float32)
    refs = [orc.Gv(th, w, C, XS, v), orc.Gv_blockdiag(th, w, C, XS, v), orc.grad(th, w, C, p["X"], p["Y"])]
    err = {}
    for mode in (0, 2):
        c = make_ctx(p, "tf32")
        c.debug_option(10, 0)
        c.debug_option(11, mode)
        if w[-1] <= 16:
            c.set_blockdiag_method(2)
        c.set_subsample(dev(p["idx"]))
        first = [c.Gv(dev(v)).clone(), c.Gv_blockdiag(dev(v)).clone(), c.grad().clone()]
        again = [c.Gv(dev(v)).clone(), c.Gv_blockdiag(dev(v)).clone(), c.grad().clone()]
        assert all(torch.equal(a, b) for a, b in zip(first, again))
        err[mode] = [relb(a.cpu().numpy(), r, w) for a, r in zip(first, refs)]
        assert max(err[mode]) <= TOL["tf32"]
        f = c.fun()
        assert abs(f - orc.fun(th, w, C, p["X"], p["Y"])) <= TOL["tf32"] * abs(f)
        c.close()
    assert all(a <= 1.02 * b + 1e-6 for a, b in zip(err[2], err[0]))


def test_saturated_neurons_and_far_features():
    """Activations and deltas of saturated neurons lie many orders below the others, and so do features with compensating weights:
    whole rows of the result depend on them, and have the mode's accuracy."""
    p = wl.make_custom([260, 392, 264, 10], l=1500, nS=1100, C=15.0, seed=57, x="uniform")
    w, th = p["widths"], p["theta"].copy()
    W1 = th[:260 * 392].reshape(392, 260)
    p["X"][:, 5] *= np.float32(1e-12)
    W1[:, 5] *= np.float32(1e12)
    th[260 * 392 + 9] -= 30.0           # b^1 of neuron 9: z about 1e-13
    p["theta"] = th
    XS = p["X"][p["idx"]]
    v = p["v"]
    ref = orc.Gv(th, w, p["C"], XS, v)
    gref = orc.grad(th, w, p["C"], p["X"], p["Y"])
    for mode in (0, 2):
        c = make_ctx(p, "tf32")
        c.debug_option(11, mode)
        c.set_subsample(dev(p["idx"]))
        assert relb(c.Gv(dev(v)).cpu().numpy(), ref, w) <= TOL["tf32"]
        g = c.grad().cpu().numpy()
        assert relb(g, gref, w) <= TOL["tf32"]
        reg = th / p["C"]               # the loss's own part of the rows in question
        got, want = (g - reg)[:260 * 392].reshape(392, 260), (gref - reg)[:260 * 392].reshape(392, 260)
        assert np.linalg.norm(got[:, 5] - want[:, 5]) <= 1e-2 * np.linalg.norm(want[:, 5]) + 1e-6 * np.linalg.norm(reg[:260 * 392])
        c.close()


@pytest.mark.parametrize("split", [[1, 2, 2, 1, 1], [2, 2, 1, 2, 1], [1, 3, 2, 2, 1], [1, 4, 3, 1, 1]])
def test_split_structures_with_copies_against_the_checker(split):
    """Sub-blocks of stored matrices as operands: groups that start on a copy's 16 bytes use it, others do not, streams beyond two
    have none of their results."""
    p = wl.make_custom([304, 528, 392, 264, 10], l=2300, nS=1700, C=23.0, seed=59, x="sparse80")
    w = p["widths"]
    ref = orc.Gv_partition(p["theta"], w, p["C"], p["X"][p["idx"]], p["v"], split)
    for mode in (0, 2):
        c = make_ctx(p, "tf32")
        c.debug_option(11, mode)
        c.set_split(split)
        c.set_subsample(dev(p["idx"]))
        for _ in range(2):
            assert relb(c.Gv_blockdiag(dev(p["v"])).cpu().numpy(), ref, w) <= TOL["tf32"]
        c.close()


@pytest.mark.parametrize("slices", [0, 1])
@pytest.mark.parametrize("k", list(range(-1, 13)) + [16, 20, 24, 31, 40, 60])
def test_scales_of_the_two_operand_pairs_lie_any_distance_apart(k, slices):
    """One weight of 2^k in every hidden layer above the first: each doubling takes the scale of R z W one power of two further
    below that of z V (5 to 8 with the other weights alone), through the 15 that one instruction can bridge."""
    p = wl.make_custom([260, 392, 520, 392, 10], l=1500, nS=1100, C=1e6, seed=67, x="sparse80")
    w, th = p["widths"], p["theta"]
    for m, (w_off, _, _) in enumerate(wl.layer_offsets(w), 1):
        if 2 <= m < 4:
            th[w_off + 7 * w[m - 1] + 11] = 2.0 ** k
    ref = orc.Gv(th, w, p["C"], p["X"][p["idx"]], p["v"])
    c = make_ctx(p, "tf32")
    c.debug_option(11, 2)
    c.debug_option(1, slices)
    c.set_subsample(dev(p["idx"]))
    assert relb(c.Gv(dev(p["v"])).cpu().numpy(), ref, w) <= TOL["tf32"]
    c.close()


def test_a_copy_ends_with_its_pass():
    """The memory of a product's vector comes back with other numbers: they are what a contraction reads there."""
    p = wl.make_custom([260, 392, 264, 10], l=1500, nS=1100, C=15.0, seed=69, x="uniform")
    w = p["widths"]
    c = make_ctx(p, "tf32")
    c.debug_option(11, 2)
    c.set_subsample(dev(p["idx"]))
    v = dev(p["v"])
    c.Gv(v)
    fresh = np.random.Generator(np.random.PCG64(71)).standard_normal(p["n"], dtype=np.float32)
    v.copy_(dev(fresh))
    w_off, b_off, _ = wl.layer_offsets(w)[1]                       # W^2: 264 x 392
    A, B = fresh[w_off:b_off].reshape(w[2], w[1]), operands(132, 132, w[1], True, True, 73)[1]
    D = c.debug_gemm(HALF, v[w_off:b_off].view(w[2], w[1]), dev(B)).cpu().numpy()
    ref = round11(A).astype(np.float64) @ round11(B).astype(np.float64).T
    assert np.linalg.norm(D - ref) <= 1e-5 * np.linalg.norm(ref)
    c.close()


def test_copies_and_memory_that_changes_hands():
    """Buffers are let go and got again (a larger subsample, other row batches, factors, the propagate form's deeper buffers,
    the caller's vector): every result is that of the matrices which are there now."""
    import torch
    p = wl.make_custom([392, 392, 392, 392, 10], l=2300, nS=1700, C=23.0, seed=75, x="sparse80")
    w, th, C, v = p["widths"], p["theta"], p["C"], p["v"]
    c = make_ctx(p, "tf32")
    c.debug_option(11, 2)
    grad_ref = orc.grad(th, w, C, p["X"], p["Y"])
    for nS, batch, method in [(600, 1000, 2), (1100, 2300, 2), (600, 700, 1), (1700, 1500, 2), (1300, 2000, 1)]:
        c.set_batch_rows(batch)
        c.set_blockdiag_method(method)
        c.set_subsample(dev(p["idx"][:nS]))
        XS = p["X"][p["idx"][:nS]]
        dv = dev(v)
        got = c.Gv(dv).cpu().numpy()
        del dv
        torch.cuda.empty_cache()
        assert relb(got, orc.Gv(th, w, C, XS, v), w) <= TOL["tf32"]
        assert relb(c.grad().cpu().numpy(), grad_ref, w) <= TOL["tf32"]
        for _ in range(2):
            assert relb(c.Gv_blockdiag(dev(v)).cpu().numpy(), orc.Gv_blockdiag(th, w, C, XS, v), w) <= TOL["tf32"]
    c.close()


@pytest.mark.parametrize("theta,outlier,rows", [("sparse", 0.0, 1104), ("sparse", 0.0, 1105), ("dense", 0.0, 1105), ("dense", 8.0, 1100), ("dense", 64.0, 1100)])
def test_copies_hold_ordinary_networks(theta, outlier, rows):
    """The initialisation of the paper (a few weights of order one per neuron, saturated neurons), and single large weights: no
    copy is refused, and results are those without copies."""
    p = wl.make_custom([392, 1000, 1000, 1000, 10], l=1501, nS=rows, C=15.0, seed=79, x="sparse80", theta=theta)
    w, th, C, v = p["widths"], p["theta"], p["C"], p["v"]
    for m, (w_off, _, _) in enumerate(wl.layer_offsets(w), 1):
        if outlier and 2 <= m < 4:
            th[w_off + 7 * w[m - 1] + 11] = outlier
    XS = p["X"][p["idx"]]
    refs = [orc.Gv(th, w, C, XS, v), orc.Gv_blockdiag(th, w, C, XS, v), orc.grad(th, w, C, p["X"], p["Y"])]
    c = make_ctx(p, "tf32")
    c.debug_option(11, 2)
    c.set_blockdiag_method(2)
    c.set_subsample(dev(p["idx"]))
    for call, ref in zip((lambda: c.Gv(dev(v)), lambda: c.Gv_blockdiag(dev(v)), c.grad), refs):
        got = call().cpu().numpy()
        known, refused = c.debug_copies()
        assert known >= 6 and (refused == 0 or outlier > 8.0)       # (64 saturates a neuron: its column lies low as a whole)
        assert relb(got, ref, w) <= TOL["tf32"]
    c.close()


def test_a_copy_that_cannot_hold_its_matrix_is_refused():
    """Far features (1e-12 of the others): the copy of X_S loses them, and is refused."""
    p = wl.make_custom([260, 392, 264, 10], l=1500, nS=1100, C=15.0, seed=57, x="uniform")
    p["X"][:, 5] *= np.float32(1e-12)
    c = make_ctx(p, "tf32")
    c.debug_option(11, 2)
    c.set_subsample(dev(p["idx"]))
    c.Gv(dev(p["v"]))
    assert c.debug_copies()[1] == 1
    c.close()


def test_copies_make_room_for_what_a_call_cannot_do_without():
    """One allocation refused at a time, on the host, in contexts that hold copies: what a pass needs gets the room of the copies,
    a copy without room is done without, and the next subsample has copies again.  No call fails."""
    p = wl.make_custom([260, 392, 520, 264, 10], l=1500, nS=1100, C=15.0, seed=81, x="sparse80")
    w, th, C, v = p["widths"], p["theta"], p["C"], dev(p["v"])
    XS, idx = p["X"][p["idx"]], dev(p["idx"])
    refs = dict(Gv=orc.Gv(th, w, C, XS, p["v"]), block=orc.Gv_blockdiag(th, w, C, XS, p["v"]), grad=orc.grad(th, w, C, p["X"], p["Y"]))
    calls = dict(Gv=lambda c: c.Gv(v), block=lambda c: c.Gv_blockdiag(v), grad=lambda c: c.grad())
    for name, call in calls.items():
        for n in range(1, 12):
            c = make_ctx(p, "tf32")
            c.debug_option(11, 2)
            c.set_blockdiag_method(2)
            c.set_subsample(idx)
            c.debug_option(2, n)
            got = call(c).cpu().numpy()
            c.debug_option(2, 0)
            assert relb(got, refs[name], w) <= TOL["tf32"]
            for other, again in calls.items():
                assert relb(again(c).cpu().numpy(), refs[other], w) <= TOL["tf32"]
            c.set_subsample(idx)
            for other, again in calls.items():
                assert relb(again(c).cpu().numpy(), refs[other], w) <= TOL["tf32"]
            assert c.debug_copies()[0] > 0
            c.close()


@pytest.mark.parametrize("widths", [[392] * 4 + [10], [520] * 3 + [10]])
def test_a_place_ends_with_its_pass(widths):
    """Row batches' buffers are let go and the subsample's got in their place, in sizes that meet at the same addresses now and
    then: what a product writes there are its own copies, not those that the gradient kept beside a matrix at that address."""
    p = wl.make_custom(widths, l=2300, nS=1700, C=23.0, seed=75, x="sparse80")
    w, v, many, refs = p["widths"], dev(p["v"]), (700, 1000, 1100, 1300, 1700), {}
    for rows in many:
        c = make_ctx(p, "tf32")
        c.debug_option(11, 0)
        c.set_subsample(dev(p["idx"][:rows]))
        refs[rows] = c.Gv(v).clone()
        c.close()
        ref = orc.Gv(p["theta"], w, p["C"], p["X"][p["idx"][:rows]], p["v"])
        assert relb(refs[rows].cpu().numpy(), ref, w) <= TOL["tf32"]
    for first in (0, 300, 600):
        for batch in (500, 800, 1000, 1300):
            for rows in many:
                for blocks in (0, 1):
                    c = make_ctx(p, "tf32")
                    c.debug_option(11, 2)
                    c.set_batch_rows(batch)
                    c.set_blockdiag_method(2)
                    if first:
                        c.set_subsample(dev(p["idx"][:first]))
                        c.Gv(v)
                    c.grad()
                    if first and blocks:
                        c.Gv_blockdiag(v)
                    c.set_batch_rows(2300)
                    c.set_subsample(dev(p["idx"][:rows]))
                    d = c.Gv(v)
                    assert float((d - refs[rows]).norm() / refs[rows].norm()) <= TOL["tf32"]
                    c.close()
