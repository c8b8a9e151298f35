"""The FP32-accurate tensor-core contraction at the sizes where it can go wrong, against a float64 product (numpy): edges
of its 256-row tiles, 64-term k-blocks and column widths, K slices, and operands whose scale, zeros or non-finite
elements its splitting pass has to cope with."""
import numpy as np
import pytest

import gn_workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    import paper_1802_00130_b200 as gn
    p = wl.make("tiny")
    c = gn.GnContext(p["widths"], p["C"], torch.from_numpy(p["X"]).cuda(), torch.from_numpy(p["Y"]).cuda())
    yield c
    c.close()


def product(ctx, A, B, a_k, b_k):
    import torch
    D = ctx.debug_gemm(8, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), a_kmajor=a_k, b_kmajor=b_k)
    return D.cpu().numpy().astype(np.float64)


def operands(M, N, K, a_k, b_k):
    rng = np.random.Generator(np.random.PCG64(M + 7 * N + 13 * K))
    A = rng.standard_normal((M, K) if a_k else (K, M), dtype=np.float32)
    B = rng.standard_normal((N, K) if b_k else (K, N), dtype=np.float32)
    return A, B, (A if a_k else A.T).astype(np.float64) @ (B.T if b_k else B).astype(np.float64)


# one element; one row / column / term; around the 256-row tile, the 64-term block and the 32-column chunk; widths that
# take each tile width; few tiles with a long K (slices); whole rounds plus left-over tiles (148 SMs = 74 pairs)
SHAPES = [(1, 1, 1), (1, 300, 65), (300, 1, 64), (255, 31, 63), (256, 32, 64), (257, 33, 129), (131, 65, 191), (513, 129, 7),
          (300, 193, 1000), (26, 803, 4001), (19201, 257, 130)]


@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
@pytest.mark.parametrize("shape", SHAPES)
def test_against_float64(ctx, shape, a_k, b_k):
    M, N, K = shape
    A, B, ref = operands(M, N, K, a_k, b_k)
    D = product(ctx, A, B, a_k, b_k)
    # operand parts: 2^-23 each plus the dropped product 2^-22; accumulation: a few truncated additions of 2^-23 per 128
    # terms, rounded sums of the chunks (measured 1.0e-7 to 4.2e-7)
    assert np.linalg.norm(D - ref) <= 1e-6 * np.linalg.norm(ref)
    bound = np.abs(A if a_k else A.T).astype(np.float64) @ np.abs(B.T if b_k else B).astype(np.float64)
    assert np.all(np.abs(D - ref) <= 2e-6 * bound)


@pytest.mark.parametrize("ea,eb", [(-100, 60), (100, -60), (-126, 126), (60, 60), (-50, -50)])
def test_scales_of_the_operands(ctx, ea, eb):
    """Whole operands far from 1 (down to the smallest normal numbers): the same bits as unscaled, shifted."""
    A, B, _ = operands(200, 96, 150, True, True)
    A, B = np.clip(A, -3.9, 3.9), np.clip(B, -3.9, 3.9)
    D = product(ctx, A, B, True, True)
    E = product(ctx, np.ldexp(A, ea - 2).astype(np.float32), np.ldexp(B, eb - 2).astype(np.float32), True, True)
    if ea > -126:
        assert np.array_equal(np.ldexp(D, ea + eb - 4), E)
    else:                                     # (elements of A below the normal range have lost bits before the call)
        assert np.linalg.norm(np.ldexp(D, ea + eb - 4) - E) <= 1e-5 * np.linalg.norm(E)


def decades(n, d):
    return 10.0 ** -np.linspace(0, d, n)


# what is scaled, over how many decades, and whether the other operand is scaled the other way (so that all terms of a sum
# are of one size); "one" = a single row of 10^-d, "half" = the first half of K
RANGES = [("m", 12, False), ("m", 30, False), ("n", 12, False), ("k", 6, True), ("k", 8, True), ("k", 10, True), ("k", 16, True),
          ("k", 30, True), ("k", 12, False), ("large m", 55, False), ("one m", 12, False), ("one k", 10, True), ("half k", 20, True)]


@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, False)])
@pytest.mark.parametrize("which,d,compensated", RANGES)
def test_wide_range_inside_an_operand(ctx, which, d, compensated, a_k, b_k):
    """Element by element as accurate as any FP32 sum, whatever the range of an operand."""
    M, N, K = 300, 200, 333
    A, B, _ = operands(M, N, K, a_k, b_k)
    Am, Bm = (A if a_k else A.T), (B.T if b_k else B)          # views: [M][K], [K][N]
    ax = which.split()[-1]
    n = {"m": M, "n": N, "k": K}[ax]
    f = decades(n, d)
    if which.startswith("one"):
        f = np.where(np.arange(n) == n // 3, 10.0 ** -d, 1.0)
    elif which.startswith("half"):
        f = np.where(np.arange(n) < n // 2, 10.0 ** -d, 1.0)
    elif which.startswith("large"):
        f *= 1e35
    if ax == "m":
        Am *= f.astype(np.float32)[:, None]
    elif ax == "n":
        Bm *= f.astype(np.float32)[None, :]
    else:
        Am *= f.astype(np.float32)[None, :]
        if compensated:
            Bm *= (1.0 / f).astype(np.float32)[:, None]
    D = product(ctx, A, B, a_k, b_k)
    ref = Am.astype(np.float64) @ Bm.astype(np.float64)
    bound = np.abs(Am).astype(np.float64) @ np.abs(Bm).astype(np.float64)
    assert np.all(np.abs(D - ref) <= 2e-6 * bound)             # (the bound of test_against_float64)
    rows, cols = np.linalg.norm(D - ref, axis=1), np.linalg.norm(D - ref, axis=0)
    assert np.all(rows <= 2e-6 * np.linalg.norm(ref, axis=1)) and np.all(cols <= 2e-6 * np.linalg.norm(ref, axis=0))


@pytest.mark.parametrize("shape", [(300, 200, 333), (26, 803, 4001), (700, 65, 64)])
@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
def test_sparse_operands_with_a_small_row_or_column(ctx, shape, a_k, b_k):
    """Mostly zeros, and one column of A of 10^-12 against a row of B of 10^12: (also where K is cut into slices)."""
    M, N, K = shape
    A, B, _ = operands(M, N, K, a_k, b_k)
    Am, Bm = (A if a_k else A.T), (B.T if b_k else B)
    Am *= np.random.Generator(np.random.PCG64(1)).random((M, K)) < 0.2
    Am[:, K // 2] *= np.float32(1e-12)
    Bm[K // 2] *= np.float32(1e12)
    D = product(ctx, A, B, a_k, b_k)
    ref = Am.astype(np.float64) @ Bm.astype(np.float64)
    bound = np.abs(Am).astype(np.float64) @ np.abs(Bm).astype(np.float64)
    assert np.all(np.abs(D - ref) <= 2e-6 * bound)


def test_zero_operands(ctx):
    A, B, _ = operands(300, 140, 200, True, True)
    assert not product(ctx, np.zeros_like(A), B, True, True).any()
    assert not product(ctx, A, np.zeros_like(B), True, True).any()


@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
def test_infinities_and_nan_as_in_any_fp32_sum(ctx, a_k, b_k):
    A, B, _ = operands(300, 140, 200, a_k, b_k)
    Am, Bm = (A if a_k else A.T), (B.T if b_k else B)
    Am[7, 11], Am[290, 3], Am[130, 199], Bm[5, 100] = np.inf, np.nan, -np.inf, -np.inf
    Bm[11, 20] = 0.0                          # inf * 0
    D = product(ctx, A, B, a_k, b_k)
    with np.errstate(invalid="ignore"):
        ref = np.stack([(Am[i].astype(np.float64)[:, None] * Bm.astype(np.float64)).sum(0) for i in range(300)])
    ok = np.isfinite(ref)
    assert ok.sum() == (300 - 3) * 139
    assert np.array_equal(D[~ok], ref[~ok], equal_nan=True)
    assert np.linalg.norm(D[ok] - ref[ok]) <= 1e-6 * np.linalg.norm(ref[ok])


def test_an_infinite_pre_activation_is_a_saturated_unit(ctx):
    """... through the epilogue: the sigmoid of an infinite sum is 0 or 1."""
    import torch
    A, B, ref = operands(260, 130, 100, True, True)
    A[3, 4], A[200, 9] = np.inf, -np.inf
    D = ctx.debug_gemm_epilogue(8, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), sigmoid=True).cpu().numpy()
    want = 1.0 / (1.0 + np.exp(-ref))
    want[3], want[200] = B[:, 4] > 0, B[:, 9] < 0
    assert np.max(np.abs(D - want)) <= 1e-5


@pytest.mark.parametrize("d", [4, 6, 8, 10])
def test_unnormalised_features(d):
    """Features over d decades with the first layer's weights scaled the other way: the gradient and the product, column by
    column of the first weight block (each belongs to one feature)."""
    import torch
    import paper_1802_00130_b200 as gn
    from oracle import gn_oracle as orc
    w = (200, 164, 5)
    p = wl.make_custom(w, 1500, 1100, 15.0, seed=4)
    f = decades(200, d)
    X = (p["X"] * f[None, :]).astype(np.float32)
    th, v = p["theta"].copy(), p["v"].copy()
    for t in (th, v):
        t[: 200 * 164] = (t[: 200 * 164].reshape(164, 200) / f[None, :]).astype(np.float32).ravel()
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    C = 1e30                                  # (the regularisation terms would hide the small columns)
    c = gn.GnContext(list(w), C, dev(X), dev(p["Y"]))
    c.profile(True)
    c.set_theta(dev(th))
    c.set_subsample(dev(p["idx"]))
    for got, want in ((c.grad(), orc.grad(th, w, C, X, p["Y"])), (c.Gv(dev(v)), orc.Gv(th, w, C, X[p["idx"]], v))):
        got, want = (np.asarray(a, np.float64)[: 200 * 164].reshape(164, 200) for a in (got.cpu().numpy(), want))
        assert np.all(np.linalg.norm(got - want, axis=0) <= 1e-5 * np.linalg.norm(want, axis=0))
    assert c.profile_read()["tensor_x3"]["launches"] > 0
    c.close()


@pytest.mark.parametrize("widths", [(37, 129, 131, 3), (617, 203, 150, 26), (50, 300, 17)])
@pytest.mark.parametrize("mode", ["fp32", "tf32"])
def test_products_and_gradient_of_ragged_networks(widths, mode):
    """Rows that are no multiple of four floats, in both modes: every contraction is computed to FP32 accuracy."""
    import torch
    import paper_1802_00130_b200 as gn
    from oracle import gn_oracle as orc
    p = wl.make_custom(widths, 1100, 777, 11.0, seed=widths[0])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    c = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]), gn.GN_TF32 if mode == "tf32" else gn.GN_FP32_ACCURATE)
    c.set_theta(dev(p["theta"]))
    c.set_subsample(dev(p["idx"]))
    th, w, C, XS = p["theta"], p["widths"], p["C"], p["X"][p["idx"]]
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
    tol = 1e-5 if mode == "fp32" or all(k % 4 for k in widths[:-1]) else 2e-3
    assert rel(c.Gv(dev(p["v"])), orc.Gv(th, w, C, XS, p["v"])) <= tol
    assert rel(c.grad(), orc.grad(th, w, C, p["X"], p["Y"])) <= tol
    assert rel(c.Gv_blockdiag(dev(p["v"])), orc.Gv_blockdiag(th, w, C, XS, p["v"])) <= tol
    c.close()


@pytest.mark.parametrize("mode", ["fp32", "tf32"])
def test_a_captured_product_follows_theta_and_the_subsample(mode):
    """A caller's own graph of a product, replayed after theta and the subsample have changed: the parts of theta and of
    the stored activations that the context keeps must be made inside the graph, not taken from before it."""
    import torch
    import paper_1802_00130_b200 as gn
    from oracle import gn_oracle as orc
    p = wl.make_custom((301, 403, 205, 5), 1500, 900, 15.0, seed=3)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    X, Y, v = dev(p["X"]), dev(p["Y"]), dev(p["v"])
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    ctx = gn.GnContext(p["widths"], p["C"], X, Y, gn.GN_TF32 if mode == "tf32" else gn.GN_FP32_ACCURATE, stream=stream)
    out = torch.empty_like(v)
    ctx.set_theta(dev(p["theta"]))
    ctx.set_subsample(dev(p["idx"]))
    ctx.Gv(v, out=out)                        # every workspace exists
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ctx.Gv(v, out=out)
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
    plain = torch.empty_like(v)
    for k in range(3):
        th = (p["theta"] * (1.0 + 0.5 * k)).astype(np.float32)
        idx = np.roll(np.arange(1500, dtype=np.int32), 37 * k)[:900].copy()
        ctx.set_theta(dev(th))
        ctx.set_subsample(dev(idx))
        graph.replay()
        torch.cuda.synchronize()
        ref = orc.Gv(th, p["widths"], p["C"], p["X"][idx], p["v"])
        assert rel(out, ref) <= 1e-5
        ctx.Gv(v, out=plain)                  # and a plain call after it
        torch.cuda.synchronize()
        assert rel(plain, ref) <= 1e-5
    ctx.close()


@pytest.mark.parametrize("first,second", [(0, 1), (1, 0)])
@pytest.mark.parametrize("blockdiag", [False, True])
def test_a_kept_solver_step_follows_the_accurate_method(blockdiag, first, second):
    """A fixed-length solve replays a captured step and keeps it for later solves.  After theta, the subsample and the way
    FP32-accurate contractions are computed have changed, the step of before must not run on the parts it was captured with."""
    import torch
    import paper_1802_00130_b200 as gn
    from oracle import gn_oracle as orc
    p = wl.make_custom((301, 403, 205, 5), 1500, 900, 15.0, seed=3)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ctx = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]))
    d = torch.empty(p["theta"].size, device="cuda")
    for k, method in enumerate((first, second, first)):
        th = (p["theta"] * (1.0 + 0.5 * k)).astype(np.float32)
        idx = np.roll(np.arange(1500, dtype=np.int32), 37 * k)[:900].copy()
        ctx.set_accurate_method(method)
        ctx.set_theta(dev(th))
        ctx.set_subsample(dev(idx))
        g = orc.grad(th, p["widths"], p["C"], p["X"], p["Y"])
        replays = ctx.graph_replays
        ctx.cg_solve(dev(g.astype(np.float32)), 1.0, blockdiag=blockdiag, max_iter=5, tol=0.0, out=d)
        assert ctx.graph_replays - replays == 4
        ref = orc.cg_solve(th, p["widths"], p["C"], p["X"][idx], g, 1.0, blockdiag, 5, 0.0)[0]
        # products within 1e-6, multiplied a few times by the five steps (systems of condition below 100)
        assert np.linalg.norm(d.cpu().numpy() - ref) <= 1e-4 * np.linalg.norm(ref)
    ctx.close()


def test_kept_parts_do_not_accumulate():
    """Parts of theta and of the activations are kept per place: neither new variable partitions nor new subsample sizes may
    leave the parts of the old ones behind."""
    import torch
    import paper_1802_00130_b200 as gn
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    p = wl.make_custom((1201, 802, 605, 5), 1500, 900, 15.0, seed=3)
    ctx = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]))
    ctx.set_theta(dev(p["theta"]))
    ctx.set_subsample(dev(p["idx"]))
    ctx.profile(True)
    v, seen = dev(p["v"]), []
    for s in [[4, 1, 1, 1], [3, 1, 1, 1], [2, 1, 1, 1]]:      # (the largest workspaces first; the parts take about the same each time)
        ctx.set_split(s)
        ctx.Gv_blockdiag(v)
        torch.cuda.synchronize()
        seen.append(ctx.workspace_bytes)
    assert ctx.profile_read()["tensor_x3"]["launches"] > 0
    parts = 4 * 900 * 1201
    assert max(seen) <= seen[0] + parts // 4
    ctx.close()


def test_parts_of_narrow_layers_do_not_accumulate_over_subsample_sizes():
    import torch
    import paper_1802_00130_b200 as gn
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    p = wl.make_custom((96, 64, 60, 10), 9000, 9000, 15.0, seed=3)
    ctx = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]), gn.GN_TF32)
    ctx.debug_option(10, 0)
    ctx.set_blockdiag_method(2)
    ctx.set_theta(dev(p["theta"]))
    v, seen = dev(p["v"]), []
    for nS in (9000, 8800, 8600, 8400, 8200):
        ctx.set_subsample(dev(p["idx"][:nS]))
        ctx.Gv_blockdiag(v)
        seen.append(ctx.workspace_bytes)
    assert len(set(seen)) == 1
    ctx.close()


def test_parts_take_the_memory_of_the_layers_that_are_split():
    """A TF32 context with one odd layer: the parts of that layer's activations, not of all."""
    import torch
    import paper_1802_00130_b200 as gn
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    w, nS = (30, 1024, 1024, 20), 20000
    p = wl.make_custom(w, 500, 500, 15.0, seed=3)
    ctx = gn.GnContext(list(w), p["C"], dev(p["X"]), dev(p["Y"]), gn.GN_TF32)
    ctx.set_theta(dev(p["theta"]))
    ctx.profile(True)
    ctx.set_subsample(dev(np.resize(p["idx"], nS)))
    v = dev(p["v"])
    ctx.Gv(v)
    assert ctx.profile_read()["tensor_x3"]["launches"] > 0
    activations = 4 * nS * (2 * sum(w) + sum(w[:-1]))          # Z, RZ, DS
    odd = 2 * 4 * nS * 32 + 4 * nS * 1024                      # parts of X_S (rows of 8), and of delta s^1 for the length of a contraction
    assert ctx.workspace_bytes <= activations + odd + 100e6    # (weights, vectors, the K slices' workspace: 50 MB)
    ctx.close()


def test_stored_activations_beyond_the_limit_of_passing_operands():
    """Z^1 of 1.6e9 elements (6.5 GB): its contractions stay on the tensor cores."""
    import torch
    import paper_1802_00130_b200 as gn
    from oracle import gn_oracle as orc
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    w, nS = (64, 4096, 20), 400000
    p = wl.make_custom(w, 1000, 1000, 15.0, seed=3)
    ctx = gn.GnContext(list(w), p["C"], dev(p["X"]), dev(p["Y"]))
    ctx.set_theta(dev(p["theta"]))
    ctx.profile(True)
    ctx.set_subsample(dev(np.resize(np.arange(1000, dtype=np.int32), nS)))
    kinds = ctx.profile_read()
    assert kinds["ffma"]["launches"] == 0 and kinds["tensor_x3"]["launches"] == 2
    z = ctx.debug_activations(2).reshape(nS, 20)
    ref = orc.forward(p["theta"], list(w), p["X"])[2]
    for at in (0, 200000, nS - 1000):
        assert np.linalg.norm(z[at:at + 1000].cpu().numpy() - ref) <= 1e-6 * np.linalg.norm(ref)
    ctx.close()
    torch.cuda.empty_cache()
