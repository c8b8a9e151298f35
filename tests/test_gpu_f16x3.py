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


def test_wide_range_inside_an_operand(ctx):
    """Rows of A over twelve decades: every row is as accurate as an absolute error of 2^-40 max|A| per element leaves it."""
    A, B, _ = operands(256, 64, 320, True, False)
    scale = 10.0 ** -np.linspace(0, 12, 256)
    A = (A * scale[:, None]).astype(np.float32)
    ref = A.astype(np.float64) @ B.astype(np.float64)
    err = np.linalg.norm(product(ctx, A, B, True, False) - ref, axis=1)
    bound = 1e-6 * np.linalg.norm(ref, axis=1) + 2.0 ** -40 * np.abs(A).max() * np.linalg.norm(B)
    assert np.all(err <= bound)


def test_zero_operands_and_non_finite_elements(ctx):
    A, B, ref = operands(300, 140, 200, True, True)
    assert not product(ctx, np.zeros_like(A), B, True, True).any()
    assert not product(ctx, A, np.zeros_like(B), True, True).any()
    A[7, 11], A[290, 3], B[100, 5] = np.inf, np.nan, -np.inf
    D = product(ctx, A, B, True, True)
    bad = np.zeros(D.shape, bool)
    bad[[7, 290], :] = True
    bad[:, 100] = True
    assert not np.isfinite(D[bad]).any()      # as in any FP32 sum: the rows and the column that meet them, and no others
    assert np.linalg.norm(D[~bad] - ref[~bad]) <= 1e-6 * np.linalg.norm(ref[~bad])


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
