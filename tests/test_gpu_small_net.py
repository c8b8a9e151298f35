"""Passes of small networks that run as one launch (product, block-diagonal product, loss, gradient, stored forward pass)
against the float64 checker: fewer rows than a block takes, exactly a block, one more; one layer to the most layers the
launch takes; widths of one; both precision modes (the pass is FP32 in both)."""
import numpy as np
import pytest

import gn_workloads as wl
from oracle import gn_oracle as orc

pytestmark = pytest.mark.gpu

NETS = [(20, 16, 16, 4), (37, 53, 19, 7), (1, 1, 1), (50, 6), (9, 33, 1), (130, 40, 3), (5, 4, 7, 3, 6, 2, 8, 5, 2), (64, 64, 64, 64, 10)]


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("mode", ["fp32", "tf32"])
@pytest.mark.parametrize("nS,l", [(1, 3), (31, 64), (32, 33), (33, 1000), (500, 700)])
@pytest.mark.parametrize("widths", NETS)
def test_against_float64(widths, nS, l, mode):
    import paper_1802_00130_b200 as gn
    p = wl.make_custom(widths, l, nS, 0.3 * l, seed=sum(widths) + l)
    ctx = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]), gn.GN_TF32 if mode == "tf32" else gn.GN_FP32_ACCURATE)
    th, w, C, XS, v = p["theta"], p["widths"], p["C"], p["X"][p["idx"]], p["v"]
    ctx.set_theta(dev(th))
    before = ctx.kernel_launches
    ctx.set_subsample(dev(p["idx"]))
    assert ctx.kernel_launches - before == 1
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy() - b) / np.linalg.norm(b)
    g, f = ctx.grad(with_f=True)
    # sums of at most 130 terms in FP32 (2^-24 each), three passes deep; the sums over blocks are in double
    assert rel(ctx.Gv(dev(v)), orc.Gv(th, w, C, XS, v)) <= 2e-6
    assert ctx.kernel_launches - before == 1 + 2 + 2
    ref_g = orc.grad(th, w, C, p["X"], p["Y"])
    assert rel(g, ref_g) <= 2e-6
    ref_f = orc.fun(th, w, C, p["X"], p["Y"])
    assert abs(f - ref_f) <= 2e-6 * abs(ref_f) and ctx.fun() == f
    ref_b = orc.Gv_blockdiag(th, w, C, XS, v)
    assert rel(ctx.Gv_blockdiag(dev(v)), ref_b) <= 2e-6
    Z = orc.forward(th, w, XS)
    for m in range(1, len(w)):
        z = ctx.debug_activations(m).cpu().numpy().reshape(nS, w[m])
        assert np.max(np.abs(z - Z[m])) <= 2e-6 * max(1.0, np.max(np.abs(Z[m])))
    ctx.debug_option(10, 0)                   # one contraction per layer: the same within the mode's bound
    assert rel(ctx.Gv(dev(v)), orc.Gv(th, w, C, XS, v)) <= (1e-5 if mode == "fp32" else 2e-3)
    ctx.close()


@pytest.mark.parametrize("mode", ["fp32", "tf32"])
@pytest.mark.parametrize("nS,l", [(1, 3), (33, 1000), (500, 700)])
@pytest.mark.parametrize("widths", NETS)
def test_the_chain_of_kernels_at_the_same_sizes(widths, nS, l, mode):
    """The same networks with the one-launch passes switched off: the contraction, streaming, column-sum, gather, loss and
    vector kernels at odd and tiny sizes, in every pass and in both solves."""
    import paper_1802_00130_b200 as gn
    p = wl.make_custom(widths, l, nS, 0.3 * l, seed=sum(widths) + l)
    ctx = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]), gn.GN_TF32 if mode == "tf32" else gn.GN_FP32_ACCURATE)
    ctx.debug_option(10, 0)
    th, w, C, XS, v = p["theta"], p["widths"], p["C"], p["X"][p["idx"]], p["v"]
    tol = 1e-5 if mode == "fp32" else 2e-3    # the modes' bounds
    rel = lambda a, b: np.linalg.norm(np.asarray(a.cpu().numpy() if hasattr(a, "cpu") else a) - b) / np.linalg.norm(b)
    ctx.set_theta(dev(th))
    before = ctx.kernel_launches
    ctx.set_subsample(dev(p["idx"]))
    assert ctx.kernel_launches - before > 1
    Z = orc.forward(th, w, XS)
    for m in range(1, len(w)):
        assert rel(ctx.debug_activations(m).reshape(nS, w[m]), Z[m]) <= tol
    g, f = ctx.grad(with_f=True)
    ref_g, ref_f = orc.grad(th, w, C, p["X"], p["Y"]), orc.fun(th, w, C, p["X"], p["Y"])
    assert rel(g, ref_g) <= tol and abs(f - ref_f) <= tol * abs(ref_f) and ctx.fun() == f
    assert rel(ctx.Gv(dev(v)), orc.Gv(th, w, C, XS, v)) <= tol
    ref_b = orc.Gv_blockdiag(th, w, C, XS, v)
    for method in [1, 2] if len(w) > 2 and w[-1] <= 16 else [1]:
        ctx.set_blockdiag_method(method)
        assert rel(ctx.Gv_blockdiag(dev(v)), ref_b) <= tol
    for block in (False, True):               # two steps: what a product's rounding does to them is a few times that rounding
        d, _, _ = ctx.cg_solve(dev(ref_g.astype(np.float32)), 1.0, blockdiag=block, max_iter=2, tol=0.0)
        assert rel(d, orc.cg_solve(th, w, C, XS, ref_g, 1.0, block, 2, 0.0)[0]) <= 10 * tol
    ctx.close()


def test_an_index_out_of_range_is_still_refused():
    import paper_1802_00130_b200 as gn
    p = wl.make("tiny")
    ctx = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]))
    ctx.set_theta(dev(p["theta"]))
    for bad in (-1, p["l"]):
        idx = p["idx"].copy()
        idx[5] = bad
        with pytest.raises(gn.GnError):
            ctx.set_subsample(dev(idx))
        with pytest.raises(gn.GnError):
            ctx.Gv(dev(p["v"]))
    ctx.set_subsample(dev(p["idx"]))
    ctx.Gv(dev(p["v"]))
    ctx.close()


@pytest.mark.parametrize("widths,nS,l", [((96, 100, 50, 200, 1), 554, 5540), ((60, 40, 20, 1), 2000, 100000), ((37, 53, 19, 7), 300, 900),
                                         ((300, 120, 80, 40), 700, 40000)])
def test_tf32_solves_round_one_operator(widths, nS, l):
    """Two steps of conjugate gradient on a TF32 context where only some of the passes would fit into one launch: the
    first residual is a thousandth of the gradient, so a gradient and products that round differently show in the second
    iterate.  Bound: the products' 1e-4, times the few times by which the second step amplifies a consistent rounding."""
    import paper_1802_00130_b200 as gn
    p = wl.make_custom(widths, l, nS, float(l), seed=5, x="sparse80")
    ctx = gn.GnContext(p["widths"], p["C"], dev(p["X"]), dev(p["Y"]), gn.GN_TF32)
    ctx.set_theta(dev(p["theta"]))
    ctx.set_subsample(dev(p["idx"]))
    d, _, _ = ctx.cg_solve(ctx.grad(), 1.0, max_iter=2, tol=0.0)
    th, w, C, XS = p["theta"], p["widths"], p["C"], p["X"][p["idx"]]
    ref = orc.cg_solve(th, w, C, XS, orc.grad(th, w, C, p["X"], p["Y"]), 1.0, False, 2, 0.0)[0]
    assert np.linalg.norm(d.cpu().numpy() - ref) <= 4e-4 * np.linalg.norm(ref)
    ctx.close()
