"""Block right-hand sides: more columns than the products' workspace holds at once (rounds), and widths
that alternate between calls, also inside captured graphs."""

import numpy as np
import pytest

from oracle import nystrom as onys
from workloads import Medium, circle, config_c2, layered_small

pytestmark = pytest.mark.gpu


def geometry(lf, wl, leaf):
    pts, w, _, _ = onys.elements(wl.bodies)
    M = lf.medium_create(wl.medium.interfaces, wl.medium.k, wl.medium.eta)
    return lf.geometry_build(M, pts, w, p=20, leaf_size=leaf)


def columns(n, cols, seed):
    import torch

    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn((cols, n, 2), dtype=torch.float64, device="cuda", generator=g))


def launches(lf, G):
    return int(lf.geometry_query(G, "launch_count", np.float64)[0])


def test_rounds_equal_single_products(gpu_lib):
    """45 columns of 65,536 points: 66 MB of workspace each, so 2 GiB takes them in two rounds (23 + 22)."""
    import torch

    lf = gpu_lib
    G = geometry(lf, config_c2(), 64)
    X = columns(G.n, 45, 1)
    count = []
    for cols in (5, 45):
        l0 = launches(lf, G)
        Y = lf.matvec(G, X[:cols].contiguous())
        count.append(launches(lf, G) - l0)
    assert count[1] > count[0], "more than one round must be in use"
    for c in (0, 1, 21, 22, 23, 44):
        assert torch.equal(Y[c], lf.matvec(G, X[c].contiguous()))
    small = geometry(lf, layered_small(n_bodies=3, nodes=150, seed=7), 16)
    xs = columns(small.n, 2, 2)
    yb, ys = lf.matvec_batch([G, small], [X, xs])
    assert torch.equal(yb, Y) and torch.equal(ys, lf.matvec(small, xs))


def test_captured_static_product_outlives_wider_blocks(gpu_lib):
    """A captured allocation-free product keeps its workspace when blocks make the geometry's grow."""
    import torch

    lf = gpu_lib
    G = geometry(lf, layered_small(n_bodies=3, nodes=150, seed=7), 16)
    x, y = columns(G.n, 1, 7)[0], torch.empty(G.n, dtype=torch.complex128, device="cuda")
    lf.matvec_static(G, x, y)
    torch.cuda.synchronize()
    ref = y.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lf.matvec_static(G, x, y)
    other = []
    for cols in (2, 9, 40):
        X = columns(G.n, cols, 10 + cols)
        other.append((X, lf.matvec(G, X)))
        y.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
        for X, Y in other:   # nothing of theirs was written by the replay
            assert torch.equal(lf.matvec(G, X), Y)


def test_captured_products_outlive_other_widths(gpu_lib):
    """A warmed-up width can be captured whatever width ran last, and its graph stays valid while
    narrower products run."""
    import torch

    lf = gpu_lib
    G = geometry(lf, layered_small(n_bodies=3, nodes=150, seed=7), 16)
    X, Y = columns(G.n, 5, 3), columns(G.n, 5, 4)
    narrow = columns(G.n, 3, 5)
    ref5, ref3 = lf.matvec(G, X), lf.matvec(G, narrow)
    new = columns(G.n, 5, 6)
    ref_new = lf.matvec(G, new)
    assert torch.equal(lf.matvec(G, narrow), ref3)   # the width used last is not the captured one
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lf.matvec(G, X, Y)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, ref5)
    for _ in range(3):
        assert torch.equal(lf.matvec(G, narrow), ref3)
        assert torch.equal(lf.matvec(G, X[:2].contiguous()), ref5[:2])
    X.copy_(new)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, ref_new)


def test_precision_form_holds_its_own_levels_only(gpu_lib):
    """The precision form's FP64 products are those of the levels above its FP32 ones: 3 MB of workspace
    per column at 65,536 points, where all levels take 66 MB.  Beside it a column holds its FP64 and
    FP32 expansions (18 MB), sorted vectors and partial sums (some 8 MB): below 50 MB in all.  The
    result is that of a geometry whose blocks have products of all levels already."""
    import torch

    lf = gpu_lib
    cols = 32
    G = geometry(lf, config_c2(), 64)
    X = columns(G.n, cols, 1)
    Y = torch.empty_like(X)
    lf.matvec(G, X[0].contiguous(), mixed=True)   # the form's tables
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    lf.matvec(G, X, Y, mixed=True)
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= cols * (50 << 20)
    S = geometry(lf, config_c2(), 64)
    lf.matvec(S, X)
    assert torch.equal(lf.matvec(S, X, mixed=True), Y)
    five = X[:5].contiguous()
    ref = lf.matvec(G, five, mixed=True)
    lf.matvec(S, five)
    assert torch.equal(lf.matvec(S, five, mixed=True), ref)


@pytest.mark.parametrize("far", [False, True])
def test_blocks_wider_than_a_grid(gpu_lib, far):
    """More columns than a launch's grid holds: 65,535 groups of four in the near field, of one in the
    evaluation of locals of order 41 and more."""
    import torch

    lf = gpu_lib
    med = Medium(interfaces=[], k=[3.0], eta=[1.0])
    bodies = [circle(-1.0, 0.2, 0.3, 12), circle(1.1, -0.1, 0.3, 12)]
    pts, w, _, _ = onys.elements(bodies)
    G = lf.geometry_build(lf.medium_create(med.interfaces, med.k, med.eta), pts, w, p=41 if far else 20,
                          leaf_size=4 if far else 64)
    tp = lf.geometry_query(G, "tree_params", np.float64)
    assert (tp[4] <= tp[3]) == far
    cols = 66000 if far else 262145
    X = columns(G.n, cols, 9)
    K = torch.from_numpy(onys.dense_matrix(med, pts, w, reaction=False)).cuda()
    ref = X @ K.T
    Y = lf.matvec(G, X)
    # truncation far below (0.547^42), rounding of 24 terms with a margin
    assert float((Y - ref).abs().max()) <= 1e-9 * float(ref.abs().max())
    for c in (0, cols - 1):
        assert torch.equal(Y[c], lf.matvec(G, X[c].contiguous()))
