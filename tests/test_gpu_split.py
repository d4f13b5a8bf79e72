"""The FP64 M2L as split integer products on the tensor cores: sizes at the edges of its row
tiles (48 and 64 complex rows, more than one tile), coefficient chunks (24, 16) and segments,
its column groups (16, 32 and ragged), and values at the ends of the double range."""

import numpy as np
import pytest

from oracle import nystrom as onys
from workloads import Medium, circle, layered_small

pytestmark = pytest.mark.gpu


def relerr(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def free_space(lf, p):
    bodies = [circle(-1.1, 0.3, 0.5, 90), circle(0.9, -0.4, 0.6, 110), circle(0.2, 1.4, 0.3, 70)]
    med = Medium(interfaces=[], k=[3.0], eta=[1.0])
    pts, w, _, _ = onys.elements(bodies)
    M = lf.medium_create(med.interfaces, med.k, med.eta)
    return med, pts, w, lf.geometry_build(M, pts, w, p=p, leaf_size=8)


# 2p+1 = 11, 41, 47, 49 (one and several segments), 63, 65 (one and two tiles), 97, 129
@pytest.mark.parametrize("p", [5, 20, 23, 24, 31, 32, 48, 64])
def test_orders_against_dense(gpu_lib, p):
    lf = gpu_lib
    med, pts, w, G = free_space(lf, p)
    tp = lf.geometry_query(G, "tree_params", np.float64)
    assert tp[4] <= tp[3], "the far field must be active"
    rng = np.random.default_rng(p)
    x = rng.standard_normal(G.n) + 1j * rng.standard_normal(G.n)
    ref = onys.dense_matrix(med, pts, w, reaction=False) @ x
    # truncation: cells a width apart, ratio sqrt(2) / (4 - sqrt(2)) = 0.547 per order; rounding
    # of some thousand terms with a margin of 10^3: 1e-10
    assert relerr(lf.matvec(G, x), ref) <= 0.547 ** (p + 1) + 1e-10


def test_columns_equal_single_products(gpu_lib):
    lf = gpu_lib
    wl = layered_small(n_bodies=3, nodes=150, seed=7)
    pts, w, _, _ = onys.elements(wl.bodies)
    M = lf.medium_create(wl.medium.interfaces, wl.medium.k, wl.medium.eta)
    G = lf.geometry_build(M, pts, w, p=20, leaf_size=16)
    rng = np.random.default_rng(3)
    for nrhs in (2, 17, 33):
        X = np.asfortranarray(rng.standard_normal((G.n, nrhs)) + 1j * rng.standard_normal((G.n, nrhs)))
        Y = lf.matvec(G, X)
        for c in (0, 1, nrhs - 1):
            assert np.array_equal(Y[:, c], lf.matvec(G, X[:, c].copy()))


def test_scales_zeros_and_values_that_are_not_finite(gpu_lib):
    lf = gpu_lib
    wl = layered_small(n_bodies=3, nodes=150, seed=7)
    pts, w, _, _ = onys.elements(wl.bodies)
    M = lf.medium_create(wl.medium.interfaces, wl.medium.k, wl.medium.eta)
    G = lf.geometry_build(M, pts, w, p=20, leaf_size=16)
    rng = np.random.default_rng(4)
    x = rng.standard_normal(G.n) + 1j * rng.standard_normal(G.n)
    y = lf.matvec(G, x)
    # powers of two pass through every exponent exactly (the leaf values of order 20 are 1e-38
    # of x and their largest factors 1e40, so +-100 stays inside the double range)
    for e in (-100, 100):
        assert np.array_equal(lf.matvec(G, x * 2.0 ** e), y * 2.0 ** e)
    assert not np.any(lf.matvec(G, np.zeros_like(x)))
    for bad in (np.nan, np.inf):
        xb = x.copy()
        xb[5] = bad
        assert not np.any(np.isfinite(lf.matvec(G, xb)))
    assert np.array_equal(lf.matvec(G, x), y)


def test_passes_as_products_in_blocks_and_batches(gpu_lib):
    """A geometry whose finest M2M and L2L passes are products too (over 1,200 families): a block's
    columns, and its share of a batch with a small geometry, equal its own single products."""
    import torch

    from workloads import config_c2

    lf = gpu_lib
    geos = []
    for wl, leaf in ((config_c2(), 64), (layered_small(n_bodies=3, nodes=150, seed=7), 16)):
        pts, w, _, _ = onys.elements(wl.bodies)
        M = lf.medium_create(wl.medium.interfaces, wl.medium.k, wl.medium.eta)
        geos.append(lf.geometry_build(M, pts, w, p=20, leaf_size=leaf))
    rng = np.random.default_rng(6)
    xs = [torch.from_numpy(rng.standard_normal((3, G.n)) + 1j * rng.standard_normal((3, G.n))).cuda() for G in geos]
    own = [torch.stack([lf.matvec(G, x[c].contiguous()) for c in range(3)]) for G, x in zip(geos, xs)]
    for G, x, y in zip(geos, xs, own):
        assert torch.equal(lf.matvec(G, x), y)
    for order in (slice(None), slice(None, None, -1)):
        for y, ref in zip(lf.matvec_batch(geos[order], xs[order]), own[order]):
            assert torch.equal(y, ref)
    single = [x[0].contiguous() for x in xs]
    for y, ref in zip(lf.matvec_batch(geos, single), own):
        assert torch.equal(y, ref[0])


def test_coarse_levels_beside_the_fp32_ones(gpu_lib):
    """Precision form: the coarse levels' chain on its own stream, beside the FP32 M2L (SIMT and, from
    16 columns, on the tensor cores), gives the bits of the chain in one stream (stage timers on)."""
    import torch

    from workloads import layered_wide

    lf = gpu_lib
    wl = layered_wide()
    pts, w, _, _ = onys.elements(wl.bodies)
    M = lf.medium_create(wl.medium.interfaces, wl.medium.k, wl.medium.eta)
    G, S = (lf.geometry_build(M, pts, w, p=20, leaf_size=8, profile=prof) for prof in (False, True))
    rng = np.random.default_rng(8)
    for cols in (1, 5, 20):
        X = torch.from_numpy(rng.standard_normal((cols, G.n)) + 1j * rng.standard_normal((cols, G.n))).cuda()
        ref = lf.matvec(S, X, mixed=True)
        for _ in range(5):
            assert torch.equal(lf.matvec(G, X, mixed=True), ref)
    lm = lf.geometry_query(G, "precision_form", np.float64)[0]
    assert lm > lf.geometry_query(G, "tree_params", np.float64)[4], "coarse levels must be in use"
