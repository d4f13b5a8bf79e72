"""The leaves' kernels at their edges: near-field rows beyond one CTA's 64 and every number of
threads per row, multipoles and locals of leaves beyond one round of 64 points, and the
preconditioner's blocked elimination for neighbourhoods around its 16-column blocks."""

import numpy as np
import pytest

from oracle import combined as ocf
from oracle import nystrom as onys
from oracle import tree as otree
from workloads import Medium, circle, layered_small

pytestmark = pytest.mark.gpu


def relerr(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def bodies_far_apart():
    return [circle(-2.6, 0.4, 0.5, 190), circle(2.4, -0.7, 0.4, 170), circle(0.1, 3.1, 0.3, 75)]


# leaves of 1..3, up to 31, 65, 131 points, and one leaf with every point (no far field)
@pytest.mark.parametrize("combined", [False, True])
@pytest.mark.parametrize("leaf", [3, 31, 65, 131, 1000])
def test_leaf_sizes_against_dense(gpu_lib, leaf, combined):
    lf = gpu_lib
    med = Medium(interfaces=[], k=[3.0], eta=[1.0])
    pts, w, nrm, _ = onys.elements(bodies_far_apart())
    M = lf.medium_create(med.interfaces, med.k, med.eta)
    G = lf.geometry_build(M, pts, w, nrm if combined else None, p=30, leaf_size=leaf, combined=combined)
    K = ocf.dense_matrix_cf(med, pts, w, nrm) if combined else onys.dense_matrix(med, pts, w, reaction=False)
    rng = np.random.default_rng(leaf)
    X = np.asfortranarray(rng.standard_normal((G.n, 6)) + 1j * rng.standard_normal((G.n, 6)))
    Y = lf.matvec(G, X)
    for c in range(6):
        # truncation 0.547^31 = 8e-9 (a dipole's terms 31 times that), rounding far below
        assert relerr(Y[:, c], K @ X[:, c]) <= 2.5e-7
    assert np.array_equal(lf.matvec(G, X[:, 5].copy()), Y[:, 5])


# neighbourhoods from a few points to all 450 of the geometry (blocks of 16 columns, clusters)
@pytest.mark.parametrize("leaf", [2, 5, 16, 60, 200, 500])
def test_preconditioner_neighbourhoods(gpu_lib, leaf):
    lf = gpu_lib
    wl = layered_small(n_bodies=3, nodes=150, seed=7)
    med = wl.medium
    pts, w, _, _ = onys.elements(wl.bodies)
    M = lf.medium_create(med.interfaces, med.k, med.eta)
    G = lf.geometry_build(M, pts, w, p=20, leaf_size=leaf)
    T = otree.Tree(pts, med.interfaces, med.k, p=20, leaf_size=leaf)
    P = otree.dd_preconditioner_dense(T, pts, w, med.k, onys.self_term(np.asarray(med.k)[onys.layer_of(med, pts[:, 1])], w))
    rng = np.random.default_rng(leaf)
    v = rng.standard_normal(G.n) + 1j * rng.standard_normal(G.n)
    ref = P @ v
    # condition numbers up to about 1e3 times FP64 rounding, with a margin
    assert np.abs(lf.precond_apply(G, v) - ref).max() <= 1e-11 * np.abs(ref).max()
