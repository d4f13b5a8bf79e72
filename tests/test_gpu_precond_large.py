"""The preconditioner for neighbourhoods whose panel does not fit shared memory."""

import numpy as np
import pytest

from oracle import nystrom as onys
from workloads import Medium, circle

pytestmark = pytest.mark.gpu


def test_neighbourhood_beyond_the_shared_panel(gpu_lib):
    """Four leaves of 820 points, all neighbours of each other: every leaf's local matrix is the whole
    one of 3,280 points, so the preconditioner is its inverse."""
    lf = gpu_lib
    med = Medium(interfaces=[], k=[3.0], eta=[1.0])
    bodies = [circle(x, y, 0.4, 820) for x in (-0.7, 0.7) for y in (-0.6, 0.6)]
    pts, w, _, _ = onys.elements(bodies)
    G = lf.geometry_build(lf.medium_create(med.interfaces, med.k, med.eta), pts, w, p=20, leaf_size=1024)
    tp = lf.geometry_query(G, "tree_params", np.float64)
    assert tp[3] == 1 and tp[5] == 5, "one root and four leaves"
    K = onys.dense_matrix(med, pts, w, reaction=False)
    rng = np.random.default_rng(1)
    v = rng.standard_normal(G.n) + 1j * rng.standard_normal(G.n)
    ref = np.linalg.solve(K, v)
    # condition number some 1e4 (first kind, 820 elements a body) times FP64 rounding, with a margin
    assert np.abs(lf.precond_apply(G, v) - ref).max() <= 1e-10 * np.abs(ref).max()
