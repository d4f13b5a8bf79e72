"""The reaction moment tables: orders at the edges of their kernels' splits.  A same-layer
table's 4p + 1 moments are summed by groups of threads (12 at p = 5, two at 31, one from 32 on,
two moments per thread from 64 on); a cross-layer table's entries go in one run (p <= 21) or
several, its nodes in one range (p = 5) or several."""

import numpy as np
import pytest

from oracle import nystrom as onys
from workloads import Medium, circle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def layers():
    med = Medium(interfaces=[0.0, -0.5], k=[2.0, 3.0, 2.5], eta=[1.0, 2.0, 1.5])
    bodies = [circle(-1.1, 0.45, 0.4, 50), circle(0.9, 0.5, 0.35, 50), circle(-0.8, -1.0, 0.4, 50),
              circle(1.0, -0.95, 0.35, 50)]
    pts, w, _, _ = onys.elements(bodies)
    rng = np.random.default_rng(17)
    x = rng.standard_normal(len(w)) + 1j * rng.standard_normal(len(w))
    return med, pts, w, x, onys.dense_matrix(med, pts, w) @ x


@pytest.mark.parametrize("p", [5, 20, 31, 32, 63, 64])
def test_orders_against_dense(gpu_lib, layers, p):
    lf = gpu_lib
    med, pts, w, x, ref = layers
    G = lf.geometry_build(lf.medium_create(med.interfaces, med.k, med.eta), pts, w, p=p, leaf_size=8)
    keys = lf.geometry_query(G, "reaction_tables", np.float64).reshape(-1, 8)
    work = lf.geometry_query(G, "table_work", np.float64)
    assert len(keys) > 0 and work[0] > 0 and work[1] > 0, "both kinds of tables must be in use"
    assert not np.any(lf.geometry_query(G, "nonfinite", np.float64))
    # truncation: cells a width apart, ratio sqrt(2) / (4 - sqrt(2)) = 0.547 per order; the
    # tables' quadrature rule agrees with the dense matrix to some 3e-10, with a margin of 10
    err = np.linalg.norm(lf.matvec(G, x) - ref) / np.linalg.norm(ref)
    assert err <= 0.547 ** (p + 1) + 3e-9
    G.destroy()
