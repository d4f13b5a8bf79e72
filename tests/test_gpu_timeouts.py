"""Time-outs (LFMM_ERR_TIMEOUT).  No wait is made to run out on the device: the test sets the word
that a kernel would set, in host memory, and looks at what the calls do with it."""

import ctypes
import threading
import time

import numpy as np
import pytest

from oracle import nystrom as onys
from workloads import config_c2, layered_wide

pytestmark = pytest.mark.gpu


def geometry(lf, wl, leaf):
    pts, w, _, _ = onys.elements(wl.bodies)
    M = lf.medium_create(wl.medium.interfaces, wl.medium.k, wl.medium.eta)
    return lf.geometry_build(M, pts, w, p=20, leaf_size=leaf)


def word(lf, G):
    address = int(lf.geometry_query(G, "wait_word", np.int64)[0])
    assert address != 0
    return ctypes.c_int32.from_address(address)


def vector(G, seed):
    import torch

    rng = np.random.default_rng(seed)
    return torch.from_numpy(rng.standard_normal(G.n) + 1j * rng.standard_normal(G.n)).cuda()


@pytest.mark.parametrize("mixed", [False, True])
def test_a_call_that_reports_a_time_out_queues_nothing(gpu_lib, mixed):
    """The earlier product's time-out is reported before any work of this one is queued (on the call's
    stream, the near field's or the precision form's coarse levels'), once, and the next call is sound."""
    import torch

    lf = gpu_lib
    G = geometry(lf, layered_wide(), 8)
    x = vector(G, 1)
    ref = lf.matvec(G, x, mixed=mixed)
    for _ in range(5):
        n0 = lf.geometry_query(G, "launch_count", np.float64)[0]
        word(lf, G).value = 1
        with pytest.raises(lf.LfmmError) as err:
            lf.matvec(G, x, mixed=mixed)
        assert err.value.status == lf.LFMM_ERR_TIMEOUT
        # the gather into the sorted order is queued by the call itself
        assert lf.geometry_query(G, "launch_count", np.float64)[0] <= n0 + 1
        assert torch.equal(lf.matvec(G, x, mixed=mixed), ref)


@pytest.mark.parametrize("cols", [1, 3])
def test_a_solve_looks_at_every_step(gpu_lib, cols):
    """A time-out of one step's product (a replayed graph, a block) ends the solve there, instead of
    after its last step or not at all."""
    lf = gpu_lib
    G = geometry(lf, config_c2(), 64)   # 300 steps take a third of a second
    rng = np.random.default_rng(2)
    b = np.asfortranarray(rng.standard_normal((G.n, cols)) + 1j * rng.standard_normal((G.n, cols)))
    b = b[:, 0].copy() if cols == 1 else b

    def solve():   # never reaches its tolerance
        t0 = time.perf_counter()
        try:
            return lf.gmres_solve(G, b, tol=1e-30, max_iter=300, precond=False), time.perf_counter() - t0
        except lf.LfmmError as e:
            return e, time.perf_counter() - t0

    solve()
    (x, info), full = solve()
    assert info["iterations"] >= 100
    w = word(lf, G)
    timer = threading.Timer(0.2 * full, lambda: setattr(w, "value", 1))
    timer.start()
    err, took = solve()
    timer.join()
    assert isinstance(err, lf.LfmmError) and err.status == lf.LFMM_ERR_TIMEOUT
    assert took <= 0.7 * full, (took, full)
    again, _ = solve()
    assert np.array_equal(again[0], x)


def test_each_geometry_of_a_batch_has_its_own_word(gpu_lib):
    """A time-out of one geometry's product is not taken for another's, alone or in a batch."""
    import torch

    lf = gpu_lib
    geos = [geometry(lf, layered_wide(), leaf) for leaf in (8, 16, 12)]
    xs = [vector(G, i) for i, G in enumerate(geos)]
    ref = lf.matvec_batch(geos, xs)
    assert len({int(lf.geometry_query(G, "wait_word", np.int64)[0]) for G in geos}) == 3
    for late in range(3):
        word(lf, geos[late]).value = 1
        for i in range(3):
            if i != late:
                assert torch.equal(lf.matvec(geos[i], xs[i]), ref[i])
        with pytest.raises(lf.LfmmError) as err:
            lf.matvec_batch(geos, xs)
        assert err.value.status == lf.LFMM_ERR_TIMEOUT
        for y, r in zip(lf.matvec_batch(geos, xs), ref):
            assert torch.equal(y, r)


def test_words_come_from_one_page(gpu_lib):
    """Builds and releases pin no memory of their own: live geometries have words of one page, and a
    released word comes back cleared."""
    lf = gpu_lib
    geos = [geometry(lf, layered_wide(), 16) for _ in range(4)]
    at = [int(lf.geometry_query(G, "wait_word", np.int64)[0]) for G in geos]
    assert len(set(at)) == 4 and max(at) - min(at) < 4096
    for _ in range(3):
        word(lf, geos[-1]).value = 1
        last = int(lf.geometry_query(geos[-1], "wait_word", np.int64)[0])
        geos.pop().destroy()
        geos.append(geometry(lf, layered_wide(), 16))
        assert int(lf.geometry_query(geos[-1], "wait_word", np.int64)[0]) == last
        assert word(lf, geos[-1]).value == 0
