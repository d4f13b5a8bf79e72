"""Serving admits by estimated device footprints: they are not below what the requests' geometries
hold, tables, digits and workspaces included, also where those are most of it."""

import math

import numpy as np
import pytest

from workloads import config_c2, config_c5_stream, layered_small

pytestmark = pytest.mark.gpu


def held(lf, wl, pts, w):
    """of a geometry that has preconditioned and multiplied once"""
    M = lf.medium_create(wl.medium.interfaces, wl.medium.k, wl.medium.eta)
    G = lf.geometry_build(M, pts, w, p=20, leaf_size=64)
    x = np.ones(G.n, dtype=np.complex128)
    lf.matvec(G, lf.precond_apply(G, x))
    total, digits, workspace = lf.geometry_query(G, "device_bytes", np.float64)
    assert 0 <= digits and digits + workspace < total
    G.destroy()
    return total


def submit(lf, srv, wl, pts, w, steps):
    return srv.submit(wl.medium.interfaces, wl.medium.k, wl.medium.eta, pts, w, math.radians(40.0), max_iter=steps)


# the serving workload's (2 to 4 layers, 2,720 to 59,787 points) and the benchmark's geometry
def test_estimates_cover_what_requests_hold(gpu_lib):
    lf = gpu_lib
    for wl in [*config_c5_stream(10, 12455, n_max=131072.0, max_bodies=128)[:9:2], config_c2(), layered_small()]:
        pts, w, _ = lf.polygon_elements(wl.bodies)
        need = held(lf, wl, pts, w) + 16 * w.size * 4   # and three Krylov vectors and the solution
        srv = lf.Server(slots=1, hbm_budget=64 << 30)
        _, _, times = srv.wait(submit(lf, srv, wl, pts, w, 3))
        peak = srv.stats()["peak_bytes"]
        srv.close()
        assert need <= times["footprint_bytes"] <= peak


def test_requests_are_counted_with_what_they_hold(gpu_lib):
    """A budget that the sizes alone would fill with three requests at once (four layers, 1.1 GB of
    tables, digits and workspace each, 300 MB by the sizes) runs them one at a time, and one whose
    estimate is above the budget by itself."""
    lf = gpu_lib
    wl = config_c5_stream(3, 12455, n_max=131072.0, max_bodies=128)[2]
    pts, w, _ = lf.polygon_elements(wl.bodies)
    need = held(lf, wl, pts, w)
    assert need > 900e6
    srv = lf.Server(slots=3, hbm_budget=1 << 30)
    got = [srv.wait(t) for t in [submit(lf, srv, wl, pts, w, 3) for _ in range(3)]]
    st = srv.stats()
    srv.close()
    assert st["peak_running"] == 1 and st["peak_bytes"] >= need
    assert all(g[1]["iterations"] == 3 for g in got)
