"""Time-outs (LFMM_ERR_TIMEOUT).  No wait is made to run out on the device: the test sets the word
that a kernel would set, in host memory, and looks at what the calls do with it."""

import ctypes

import numpy as np
import pytest

from oracle import nystrom as onys
from workloads import layered_wide

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
