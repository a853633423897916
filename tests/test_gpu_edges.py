"""Calls at the ends of the accepted range:

* objective and adjoint at resolutions where the shared memory holds two
  8-lane stitching tiles per block, which are half a warp.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2405_15197_gb300 import lattices as L  # noqa: E402
from paper_2405_15197_gb300 import liblm  # noqa: E402
from tests import parity as P  # noqa: E402


@pytest.mark.parametrize("dtype,k,adjoint", [(np.float32, 1200, True), (np.float64, 650, True),
                                             (np.float32, 1700, False), (np.float64, 1000, False)])
def test_objective_at_fine_resolution(dtype, k, adjoint):
    """Area and volume against the FP64 oracle where a block has 16 threads
    (a tile of the adjoint takes 48 B per loop point in FP32 and 82 in FP64,
    of the objective 32 and 66; four tiles exceed 200 KB from about 1,060,
    620, 1,600 and 770 points on).  FP32: a triangle's width is 2 pi R / k,
    its relative error from rounded points up to 1e-4 and random over more
    than 10^4 triangles, so the sums are within 1e-5; FP64 1e-10."""
    lat = P.lattice_as(L.bcc(1, jitter=0.05, radius_range=(0.05, 0.09)), dtype)
    mm = liblm.MetaMesh(*P.to_device(lat, dtype))
    o = oracle.Oracle(lat)
    _, area, vol = o.triangulate(k, want_tris=False)
    tol = 1e-5 if dtype == np.float32 else 1e-10
    assert mm.tri_count(k) == int(o.tri_counts(k).sum())
    assert mm.objective(k) == pytest.approx((area, vol), rel=tol)
    if adjoint:
        _, _, a, v = mm.backward(k, 1.0, 0.5)
        assert (a, v) == pytest.approx((area, vol), rel=tol)
    assert liblm.lm_last_error(mm.h) == 0
    mm.close()
