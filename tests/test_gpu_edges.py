"""Calls at the ends of the accepted range:

* objective and adjoint at resolutions where the shared memory holds two
  8-lane stitching tiles per block, which are half a warp;
* lattices without struts whose node arrays span several scan tiles.
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


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("nodes", [4096, 4097, 5000, 10000])
def test_nodes_without_struts(nodes, dtype):
    """An empty meta-mesh: the scan over the strut ends is of an empty array
    beside arrays of several tiles (4,096 elements).  The memory is that of a
    larger build freed before, so what is not written shows."""
    dirty = liblm.MetaMesh(*P.to_device(P.lattice_as(L.octet(8), dtype), dtype))
    dirty.tri_count(8)
    dirty.close()
    t = torch.float32 if dtype == np.float32 else torch.float64
    mm = liblm.MetaMesh(torch.rand((nodes, 3), dtype=t, device="cuda"),
                        torch.zeros((0, 2), dtype=torch.int32, device="cuda"),
                        torch.zeros((0, 2), dtype=t, device="cuda"))
    assert mm.counts()[:5] == [0, 0, 0, 0, 0]
    g = mm.download()
    assert len(g["loop_ent"]) == 0 and np.array_equal(g["end_off"], [0])
    for key in ("row_ptr", "vtx_off", "arc_off", "hole_off_n"):
        assert np.array_equal(g[key], np.zeros(nodes + 1)), key
    assert mm.tri_count(8) == 0 and mm.objective(8) == (0.0, 0.0)
    assert liblm.lm_last_error(mm.h) == 0
    mm.close()
