"""Calls at the ends of the accepted range:

* objective and adjoint at resolutions where the shared memory holds two
  8-lane stitching tiles per block, which are half a warp;
* lattices without struts whose node arrays span several scan tiles;
* struts whose length, radius or taper leaves the range of the lattice's type;
* an objective whose sums leave the range of FP32;
* a device with room for the build but not for the arena beside it;
* memory that the pool keeps, and gives back on request or when PyTorch's
  allocator has no other.
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


@pytest.mark.parametrize("dtype,k", [(np.float32, 1200), (np.float64, 650)])
def test_adjoint_at_fine_resolution(dtype, k):
    """Gradients where the adjoint takes 16-lane tiles, against central
    differences of the oracle's frozen structure (bounds of test_gpu_adjoint)."""
    lat = P.lattice_as(L.bcc(1, jitter=0.05, radius_range=(0.05, 0.09)), dtype)
    o = oracle.Oracle(lat)
    fz = oracle.Frozen(o, k)
    d1, d2 = (np.stack(fz.fd(h, np.arange(o.N))) for h in (1e-4, 5e-5))
    ref = (4.0 * d2 - d1) / 3.0
    ref = 1.0 * ref[0] + 0.5 * ref[1]
    mm = liblm.MetaMesh(*P.to_device(lat, dtype))
    gx, gr, _, _ = mm.backward(k, 1.0, 0.5)
    g = np.concatenate([gx.cpu().numpy(), gr.cpu().numpy()[:, None]], 1).astype(np.float64)
    err = np.abs(g - ref)
    if dtype == np.float32:
        assert err.max() < 1e-3 * np.abs(ref).max()
    else:
        assert (err / np.maximum(np.abs(ref), 1e-3 * np.abs(ref).max())).max() < 1e-6
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


def one_strut(length, ra, rb):
    return {"xyz": np.array([[0.0, 0.0, 0.0], [0.0, 0.0, length]]), "ends": np.array([[0, 1]], dtype=np.int32),
            "radii": np.array([[ra, rb]]), "name": "one"}


# Refused: squared length or radius below or above the type's normal numbers,
# taper within the rounding of 1 - s^2 of the limit.
@pytest.mark.parametrize("dtype,length,ra,rb", [
    (np.float32, 1e-20, 1e-21, 1e-21), (np.float32, 1e-19, 1e-20, 1e-20), (np.float32, 3e19, 1.0, 1.0),
    (np.float32, 1e10, 1e20, 1e20), (np.float32, 1.0, 1.5, 0.5 + 2.0 ** -24), (np.float32, 1.0, 0.5 + 2.0 ** -24, 1.5),
    (np.float64, 1e-155, 1e-156, 1e-156), (np.float64, 1e155, 1.0, 1.0), (np.float64, 1e10, 1e155, 1e155),
    (np.float64, 1.0, 1.5, 0.5 + 2.0 ** -53)])
def test_struts_outside_the_range_of_the_type(dtype, length, ra, rb):
    """Such a strut's direction or cone would be infinite or NaN in the
    kernels, and with it angles that loops are ordered by."""
    x, e, r = P.to_device(one_strut(length, ra, rb), dtype)
    assert float(r[0, 0]) > 0 and abs(float(r[0, 0]) - float(r[0, 1])) < float(x[1, 2])
    with pytest.raises(liblm.LmError) as ei:
        liblm.MetaMesh(x, e, r)
    assert ei.value.status == 3


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_struts_inside_the_range_of_the_type(dtype):
    """Scaled by a power of two, a lattice keeps its meta-mesh; a steep taper
    above the rounding is accepted."""
    lat = P.lattice_as(L.bcc(2, jitter=0.05, radius_range=(0.05, 0.09)), dtype)
    mm = liblm.MetaMesh(*P.to_device(lat, dtype))
    want = mm.counts()
    mm.close()
    for s in (2.0 ** -50, 2.0 ** 50):
        mm = liblm.MetaMesh(*P.to_device(dict(lat, xyz=lat["xyz"] * s, radii=lat["radii"] * s), dtype))
        assert mm.counts() == want
        mm.close()
    mm = liblm.MetaMesh(*P.to_device(one_strut(1.0, 1.5, 0.5 + 1e-5), dtype))
    assert mm.counts()[:4] == [2, 0, 2, 2]
    mm.close()


def test_objective_sums_beyond_fp32():
    """The sums are FP64: a lattice 1,024 cells from the origin, scaled by
    2^42, has terms of the volume above 10^39.  Scaling by a power of two
    changes no rounding, so the volume scales by 2^126; the order of the sums
    is free (terms 100 times the total, 10^-14 each)."""
    lat = P.lattice_as(L.bcc(2, radius=0.0625), np.float32)
    got = []
    for s in (1.0, 2.0 ** 42):
        mm = liblm.MetaMesh(*P.to_device(dict(lat, xyz=(lat["xyz"] + 1024.0) * s, radii=lat["radii"] * s), np.float32))
        mm.tri_count(8)
        v = mm.objective(8)[1] / s ** 3
        assert mm.backward(8, 0.0, 1.0)[3] / s ** 3 == pytest.approx(v, rel=1e-10)
        got.append(v)
        mm.close()
    assert got[1] == pytest.approx(got[0], rel=1e-10)


def test_build_where_the_arena_leaves_no_room():
    """What fits without the arena fits with it: on a device filled up to 64
    MB above the needs of a build without one, the default build (an arena of
    about 140 MB) gives way, also after its outputs are allocated (the FP64
    contexts come last, about 160 MB)."""
    x, e, r = P.to_device(P.lattice_as(L.bcc(40, radius=0.05), np.float32), np.float32)
    none = liblm.lm_options()
    none.arena_bytes = -1
    liblm.MetaMesh(x, e, r).close()  # every kernel is loaded
    liblm.lm_pool_retain(0)
    filler = None
    try:
        liblm.lm_pool_retain((1 << 64) - 1)
        torch.cuda.empty_cache()
        free0 = torch.cuda.mem_get_info()[0]
        mm = liblm.MetaMesh(x, e, r, options=none)
        need = free0 - torch.cuda.mem_get_info()[0]
        want = mm.counts()
        mm.close()
        liblm.lm_pool_retain(0)
        filler = torch.empty(torch.cuda.mem_get_info()[0] - need - (64 << 20), dtype=torch.uint8, device="cuda")
        for opt in (none, None):
            mm = liblm.MetaMesh(x, e, r, options=opt)
            assert mm.counts() == want
            assert mm.tri_count(8) > 0
            mm.close()
            liblm.lm_pool_retain(0)
    finally:
        del filler
        torch.cuda.empty_cache()


def test_pool_keeps_and_gives_back():
    """A build of about 440 MB (BCC 40^3 with its arena) stays mapped after it
    is freed, up to the limit; lm_pool_retain(0) returns it to the device."""
    x, e, r = P.to_device(P.lattice_as(L.bcc(40, radius=0.05), np.float32), np.float32)
    liblm.MetaMesh(x, e, r).close()  # every kernel is loaded
    liblm.lm_pool_retain(0)
    torch.cuda.synchronize()
    free0, total = torch.cuda.mem_get_info()
    liblm.lm_pool_retain(total // 16)
    liblm.MetaMesh(x, e, r).close()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] < free0 - (200 << 20)
    liblm.lm_pool_retain(0)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] > free0 - (64 << 20)


def test_records_where_the_pool_holds_the_room():
    """The records of a build fit on a device whose last room the library's
    pool keeps idle (the arena and the temporaries of BCC 64^3, about 670 MB):
    PyTorch's cudaMalloc gets it."""
    x, e, r = P.to_device(P.lattice_as(L.bcc(64, radius=0.05), np.float32), np.float32)
    mm = liblm.MetaMesh(x, e, r)
    size = 50 * mm.tri_count(8)
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - size + (300 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert mm.triangulate(8).shape[0] * 50 == size
        assert liblm.lm_last_error(mm.h) == 0
    finally:
        del filler
        mm.close()
        torch.cuda.empty_cache()
