"""What the library's host code decides, on a stand-in runtime: no device."""
import ctypes as C

import numpy as np
import pytest

from paper_1008_0135_gb300 import _abi
from host_helpers import Host, fake_lib, launches


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_lib(tmp_path_factory.mktemp("fake"))


def _view(R, t):
    v = np.eye(4)
    v[:3, :3], v[:3, 3] = R, t
    return v


SHEAR = np.eye(3)
SHEAR[0, 2] = 1e6
STEEP = np.eye(3)
STEEP[0, 2] = 2.0 ** 40
# view, projection, whether unclamped reads are safe: rays of the sheared view start up to 6 10^7 voxels away
# although R^T t is beside the cube; the steep one's eye is a sum of terms of 3 10^13, whose FP32 rounding is 10^6
VIEWS = [(_view(np.eye(3), (-32, -32, -100)), 0, True), (_view(1.1 * np.eye(3), (-32, -32, -100)), 0, True),
         (_view(np.eye(3), (-32, -32, -100)), 1, True), (_view(np.eye(3), (-32, -32, -3e5)), 1, False),
         (_view(SHEAR, (0, -32, -80)), 0, False), (_view(STEEP, (-32, -32, 2.0 ** 45)), 1, False)]


@pytest.mark.parametrize("view,proj,near", VIEWS)
def test_cameras_whose_rays_start_far_away_read_clamped_stencils(lib, view, proj, near):
    with Host(lib) as h:
        for layouts in (1, 7, 9):
            cid = h.load((64, 60, 62))
            h.ok(h.brick(cid, (32, 32, 32), layouts))
            for mode in (0, 1):
                for mask in (None, bytes([1, 0] * 31)):
                    h.ok(lib.vr_set_channel_mask(h.h, mask, 62 if mask else 0))
                    h.camera(view, proj, 64.0 if proj == 0 else 1.0, mode=mode)
                    launches(lib)
                    h.ok(h.frame(cid))
                    fetch = [a[2] for k, a in launches(lib) if k == "k_raycast"]
                    assert len(fetch) == 1 and (fetch[0] == 0) == (not near), (layouts, mode, fetch)
            h.ok(lib.vr_set_channel_mask(h.h, None, 0))
            h.camera(view, proj, 64.0 if proj == 0 else 1.0)
            launches(lib)
            g, gl, gv = np.zeros((24, 32, 4), np.float32), np.zeros((2, 4), np.float32), np.zeros((62, 60, 64), np.float32)
            h.ok(lib.vr_render_backward(h.h, cid, g.ctypes.data, gl.ctypes.data, gv.ctypes.data, None))
            atlas = [a[0] for k, a in launches(lib) if k == "k_adjoint"]
            assert atlas == [int(near and layouts == 9)]


@pytest.mark.parametrize("offset,short,kernel", [(0, 0, True), (4, 0, True), (12, 0, True), (1, 0, False), (2, 0, False),
                                                 (0, 4, False), (4, 4, False)])
def test_device_sources_that_a_kernel_cannot_read_go_to_the_copy_engine(lib, offset, short, kernel):
    """Voxels at an address that is no multiple of 4, or (from the copy engine: an error) beyond their allocation."""
    n, cid = 4 * 9 * 7 * 5, C.c_int()
    with Host(lib) as h:
        src = lib.fake_device_alloc(n + offset - short) + offset
        launches(lib)
        h.ok(lib.vr_load_cube(h.h, src, 0, 9, 7, 5, 1, None, None, C.byref(cid)))
        assert launches(lib) == [("k_copy" if kernel else "cudaMemcpy3DAsync", ())]
        rc = lib.vr_update_cube(h.h, cid.value, src, 1, None)
        assert launches(lib) == [("k_copy" if kernel else "cudaMemcpyAsync", ())]
        assert rc == (-3 if short else 0)


@pytest.mark.parametrize("without", [(), (0,), (1,)])
def test_atlas_arrays_with_and_without_surfaces(lib, without):
    """Two arrays, one of which the device gives no surface: both bricks' atlases are packed through staging."""
    with Host(lib) as h:
        cid = h.load((2048, 64, 248))                  # a shelf each: 1026 texels wide, 16500 high
        launches(lib)
        for nth in without:
            lib.fake_fail_surface_array(nth, 801)
        h.ok(h.brick(cid, (1024, 64, 248)))
        assert lib.fake_arrays() == 2
        ran = launches(lib)
        assert [a for k, a in ran if k == "k_brick_build"] == [(0, 0 if without else 1)]
        assert [k for k, _ in ran].count("k_atlas_pack") == [k for k, _ in ran].count("cudaMemcpy2DToArrayAsync")
        assert [k for k, _ in ran].count("k_atlas_pack") == (2 if without else 0)


@pytest.mark.parametrize("what", ["load", "short source", "bricking", "cache"])
def test_the_call_after_a_failed_one_does_not_fail_with_its_error(lib, what):
    with Host(lib, cache=1 << 20) as h:
        cid, other = h.load((64, 60, 62)), C.c_int()
        h.ok(h.brick(cid, (32, 32, 32)))
        h.camera(_view(np.eye(3), (-32, -32, -100)))
        h.ok(h.frame(cid))
        src = lib.fake_device_alloc(64)
        lib.fake_limit(lib.fake_reserved() + (1 << 16))
        if what == "load":
            cube = np.zeros((64, 64, 64), np.float32)
            rc = lib.vr_load_cube(h.h, cube.ctypes.data, 0, 64, 64, 64, 0, None, None, C.byref(other))
        elif what == "short source":
            rc = lib.vr_update_cube(h.h, cid, src, 1, None)
        elif what == "bricking":
            rc = lib.vr_set_brick_layouts(h.h, cid, 31)
        else:
            h.ok(lib.vr_load_cube_procedural(h.h, 1, 20, 20, 20, C.byref(other)))
            h.ok(h.brick(other.value, (16, 16, 16), 1))
            rc = h.frame(other.value)
        assert rc == (-3 if what == "short source" else -2)
        h.ok(lib.vr_compute_minmax(h.h, cid, C.byref(C.c_float()), C.byref(C.c_float())))
        if what != "bricking":
            h.ok(h.frame(cid))


FLAT = np.diag([1e3, 1e3, 1e-6])


@pytest.mark.parametrize("R,proj,counts", [(np.eye(3), 0, True), (np.eye(3), 1, True), (0.9 * np.eye(3), 1, True), (SHEAR, 0, True),
                                           (FLAT, 0, False), (FLAT, 1, True)])
def test_directions_too_short_to_count_samples_along_are_refused(lib, R, proj, counts):
    """A direction of length 1e-6 puts 2 10^8 samples of step 0.5 into 110 voxels: a float does not count them.
    (A perspective view's directions are only as short in single pixels.)"""
    view, err = _view(R, (-32, -32, -100)), -1
    with Host(lib) as h:
        cid = h.load((64, 60, 62))
        h.ok(h.brick(cid, (32, 32, 32)))
        g, gl = np.zeros((24, 32, 4), np.float32), np.zeros((2, 4), np.float32)
        arr = (_abi.VrView * 1)()
        arr[0].view[:], arr[0].proj, arr[0].param = [float(x) for x in view.ravel()], proj, 1.0
        h.camera(np.eye(4), step=0.5)
        assert lib.vr_render_backward_views(h.h, cid, 1, arr, g.ctypes.data, gl.ctypes.data, None, None) == (0 if counts else err)
        for mode in (0, 1):
            h.camera(view, proj, 1.0, mode=mode, step=0.5)
            launches(lib)
            assert h.frame(cid) == (0 if counts else err)
            assert any(k == "k_raycast" for k, _ in launches(lib)) == counts


@pytest.mark.parametrize("how", ["free", "compress", "rebrick"])
def test_memory_that_a_cube_leaves_is_bounded_when_the_call_returns(lib, how):
    """At most 2 GiB of it stays with the context (vr_create), not what the next wait would give back."""
    n, kept = (1000, 1000, 700), 2 << 30                       # 2.6 GiB of voxels, 2.7 of bricks
    with Host(lib) as h:
        base = lib.fake_reserved()
        cid = h.load(n)
        if how != "compress":
            h.ok(h.brick(cid, (128, 128, 128), 7))
        if how == "free":
            h.ok(lib.vr_free_cube(h.h, cid))
            assert lib.fake_reserved() - base <= kept
        elif how == "compress":
            h.ok(lib.vr_compress_cube(h.h, cid))
            assert lib.fake_reserved() - base <= kept + 544 * 125 * 125 * 88
        else:
            h.ok(lib.vr_set_brick_layouts(h.h, cid, 1))
            assert lib.fake_reserved() - base <= kept + int(2.2 * 4 * n[0] * n[1] * n[2])


def test_the_scratch_of_a_voxel_gradient_is_exact_and_given_back(lib):
    def backward(h, cid, n, nlut=2):
        lut = np.zeros((nlut, 4), np.float32)
        h.ok(lib.vr_set_transfer_function(h.h, lut.ctypes.data, nlut, 0.0, 1.0))
        h.camera(_view(np.eye(3), (-n / 2, -n / 2, -2 * n)), param=1.5 * n, W=512, H=512, step=0.5)
        return lib.vr_render_backward(h.h, cid, h.out.ctypes.data, h.out.ctypes.data, h.out.ctypes.data, None)

    size = lambda n: 16 * (n + 1) ** 2 * (n + 2)
    with Host(lib) as h:
        small, large = h.load((200, 200, 200)), h.load((204, 204, 204))
        h.ok(h.brick(small, (256, 256, 256)))
        h.ok(h.brick(large, (256, 256, 256)))
        h.ok(backward(h, small, 200))
        before = lib.fake_reserved()
        h.ok(backward(h, large, 204))                     # not 1.5 times the last one's
        assert lib.fake_reserved() - before < size(204) - size(200) + (16 << 20)
        # an allocation of the call itself that finds no memory leaves the sums it is using
        lib.fake_limit(lib.fake_reserved() + (1 << 20))
        before = lib.fake_reserved()
        assert backward(h, large, 204, nlut=4096) == -2
        assert before - lib.fake_reserved() < size(204) // 2
        # another call's takes them back
        cube, cid = np.zeros((150, 200, 200), np.float32), C.c_int()
        h.ok(lib.vr_load_cube(h.h, cube.ctypes.data, 0, 200, 200, 150, 0, None, None, C.byref(cid)))
        lib.fake_limit((1 << 64) - 1)
        h.ok(backward(h, small, 200))


@pytest.mark.parametrize("others,again", [([(3 + k, 4, 5) for k in range(260)], (90, 80, 70)),       # more arrays than are kept
                                          ([(500, 500 - 9 * k, 330) for k in range(5)], (400, 300, 200))])  # more bytes: 340 MB each
def test_the_arrays_of_the_last_cubes_are_the_ones_kept(lib, others, again):
    """A viewer that has opened cubes of many sizes and now opens one size again and again."""
    with Host(lib) as h:
        made = []
        for n in others + 3 * [again]:
            cid, before = h.load(n), lib.fake_surface_arrays_made()
            h.ok(h.brick(cid, (512, 512, 512)))
            made.append(lib.fake_surface_arrays_made() - before)
            h.ok(lib.vr_free_cube(h.h, cid))
        assert made[-3:] == [1, 0, 0]
        assert lib.fake_arrays() <= 256 and lib.fake_reserved() <= (3 << 30) + (1 << 20)


def test_idle_memory_can_be_released(lib):
    with Host(lib) as h:
        for _ in range(2):
            cid = h.load((100, 100, 100))
            h.ok(h.brick(cid, (64, 64, 64)))
            h.camera(_view(np.eye(3), (-50, -50, -200)), param=150.0, W=512, H=512)
            h.ok(lib.vr_render_backward(h.h, cid, h.out.ctypes.data, h.out.ctypes.data, h.out.ctypes.data, None))
            h.ok(lib.vr_free_cube(h.h, cid))
        kept = lib.fake_reserved()
        h.ok(lib.vr_release_idle(h.h))
        # voxels, bricks and atlases, and the sums
        assert kept - lib.fake_reserved() > 4 * 3 * 100 ** 3 + 16 * 101 * 101 * 102
        assert lib.fake_arrays() == 0
        cid = h.load((100, 100, 100))
        h.ok(h.brick(cid, (64, 64, 64)))
        h.ok(h.frame(cid))
    assert lib.vr_release_idle(None) == -1


@pytest.mark.parametrize("n", [(11000, 11000, 2), (7000, 11000, 4), (1000, 1000, 1000)])
@pytest.mark.parametrize("storage", [0, 1])
def test_bricks_near_the_gather_size_are_read_from_atlases(lib, n, storage):
    """Admitted bricks all get an atlas, without copies of slices where those do not fit (fetch mode 3)."""
    with Host(lib) as h:
        cid = h.load(n)
        h.ok(h.brick(cid, n, 9, storage))
        assert lib.fake_arrays() == 1
        h.camera(_view(np.eye(3), (-n[0] / 2, -n[1] / 2, -2 * n[0])), param=1.5 * n[0], step=1.0)
        launches(lib)
        h.ok(h.frame(cid))
        assert [a[2] for k, a in launches(lib) if k == "k_raycast"] == [3]
        h.ok(lib.vr_set_termination(h.h, 1))
        h.ok(h.frame(cid))
        assert [a[1] for k, a in launches(lib) if k == "k_raymarch"] == [3]


@pytest.mark.parametrize("layouts,storage,last", [(9, 0, 768), (41, 1, 768), (7, 0, 384)])
def test_large_tables_are_shared_by_whole_work_items(lib, layouts, storage, last):
    with Host(lib) as h:
        cid = h.load((64, 60, 62))
        h.ok(h.brick(cid, (32, 32, 32), layouts, storage))
        h.camera(_view(np.eye(3), (-32, -32, -100)))
        for n in (2, last, last + 1, 4096):
            lut = np.zeros((n, 4), np.float32)
            h.ok(lib.vr_set_transfer_function(h.h, lut.ctypes.data, n, 0.0, 1.0))
            launches(lib)
            h.ok(h.frame(cid))
            assert [a[4] for k, a in launches(lib) if k == "k_raycast"] == [int(n <= last)]


def test_a_cache_that_could_not_be_sized_at_first_serves_large_bricks_right(lib):
    """The layout call finds no memory, the frame later does: slots without copies, read without them."""
    n = (11000, 11000, 2)
    with Host(lib, cache=4 << 30) as h:
        cid = h.load(n)
        h.ok(lib.vr_compress_cube(h.h, cid))
        h.ok(lib.vr_set_bricking(h.h, cid, *n, 1, 0))
        lib.fake_limit(lib.fake_reserved())
        assert lib.vr_set_brick_layouts(h.h, cid, 9) == -2
        lib.fake_limit((1 << 64) - 1)
        h.camera(_view(np.eye(3), (-5500, -5500, -22000)), param=16500.0, step=1.0)
        launches(lib)
        h.ok(h.frame(cid))
        assert [a[2] for k, a in launches(lib) if k == "k_raycast"] == [3]


def test_the_binding_refuses_an_update_shorter_than_the_cube(lib, monkeypatch):
    import paper_1008_0135_gb300 as P
    monkeypatch.setattr(_abi, "_lib", lib)
    lib.fake_reset()
    ctx = P.Context(0)
    cid = ctx.load_cube(np.zeros((5, 7, 9), np.float32))
    sub = ctx.load_cube(np.zeros((5, 7, 9), np.float32), sub_origin=(1, 1, 1), sub_extent=(4, 3, 2))
    for good in (np.zeros((5, 7, 9), np.float32), np.zeros(400, np.float32)):
        ctx.update_cube(cid, good)
    ctx.update_cube(sub, np.zeros((2, 3, 4), np.float32))
    for c, n in ((cid, 314), (sub, 23)):
        with pytest.raises(ValueError):
            ctx.update_cube(c, np.zeros(n, np.float32))
    ctx.close()
