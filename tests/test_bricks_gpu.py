"""Bricking kernels at their edges: sources off a 16-byte boundary and of sizes that are no multiple
of 4, rows shorter and longer than a warp, scale exponents beyond one multiplication, more bricks
than one shelf of an atlas array holds, and arrays written again by an update."""
import ctypes as C

import numpy as np
import pytest

import synth
from gpu_helpers import gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gpu_ctx()
    yield c
    c.close()


def _check_bricks(ctx, orc, cid, cube, brick, storage):
    exps = None if storage == "f32" else orc.brick_exponents(cube, brick, 1, storage)
    nb, _ = ctx.brick_grid(cid)
    pad = np.pad(cube, 1, mode="edge")
    for b in range(int(np.prod(nb))):
        dims, org, e, data = ctx.get_brick(cid, b)
        want = pad[org[2] + 1:org[2] + 1 + dims[2], org[1] + 1:org[1] + 1 + dims[1], org[0] + 1:org[0] + 1 + dims[0]]
        if storage == "f32":
            assert np.array_equal(data, want)
            continue
        c = (b % nb[0], b // nb[0] % nb[1], b // (nb[0] * nb[1]))
        assert e == exps[c[2], c[1], c[0]]
        scaled = np.ldexp(want.astype(np.float64), -e)
        codes = (orc.round_fp16 if storage == "f16" else orc.round_bf16)(scaled.ravel()).reshape(want.shape)
        got = data.view(np.float16).astype(np.float64) if storage == "f16" else \
            (data.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
        assert np.array_equal(got, codes)


@pytest.mark.parametrize("shape,brick", [((13, 7, 5), (64, 64, 64)), ((131, 9, 33), (64, 8, 16)), ((301, 6, 4), (300, 3, 3))])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("scale", [1.0, 1e-38, 1e37])
def test_bricks_hold_the_voxels(ctx, orc, shape, brick, storage, scale):
    import torch
    rng = np.random.default_rng(shape[0])
    n = int(np.prod(shape))
    buf = torch.from_numpy((scale * rng.standard_normal(2 * n + 9)).astype(np.float32)).cuda()
    for off in (0, 1):                     # a source on a 16-byte boundary and one off it
        a = buf[off:off + n].view(shape[::-1])
        b = buf[n + 3 + off:2 * n + 3 + off].view(shape[::-1])
        cid = ctx.load_cube(a)
        ctx.set_brick_layouts(cid, 9)
        ctx.set_bricking(cid, brick, 1, storage)
        _check_bricks(ctx, orc, cid, a.cpu().numpy(), brick, storage)
        assert ctx.compute_minmax(cid) == (float(a.min()), float(a.max()))
        ctx.update_cube(cid, b)
        _check_bricks(ctx, orc, cid, b.cpu().numpy(), brick, storage)
        ctx.free_cube(cid)


@pytest.mark.parametrize("storage,mask", [("f32", 9), ("f16", 9), ("bf16", 41)])
def test_shelves_of_small_bricks_and_updates(ctx, storage, mask):
    import torch
    rng = np.random.default_rng(8)
    shape = (171, 60, 63)                  # 20 x 7 x 7 bricks: several shelves of one array
    first, second = (torch.from_numpy((2.0 * rng.standard_normal(shape[::-1])).astype(np.float32)).cuda() for _ in range(2))
    ctx.set_transfer_function(synth.random_lut(4, n=33), -6.0, 6.0)
    ctx.set_render_params("dvr", 0.7, 0.98)
    ctx.set_camera_dict(synth.random_camera(rng, shape, 90, 70, proj=1))
    frames = []
    for m in (1, mask):
        cid = ctx.load_cube(first)
        ctx.set_brick_layouts(cid, m)
        ctx.set_bricking(cid, (9, 9, 9), 1, storage)
        frames.append(ctx.render_frame(cid).cpu().numpy())
        ctx.update_cube(cid, second)       # the arrays are written again
        frames.append(ctx.render_frame(cid).cpu().numpy())
        ctx.free_cube(cid)
    assert np.array_equal(frames[0], frames[2]) and np.array_equal(frames[1], frames[3])
    assert not np.array_equal(frames[0], frames[1])


@pytest.mark.parametrize("offset", [1, 2, 4, 12])
def test_device_voxels_at_any_address(offset):
    """Sources that start between floats (copied by the copy engine) and between 16-byte pieces."""
    import torch
    ctx = gpu_ctx()
    cube = np.random.default_rng(4).standard_normal((11, 13, 21)).astype(np.float32)
    buf = torch.zeros(cube.nbytes + 16, dtype=torch.uint8, device="cuda")
    buf[offset:offset + cube.nbytes] = torch.from_numpy(cube.view(np.uint8).ravel()).cuda()
    torch.cuda.synchronize()
    cid = C.c_int()
    assert ctx._L.vr_load_cube(ctx._h, buf.data_ptr() + offset, 0, 21, 13, 11, 1, None, None, C.byref(cid)) == 0
    ctx.set_bricking(cid.value, (32, 32, 32), 1, "f32")
    assert np.array_equal(ctx.get_brick(cid.value, 0)[3][1:-1, 1:-1, 1:-1], cube)
    buf[offset:offset + cube.nbytes] = torch.from_numpy((2 * cube).view(np.uint8).ravel()).cuda()
    torch.cuda.synchronize()
    assert ctx._L.vr_update_cube(ctx._h, cid.value, buf.data_ptr() + offset, 1, None) == 0
    assert np.array_equal(ctx.get_brick(cid.value, 0)[3][1:-1, 1:-1, 1:-1], 2 * cube)
    ctx.close()
