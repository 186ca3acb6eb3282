"""Frames read from linear copies row by row, and channel masks as plane bits in shared memory: against
the FP64 oracle, and masked frames against frames of a cube edited to the same values."""
import numpy as np
import pytest

import synth
from gpu_helpers import compare_dvr, gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gpu_ctx()
    yield c
    c.close()


# every contiguous axis, aligned and oblique views, bricks of one voxel and of the whole cube
@pytest.mark.parametrize("shape,brick", [((37, 29, 31), (16, 29, 9)), ((5, 4, 3), (1, 1, 1))])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("masked", [False, True])
def test_linear_frames_match_the_oracle(ctx, orc, shape, brick, storage, masked):
    rng = np.random.default_rng(shape[2])
    cube = (2.0 * rng.standard_normal(shape[::-1])).astype(np.float32)
    lut = synth.random_lut(5, n=64)
    vr, step = (-7.0, 7.0), 0.7
    mask = (rng.uniform(size=shape[2]) < 0.6).astype(np.uint8) if masked else None
    cid = ctx.load_cube(cube)
    ctx.set_transfer_function(lut, *vr)
    ctx.set_channel_mask(mask)
    mips = []
    for layouts in (1, 7):
        ctx.set_brick_layouts(cid, layouts)
        ctx.set_bricking(cid, brick, 1, storage)
        for k, eye in enumerate(((0.0, 0.1, 1.0), (1.0, 0.05, 0.1), (0.6, 0.5, 0.6))):
            m = np.array(shape, np.float64) / 2
            d = 1.2 * float(np.linalg.norm(shape))
            cam = dict(view=synth.look_at(m + d * np.array(eye) / np.linalg.norm(eye), m), proj=k % 2,
                       param=float(np.linalg.norm(shape)) if k % 2 == 0 else 0.9, W=53, H=41)
            ctx.set_camera_dict(cam)
            ctx.set_render_params("dvr", step, 2.0)
            img = ctx.render_frame(cid).cpu().numpy().reshape(-1, 4)
            # (the oracle samples the same 16-bit codes: FP32 arithmetic alone separates the two)
            ref, flags, _ = orc.render(cube, lut, vr, cam, step=step, tau=2.0, brick=brick, quant=storage, channels=mask)
            compare_dvr(img, ref, flags, 2.0)
            ctx.set_render_params("mip", step, 2.0)
            mip = ctx.render_frame(cid).cpu().numpy().reshape(-1)
            m32, _, _ = orc.render(cube, lut, vr, cam, mode="mip32", step=step, brick=brick, quant=storage, channels=mask)
            assert np.array_equal(mip, m32.astype(np.float32))
    ctx.set_channel_mask(None)
    ctx.free_cube(cid)


# a disabled channel's voxels hold the bottom of the table range: FP32 frames equal, bit for bit, those of a
# cube edited so.  4097 stencil planes do not fit shared memory (the mask is read from global
# memory), 4096 just do; rows of layouts 1 and 7, gathers
@pytest.mark.parametrize("nz", [40, 4095, 4096])
@pytest.mark.parametrize("layouts", [1, 7, 9])
def test_masked_frames_equal_frames_of_the_edited_cube(ctx, nz, layouts):
    rng = np.random.default_rng(nz)
    cube = (2.0 * rng.standard_normal((nz, 9, 11))).astype(np.float32)
    mask = (rng.uniform(size=nz) < 0.6).astype(np.uint8)
    edited = np.where(mask[:, None, None] != 0, cube, np.float32(-7.0)).astype(np.float32)
    shape = (11, 9, nz)
    ctx.set_transfer_function(synth.random_lut(7, n=64), -7.0, 7.0)
    got = []
    for data, ch in ((cube, mask), (edited, None)):
        cid = ctx.load_cube(data)
        ctx.set_brick_layouts(cid, layouts)
        ctx.set_bricking(cid, (6, 9, 5000), 1, "f32")
        ctx.set_channel_mask(ch)
        frames = []
        for eye in ((0.0, 0.1, 1.0), (1.0, 0.05, 0.1), (0.7, 0.5, 0.1)):
            m = np.array(shape, np.float64) / 2
            d = 1.2 * float(np.linalg.norm(shape))
            ctx.set_camera_dict(dict(view=synth.look_at(m + d * np.array(eye) / np.linalg.norm(eye), m), proj=1, param=0.9, W=53, H=41))
            for mode, term in (("dvr", "segment"), ("dvr", "global"), ("mip", "segment")):
                ctx.set_render_params(mode, 0.7, 0.98)
                ctx.set_termination(term)
                frames.append(ctx.render_frame(cid).cpu().numpy())
        got.append(frames)
        ctx.set_channel_mask(None)
        ctx.set_termination("segment")
        ctx.free_cube(cid)
    assert all(np.array_equal(a, b) for a, b in zip(*got))
