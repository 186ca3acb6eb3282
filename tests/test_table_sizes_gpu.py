"""Tables on either side of the sizes at which a CTA takes a whole work item instead of half of one, and
table gradients whose partial rows are shared: against the FP64 oracle."""
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


def _table(n):
    """Smooth: its slope, and so what FP32 rounding of a value does to a colour, is that of a small table."""
    t = np.arange(n)[:, None] / max(1, n - 1) * np.array([2.0, 3.0, 5.0, 2.5]) + np.array([0.1, 0.3, 0.6, 0.2])
    return ((0.5 + 0.5 * np.sin(2 * np.pi * t)) * np.array([1.0, 1.0, 1.0, 0.3])).astype(np.float32)


@pytest.mark.parametrize("nlut", [2, 384, 385, 768, 769, 4096])
@pytest.mark.parametrize("storage,layouts", [("f32", 9), ("f16", 9), ("bf16", 41), ("f32", 7), ("f16", 7)])
@pytest.mark.parametrize("masked", [False, True])
def test_frames_of_any_table_match_the_oracle(ctx, orc, nlut, storage, layouts, masked):
    shape, brick, vr = (37, 29, 31), (16, 29, 9), (-7.0, 7.0)
    cube = (2.0 * np.random.default_rng(4).standard_normal(shape[::-1])).astype(np.float32)
    mask = (np.arange(31) % 3 > 0).astype(np.uint8) if masked else None
    cid = ctx.load_cube(cube)
    ctx.set_brick_layouts(cid, layouts)
    ctx.set_bricking(cid, brick, 1, storage)
    ctx.set_transfer_function(_table(nlut), *vr)
    ctx.set_channel_mask(mask)
    m = np.array(shape, np.float64) / 2
    for eye in ((0.0, 0.1, 1.0), (1.0, 0.1, 0.05)):        # aligned, so that linear copies are read in rows
        cam = dict(view=synth.look_at(m + 90.0 * np.array(eye), m), proj=1, param=0.6, W=61, H=47)
        ctx.set_camera_dict(cam)
        ctx.set_render_params("dvr", 0.7, 2.0)
        img = ctx.render_frame(cid).cpu().numpy().reshape(-1, 4)
        ref, flags, _ = orc.render(cube, _table(nlut), vr, cam, step=0.7, tau=2.0, brick=brick, quant=storage, channels=mask)
        compare_dvr(img, ref, flags, 2.0)
    ctx.set_channel_mask(None)
    ctx.free_cube(cid)


# A table of n entries that refines one of m, k intervals to each of its own (n = k (m - 1) + 1), is the same
# function; the gradients of its entries, weighted by the coarse entries' hats, are the coarse table's.  (Entry
# by entry a fine table's gradient moves with the rounding of a sample's fraction, n 2^-24.)
# 512^2 frames that eight bricks each fill half of: more than 2048 work items, whose partial rows of 4096
# entries would pass 256 MB
@pytest.mark.parametrize("m,k,W,H", [(72, 9, 61, 47), (65, 10, 61, 47), (94, 11, 61, 47), (65, 16, 61, 47), (64, 65, 61, 47), (64, 65, 512, 512)])
@pytest.mark.parametrize("layouts", [9, 1])
def test_gradients_of_any_table_match_the_oracle(ctx, orc, m, k, W, H, layouts):
    import torch
    shape, brick, vr = (24, 22, 20), (12, 11, 10), (-9.0, 13.0)
    rng = np.random.default_rng(W)
    cube = (2.0 + 2.0 * rng.standard_normal(shape[::-1])).astype(np.float32)
    coarse, n = _table(m), k * (m - 1) + 1
    hat = np.maximum(0.0, 1.0 - np.abs(np.arange(n) / k - np.arange(m)[:, None]))
    fine = (hat.T @ coarse).astype(np.float32)
    cid = ctx.load_cube(cube)
    ctx.set_brick_layouts(cid, layouts)
    ctx.set_bricking(cid, brick, 1, "f32")
    ctx.set_transfer_function(fine, *vr)
    ctx.set_render_params("dvr", 0.6, 2.0)
    c = np.array(shape, np.float64) / 2
    cam = dict(view=synth.look_at(c + np.array([30.0, 12.0, 40.0]), c), proj=0, param=26.0, W=W, H=H)
    ref, flags, _ = orc.render(cube, coarse, vr, cam, step=0.6, tau=2.0, brick=brick)
    gout = rng.standard_normal((H, W, 4)).astype(np.float32)
    gout[flags.reshape(H, W) != 0] = 0.0                 # samples within rounding of a table entry
    gl_ref, gv_ref = orc.render_grad(cube, coarse, vr, cam, gout.reshape(-1, 4), step=0.6, tau=2.0, brick=brick)
    ctx.set_camera_dict(cam)
    gl, gv = torch.empty((n, 4), device="cuda"), torch.zeros(cube.shape, device="cuda")
    ctx.render_backward(cid, torch.from_numpy(gout).cuda(), gl, gv)
    # FP32 sums of a few thousand terms: 2e-4 of the largest entry, as the repository's gradient tests
    assert np.abs(hat @ gl.cpu().numpy() - gl_ref).max() <= 2e-4 * np.abs(gl_ref).max()
    assert np.abs(gv.cpu().numpy() - gv_ref).max() <= 2e-4 * np.abs(gv_ref).max()
    ctx.free_cube(cid)
