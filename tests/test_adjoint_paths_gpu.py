"""The adjoint's two ways of adding voxel gradients (corner sums, one atomic per corner) and its table
partials at their edges: cubes of one voxel's width, borders and ghost copies, tables of two entries,
odd frames, batches on either side of the rule; against the FP64 oracle."""
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


# frames of 61x47 take the corner sums on these cubes, the 3x2 frame of the larger one does not
@pytest.mark.parametrize("shape,brick,W,H", [((9, 7, 5), (4, 4, 4), 61, 47), ((1, 12, 9), (8, 8, 8), 61, 47),
                                             ((13, 1, 1), (5, 5, 5), 61, 47), ((33, 34, 31), (16, 32, 11), 61, 47),
                                             ((64, 60, 62), (32, 32, 32), 3, 2)])
@pytest.mark.parametrize("layouts,nlut", [(9, 256), (1, 2)])
def test_gradients_of_both_paths_match_the_oracle(ctx, orc, shape, brick, W, H, layouts, nlut):
    import torch
    rng = np.random.default_rng(shape[0] + W)
    cube = (2.0 + 2.0 * rng.standard_normal(shape[::-1])).astype(np.float32)
    lut = synth.random_lut(11, n=nlut)
    vr = (-9.0, 13.0)
    cid = ctx.load_cube(cube)
    ctx.set_brick_layouts(cid, layouts)
    ctx.set_bricking(cid, brick, 1, "f32")
    ctx.set_transfer_function(lut, *vr)
    ctx.set_render_params("dvr", 0.6, 2.0)              # no termination: nothing is decided by rounding
    cams = [synth.random_camera(rng, shape, W, H, proj=k) for k in range(2)]
    gout = rng.standard_normal((2, H, W, 4)).astype(np.float32)
    gl_ref, gv_ref = np.zeros((nlut, 4)), np.zeros(cube.shape)
    for k, cam in enumerate(cams):
        ref, flags, _ = orc.render(cube, lut, vr, cam, step=0.6, tau=2.0, brick=brick)
        gout[k][flags.reshape(H, W) != 0] = 0.0          # samples within rounding of a table entry
        gl, gv = orc.render_grad(cube, lut, vr, cam, gout[k].reshape(-1, 4), step=0.6, tau=2.0, brick=brick)
        gl_ref += gl
        gv_ref += gv
    gl = torch.empty((nlut, 4), device="cuda")
    gv = torch.full(cube.shape, 0.5, device="cuda")     # added to what is there
    ctx.set_camera_dict(cams[0])
    ctx.render_backward_views(cid, cams, torch.from_numpy(gout).cuda(), gl, gv)
    # FP32 sums of a few thousand terms: 2e-4 of the largest entry, as the repository's gradient tests
    assert np.abs(gl.cpu().numpy() - gl_ref).max() <= 2e-4 * max(1e-3, np.abs(gl_ref).max())
    assert np.abs(gv.cpu().numpy() - 0.5 - gv_ref).max() <= 2e-4 * max(1e-3, np.abs(gv_ref).max())
    one = torch.empty((nlut, 4), device="cuda")
    both = torch.zeros_like(one)
    for k, cam in enumerate(cams):                       # the single-view call: the same sums
        ctx.set_camera_dict(cam)
        ctx.render_backward(cid, torch.from_numpy(gout[k]).cuda().contiguous(), one)
        both += one
    assert np.abs(both.cpu().numpy() - gl_ref).max() <= 2e-4 * max(1e-3, np.abs(gl_ref).max())
    ctx.free_cube(cid)
