"""Compositing of many and few bricks of a screen tile: entries are read 128 at a time and blended four
at a time, so one, a remainder, exactly 128, one more and many times 128 bricks of a tile."""
import numpy as np
import pytest

import synth
from gpu_helpers import compare_dvr, gpu_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,brick", [((4, 3, 5), (8, 8, 8)), ((5, 1, 1), (1, 1, 1)), ((8, 8, 8), (2, 2, 1)), ((3, 43, 1), (1, 1, 1)),
                                         ((12, 12, 12), (1, 1, 1))])
@pytest.mark.parametrize("W,H", [(16, 16), (21, 18)])
def test_tiles_of_few_and_many_bricks_match_the_oracle(orc, shape, brick, W, H):
    ctx = gpu_ctx()
    rng = np.random.default_rng(shape[1])
    cube = (2.0 * rng.standard_normal(shape[::-1])).astype(np.float32)
    lut = synth.random_lut(5, n=64)
    vr, step = (-7.0, 7.0), 0.3
    cid = ctx.load_cube(cube)
    ctx.set_bricking(cid, brick, 1, "f32")
    ctx.set_transfer_function(lut, *vr)
    m = np.array(shape, np.float64) / 2
    d = 1.2 * float(np.linalg.norm(shape))
    cam = dict(view=synth.look_at(m + d * np.array((0.6, 0.5, 0.62)), m), proj=1, param=0.9, W=W, H=H)
    ctx.set_camera_dict(cam)
    for _ in range(2):                 # back to back: the second frame's uploads follow the first one's compositing
        ctx.set_render_params("dvr", step, 2.0)
        img = ctx.render_frame(cid)
        ctx.set_render_params("mip", step, 2.0)
        mip = ctx.render_frame(cid)
    ref, flags, _ = orc.render(cube, lut, vr, cam, step=step, tau=2.0, brick=brick)
    compare_dvr(img.cpu().numpy().reshape(-1, 4), ref, flags, 2.0)
    m32, _, _ = orc.render(cube, lut, vr, cam, mode="mip32", step=step, brick=brick)
    assert np.array_equal(mip.cpu().numpy().reshape(-1), m32.astype(np.float32))
    ctx.close()
