"""Slice and pair atlases against the linear copy, bit for bit, where their columns can go wrong:
one column, a last column of one slice, several columns with copies, and cameras so far away that
atlas frames fall back to the clamped linear copy."""
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


def _frames(ctx, cid, shape, far):
    nx, ny, nz = shape
    out = []
    rng = np.random.default_rng(5)
    for k in range(2):
        if far:
            c = np.array(shape, np.float64) / 2
            d = 3e5 if k else 2.7e5
            cam = dict(view=synth.look_at(c + d * np.array([0.6, 0.0, 0.8]), c), proj=1, param=float(1.2 * max(shape) / d), W=60, H=50)
        else:
            cam = synth.random_camera(rng, shape, 70, 52, proj=k)
        ctx.set_camera_dict(cam)
        for mask in (None, (np.arange(nz) % 3 > 0).astype(np.uint8)):
            ctx.set_channel_mask(mask)
            for mode, term in (("dvr", "segment"), ("dvr", "global"), ("mip", "segment")):
                ctx.set_render_params(mode, 1.0, 0.97)
                ctx.set_termination(term)
                out.append(ctx.render_frame(cid).cpu().numpy())
    ctx.set_channel_mask(None)
    ctx.set_termination("segment")
    return out


# stored slices (dz) x stored rows (dy) against the 32768 texels of a column: the whole brick in one
# column (40 * 52), two columns (the second of few slices), three columns, and bricks of several sizes
@pytest.mark.parametrize("shape,brick", [((21, 50, 38), (64, 64, 64)), ((5, 250, 131), (64, 256, 256)),
                                         ((7, 300, 230), (8, 512, 512)), ((33, 190, 191), (20, 190, 100))])
@pytest.mark.parametrize("storage,mask", [("f32", 9), ("f16", 9), ("bf16", 9), ("f16", 41), ("bf16", 41)])
def test_atlas_frames_equal_linear_frames(ctx, shape, brick, storage, mask):
    rng = np.random.default_rng(shape[2])
    cube = (3.0 * rng.standard_normal(shape[::-1])).astype(np.float32)
    cid = ctx.load_cube(cube)
    ctx.set_transfer_function(synth.random_lut(3, n=37), -8.0, 9.0)
    for far in (False, True):
        ctx.set_brick_layouts(cid, 1)
        ctx.set_bricking(cid, brick, 1, storage)
        want = _frames(ctx, cid, shape, far)
        ctx.set_brick_layouts(cid, mask)
        got = _frames(ctx, cid, shape, far)
        assert all(np.array_equal(a, b) for a, b in zip(want, got))
        assert max(float(np.abs(a).max()) for a in want) > 0.05
    ctx.free_cube(cid)


# stored bricks of 4 and 6 slices that a gather array only takes without the columns' copies (11002^2 x 4: two
# columns of two slices; 7002 x 11002 x 6: three; the second with a small brick beside it)
@pytest.mark.parametrize("shape,brick", [((11000, 11000, 2), (11000, 11000, 2)), ((7040, 11000, 4), (7000, 11000, 4))])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "compressed"])
def test_bricks_near_the_gather_size_keep_their_atlases(shape, brick, storage):
    import torch
    gpu_ctx().close()
    import paper_1008_0135_gb300 as P
    sto = "f32" if storage == "compressed" else storage
    ctx = P.Context(0, cache_bytes=6 << 30 if storage == "compressed" else 0)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    cid = ctx.load_cube(3.0 * torch.randn(shape[::-1], device="cuda", generator=g))
    ctx.set_transfer_function(synth.random_lut(3, n=37), -8.0, 9.0)
    if storage == "compressed":
        ctx.compress_cube(cid)
    got = []
    for mask in (1, 9):
        ctx.set_brick_layouts(cid, mask)
        ctx.set_bricking(cid, brick, 1, sto)
        got.append(_frames(ctx, cid, shape, False))
        if storage == "f32":                             # the adjoint: corner sums and single atomics
            for W, H in ((70, 52), (40, 30)):
                cam = synth.random_camera(np.random.default_rng(W), shape, W, H, proj=1)
                ctx.set_camera_dict(cam)
                ctx.set_render_params("dvr", 1.0, 0.97)
                grad = torch.randn((H, W, 4), device="cuda", generator=torch.Generator(device="cuda").manual_seed(W))
                gl, gv = torch.empty((37, 4), device="cuda"), torch.zeros(shape[::-1], device="cuda")
                ctx.render_backward(cid, grad, gl, gv)
                got[-1] += [gl.cpu().numpy(), gv[:, ::7, ::5].cpu().numpy()]
                del gv
    ctx.close()
    assert max(float(np.abs(a).max()) for a in got[0][:6]) > 0.05
    for i, (a, b) in enumerate(zip(*got)):
        # frames bit for bit; gradients to the order of their FP32 sums
        assert np.array_equal(a, b) if i < 12 else np.abs(a - b).max() <= 2e-4 * np.abs(a).max()
