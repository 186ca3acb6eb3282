"""Memory that freed cubes and closed serving loops leave to the next ones: whatever it held before, a
frame is that of a fresh context, and everything is given back with the context."""
import numpy as np
import pytest

import synth
from gpu_helpers import gpu_ctx

pytestmark = pytest.mark.gpu

CAM = dict(view=synth.look_at((120.0, 40.0, -60.0), (20.0, 25.0, 19.0)), proj=1, param=0.4, W=90, H=70)


def _ctx():
    gpu_ctx().close()                  # (builds; skips without a device)
    import paper_1008_0135_gb300 as P
    return P.Context(0, cache_bytes=64 << 20)


def _frames(ctx, cid):
    out = []
    ctx.set_camera_dict(CAM)
    for mode in ("dvr", "mip"):
        ctx.set_render_params(mode, 0.5, 0.97)
        out.append(ctx.render_frame(cid).cpu().numpy())
    return out


def _cycle(ctx, cube, storage, mask, brick, compressed):
    cid = ctx.load_cube(cube)
    ctx.set_brick_layouts(cid, mask)
    ctx.set_transfer_function(synth.random_lut(3, n=37), -8.0, 9.0)
    if compressed:
        ctx.compress_cube(cid)
    ctx.set_bricking(cid, brick, 1, storage)
    out = _frames(ctx, cid)
    ctx.free_cube(cid)
    return out


# odd bricks whose records, rows and atlas cells leave gaps that no build writes; one brick; compressed
@pytest.mark.parametrize("shape,brick,storage,mask,compressed",
                         [((41, 50, 38), (16, 19, 13), "f32", 9, False), ((41, 50, 38), (16, 19, 13), "f16", 31, False),
                          ((41, 50, 38), (16, 19, 13), "bf16", 41, False), ((41, 50, 38), (64, 64, 64), "f16", 9, False),
                          ((41, 50, 38), (16, 19, 13), "f32", 9, True)])
def test_a_cube_in_left_memory_is_a_cube_in_fresh_memory(shape, brick, storage, mask, compressed):
    import torch
    rng = np.random.default_rng(1)
    cube = (3.0 * rng.standard_normal(shape[::-1])).astype(np.float32)
    left = np.full_like(cube, np.nan if not compressed else 3e38)
    free = []
    for k in range(3):
        fresh, used = _ctx(), _ctx()
        want = _cycle(fresh, cube, storage, mask, brick, compressed)
        fresh.close()
        _cycle(used, left, storage, mask, brick, compressed)
        for _ in range(2):
            got = _cycle(used, cube, storage, mask, brick, compressed)
            assert all(np.array_equal(a, b) for a, b in zip(want, got))
        used.close()
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    assert max(float(np.abs(a).max()) for a in want) > 0.05
    assert free[2] >= free[1]


def test_serving_loops_hand_their_slots_on():
    """Loops of more, fewer and larger frames one after the other, and an online loop between: every
    frame is the one the context renders by itself."""
    import torch
    ctx = gpu_ctx()
    cube = (3.0 * np.random.default_rng(2).standard_normal((38, 50, 41))).astype(np.float32)
    cid = ctx.load_cube(cube)
    ctx.set_brick_layouts(cid, 9)
    ctx.set_bricking(cid, (16, 16, 16), 1, "f16")
    lut = synth.random_lut(3, n=37)
    ctx.set_transfer_function(lut, -8.0, 9.0)
    ctx.set_render_params("dvr", 0.5, 0.97)

    def reqs(n, W, H):
        rng = np.random.default_rng(n)
        cams = [synth.random_camera(rng, (41, 50, 38), W, H, proj=k % 2) for k in range(n)]
        return [dict(cube=cid, cam=c, mode="dvr", step=0.5, tau=0.97, lut=lut, vrange=(-8.0, 9.0), arrival_ms=0.0,
                     out=torch.full((H, W, 4), float("nan"), device="cuda")) for c in cams]

    def check(rs):
        for r in rs:
            ctx.set_camera_dict(r["cam"])
            assert torch.equal(ctx.render_frame(cid), r["out"])

    for n, inflight, W, H in ((3, 2, 40, 30), (9, 20, 150, 130), (5, 1, 64, 48), (20, 17, 33, 21)):
        rs = reqs(n, W, H)
        results, _ = ctx.serve(rs, max_inflight=inflight)
        assert all(r["status"] == 0 for r in results)
        check(rs)
    rs = reqs(4, 70, 60)
    server = ctx.serve_online(3)
    for r in rs:
        server.submit(r)
    server.close()
    check(rs)
    ctx.close()


def test_a_freed_cube_leaves_no_more_than_its_bound():
    """What vr_free_cube keeps above 2 GiB is back with the device when it returns (32 MiB for other users)."""
    import torch
    ctx = _ctx()
    cid = ctx.load_cube(np.zeros((700, 1000, 1000), np.float32))
    torch.cuda.synchronize()
    with_cube = torch.cuda.mem_get_info()[0]
    ctx.free_cube(cid)
    freed = torch.cuda.mem_get_info()[0] - with_cube
    ctx.close()
    assert freed >= 4 * 700 * 1000 * 1000 - (2 << 30) - (32 << 20)
