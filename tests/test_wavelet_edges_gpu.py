"""Wavelet encoder and decoder at their edges, bit for bit against the oracle, and slots decoded into
atlases alone."""
import numpy as np
import pytest

import synth
from gpu_helpers import gpu_ctx

pytestmark = pytest.mark.gpu


def _ctx(nbytes=64 << 20):
    gpu_ctx().close()                      # skips without a GPU, builds the library
    import paper_1008_0135_gb300 as P
    return P.Context(0, cache_bytes=nbytes)


@pytest.mark.parametrize("shape", [(8, 8, 8), (9, 7, 5), (34, 17, 23), (70, 24, 41)])
def test_store_and_bricks_of_ragged_and_special_cubes(orc, shape):
    """Encoder and decoder against the oracle bit for bit: whole and ragged blocks, odd rows (no paired
    loads), zeros, denormals, huge values; bricks that start inside blocks."""
    rng = np.random.default_rng(shape[0])
    c = _ctx()
    for kind in range(4):
        cube = rng.standard_normal(shape[::-1]).astype(np.float32)
        if kind == 1:
            cube[...] = 0.0
            cube[0, 0, 0] = 3.0
        elif kind == 2:
            cube *= np.float32(1e-40)
        elif kind == 3:
            cube *= np.exp(40.0 * rng.uniform(-1, 1, cube.shape)).astype(np.float32)
        cid = c.load_cube(cube)
        c.compress_cube(cid)
        store = orc.wavelet_encode(cube)
        assert np.array_equal(c.wavelet_store(cid), np.asarray(store).ravel())
        want = np.pad(orc.wavelet_decode(store, cube.shape), 1, mode="edge")
        c.set_bricking(cid, (13, 8, 21), 1, "f32")
        nb, _ = c.brick_grid(cid)
        for b in range(int(np.prod(nb))):
            dims, org, _, data = c.get_brick(cid, b)
            assert np.array_equal(data, want[org[2] + 1:org[2] + 1 + dims[2], org[1] + 1:org[1] + 1 + dims[1],
                                             org[0] + 1:org[0] + 1 + dims[0]])
        c.free_cube(cid)
    c.close()


def test_slots_decoded_into_atlases_serve_linear_frames_and_other_cubes():
    """A compressed cube's bricks are decoded into the slots' atlases alone: a camera that needs the
    linear copies, and slots whose arrays another cube replaced, decode them again."""
    rng = np.random.default_rng(2)
    cube = (3.0 * rng.standard_normal((40, 44, 50))).astype(np.float32)
    lut = synth.random_lut(6, n=40)
    near = synth.random_camera(rng, (50, 44, 40), 80, 60, proj=1)
    m = np.array([25.0, 22.0, 20.0])
    far = dict(view=synth.look_at(m + 3e5 * np.array([0.0, 0.0, 1.0]), m), proj=1, param=2e-4, W=80, H=60)
    got = []
    for mask in (1, 9):
        c = _ctx()
        c.set_transfer_function(lut, -8.0, 8.0)
        cid = c.load_cube(cube)
        c.compress_cube(cid)
        c.set_brick_layouts(cid, mask)
        c.set_bricking(cid, (24, 24, 24), 1, "f32")
        c.set_render_params("dvr", 0.8, 0.98)
        frames = []
        c.set_camera_dict(near)
        frames.append(c.render_frame(cid).cpu().numpy())
        # another cube, whose stored bricks (40x20x20) fit the slots cut for 26^3 but not their arrays: its
        # bricking replaces the arrays of as many slots as it has bricks, the first cube's among them
        other = c.load_cube((3.0 * rng.standard_normal((36, 54, 76))).astype(np.float32))
        c.compress_cube(other)
        c.set_brick_layouts(other, mask)
        c.set_bricking(other, (38, 18, 18), 1, "f32")
        misses, hits = c.stats()["cache_misses"], c.stats()["cache_hits"]
        frames.append(c.render_frame(cid).cpu().numpy())      # all still in their slots, their atlases gone
        assert c.stats()["cache_misses"] == misses and c.stats()["cache_hits"] == hits + 12
        for cam in (far, near):
            c.set_camera_dict(cam)
            frames.append(c.render_frame(cid).cpu().numpy())
        c.render_frame(other)
        frames.append(c.render_frame(cid).cpu().numpy())
        got.append(frames)
        c.close()
    assert all(np.array_equal(a, b) for a, b in zip(*got))
    assert np.abs(got[0][2]).max() > 0.05
