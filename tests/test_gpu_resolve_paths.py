"""GPU parity of the resolve kernels at the edges of their tiles: images one
pixel short of, equal to and one past the tiles of 32x16 and 32x32 pixels, the
separate motion and TAA passes against the FP64 oracle and the fused resolve
bitwise against both, and the composite at the edges of its 32x8 tiles.

Tolerances: motion 1e-4 px, FP32 history 1e-6, FP16 history its storage rounding
(2e-3 for values up to 2), composite 2e-6 (values up to 2)."""
import numpy as np
import pytest

from paper_1609_05344_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_05344_gb300 import _native, api as A
    _native.build()
    return A


def _t(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("w,h", [(31, 15), (32, 16), (33, 17), (32, 32), (65, 33), (2, 49), (97, 1)])
@pytest.mark.parametrize("fmt", ["fp32", "fp16"])
def test_tile_edges(api, oracle, w, h, fmt):
    import torch
    rng = np.random.default_rng(100 * w + h)
    hist, cur = I.synthetic_frame(rng, h, w), I.synthetic_frame(rng, h, w)
    hist = hist.astype(np.float16) if fmt == "fp16" else hist
    mot = I.synthetic_motion(rng, h, w, offscreen_frac=0.1)
    got = api.taa(_t(hist), _t(cur), _t(mot), history_fmt=fmt).cpu().numpy()
    ref = oracle.taa(hist.astype(np.float64), cur, mot)
    assert np.abs(got.astype(np.float64) - ref).max() <= (1e-6 if fmt == "fp32" else 2e-3)
    # motion, and the fused resolve equal to motion followed by TAA
    desc, prm = I.volume_desc("tiny", seed=1), I.params()
    vol = api.Volume(desc)
    prev, cam = I.orbit_camera(4, 3), I.orbit_camera(5, 3)
    m = api.motion(vol, prm, prev, cam, w, h)
    assert np.abs(m.cpu().numpy() - oracle.motion(desc, prm, prev, cam, w, h)).max() <= 1e-4
    sep = api.taa(_t(hist), _t(cur), m, history_fmt=fmt)
    fused = api.taa_reproject(vol, prm, prev, cam, _t(hist), _t(cur), history_fmt=fmt)
    assert torch.equal(sep, fused)


# a first frame is the current frame in the history's format, whatever the motion
@pytest.mark.parametrize("w,h", [(1, 1), (255, 1), (16, 16), (257, 1), (97, 61)])
@pytest.mark.parametrize("fmt", ["fp32", "fp16"])
def test_first_frame_is_the_current_frame(api, w, h, fmt):
    import torch
    rng = np.random.default_rng(w + h)
    cur, mot = _t(I.synthetic_frame(rng, h, w)), _t(I.synthetic_motion(rng, h, w))
    got = api.taa(None, cur, mot, history_fmt=fmt)
    assert torch.equal(got, cur if fmt == "fp32" else cur.half())


# on both sides of the rules that give small images fewer pixels a thread: 152 tiles of
# 32x32 pixels (motion) and of 32x16 (TAA), and the rows that a thread has beyond the image
@pytest.mark.parametrize("w,h", [(31, 1), (33, 17), (608, 255), (609, 225), (304, 256), (577, 129), (640, 305)])
@pytest.mark.parametrize("fmt", ["fp32", "fp16"])
def test_small_images_resolve_as_large_ones(api, oracle, w, h, fmt):
    import torch
    rng = np.random.default_rng(w * h)
    hist, cur = I.synthetic_frame(rng, h, w), I.synthetic_frame(rng, h, w)
    hist = hist.astype(np.float16) if fmt == "fp16" else hist
    desc, prm = I.volume_desc("tiny", seed=1), I.params()
    prev, cam = I.orbit_camera(7, 3), I.orbit_camera(8, 3)
    vol = api.Volume(desc)
    mot = api.motion(vol, prm, prev, cam, w, h)
    assert np.abs(mot.cpu().numpy() - oracle.motion(desc, prm, prev, cam, w, h)).max() <= 1e-4
    got = api.taa(_t(hist), _t(cur), mot, history_fmt=fmt)
    ref = oracle.taa(hist.astype(np.float64), cur, mot.cpu().numpy())
    assert np.abs(got.cpu().numpy().astype(np.float64) - ref).max() <= (1e-6 if fmt == "fp32" else 2e-3)
    fused = api.taa_reproject(vol, prm, prev, cam, _t(hist), _t(cur), history_fmt=fmt)
    assert torch.equal(got, fused)


# one pixel, one short of, equal to and one past the 32x8 tiles; the cloud at the display's size,
# odd fractions of it and larger than it
@pytest.mark.parametrize("w,h,cw,ch", [(1, 1, 1, 1), (31, 7, 13, 3), (32, 8, 32, 8), (33, 9, 11, 9),
                                       (97, 61, 32, 21), (40, 17, 81, 35)])
@pytest.mark.parametrize("fmt", ["fp32", "fp16"])
def test_composite_tile_edges(api, oracle, w, h, cw, ch, fmt):
    rng = np.random.default_rng(w * h + cw)
    cloud, bg = I.synthetic_frame(rng, ch, cw), rng.uniform(0.0, 2.0, (h, w, 4)).astype(np.float32)
    cloud = cloud.astype(np.float16) if fmt == "fp16" else cloud
    got = api.composite(_t(cloud), _t(bg)).cpu().numpy()
    assert np.abs(got - oracle.composite(cloud.astype(np.float64), bg)).max() <= 2e-6
