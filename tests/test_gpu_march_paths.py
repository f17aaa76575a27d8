"""GPU parity of the raymarch's special paths against the FP64 oracle: tile
periods so short that a ray spans thousands of them, light samples that leave
the layer, step counts that do not fill a chunk, and rays in clear air.

Tolerances (max-abs RGBA) are those of every other render: 1e-4 for FP32
volumes, 3e-3 for FP16 volumes."""
import ctypes

import numpy as np
import pytest

from paper_1609_05344_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-4, "fp16": 3e-3}


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1609_05344_gb300 import _native, api as A
    _native.build()
    return A


def _check(api, oracle, desc, prm, cam, w, h, steps, light_steps, frame=-1):
    vol, ovol = api.Volume(desc), oracle.Volume(desc)
    got, count = api.render(vol, cam, prm, w, h, steps, light_steps, jitter_frame=frame, count=True)
    ref, n = oracle.render(ovol, cam, prm, w, h, steps, light_steps, jitter_frame=frame, nthreads=8)
    assert np.abs(got.cpu().numpy() - ref).max() <= TOL[desc["precision"]]
    return ref, int(count.item()), n


# 40 km rays: 1000 periods of 39 m or less take the reduction modulo 2^32; at 1 m a ray spans
# 2^47 fixed-point units and the low part of the double-float product is far above one of them
@pytest.mark.parametrize("kind,base_period", [("tiny", 1.0), ("tiny", 4.0), ("tiny", 39.0),
                                              ("tiny", 41.0), ("full", 16.0), ("full", 256.0),
                                              ("full", 400.0)])
@pytest.mark.parametrize("height", [500.0, 2500.0])
def test_short_tile_periods(api, oracle, kind, base_period, height):
    desc = I.volume_desc(kind, seed=5, base_period=base_period, detail_period=base_period / 8.0)
    cam = I.camera((12345.6, -2345.6, height), 33.0, 36.0, 60.0)
    ref, _, _ = _check(api, oracle, desc, I.params(), cam, 45, 31, 9, 6, frame=2)
    assert ref[..., 3].max() > 0.1


# the light march ends 2.0 km (0.8 km, 0.5 km) above its view sample in a 2.5 km layer
@pytest.mark.parametrize("light_step,light_steps", [(420.0, 6), (180.0, 6), (100.0, 9)])
@pytest.mark.parametrize("kind,precision", [("full", "fp32"), ("full", "fp16"), ("tiny", "fp32")])
@pytest.mark.parametrize("height,pitch", [(500.0, 36.0), (5200.0, -40.0)])
def test_light_samples_above_the_layer(api, oracle, light_step, light_steps, kind, precision, height,
                                       pitch):
    desc = I.volume_desc(kind, seed=6, precision=precision)
    cam = I.camera((800.0, 300.0, height), 120.0, pitch, 60.0)
    ref, _, _ = _check(api, oracle, desc, I.params(light_step=light_step), cam, 40, 27, 17,
                       light_steps, frame=3)
    assert ref[..., 3].max() > 0.1


# 1 and 7: part of a chunk; 11 and 17: whole chunks and a part; 130: mostly clear chunks
@pytest.mark.parametrize("steps", [1, 7, 11, 17, 130])
@pytest.mark.parametrize("config", [0, 4])
def test_partial_and_clear_chunks(api, oracle, steps, config):
    desc = I.volume_desc("full", seed=7)
    api.set_launch_config("fp32", 6, config)
    try:
        cam = I.camera((0.0, 0.0, 500.0), 70.0, 36.0, 60.0)
        ref, count, n = _check(api, oracle, desc, I.params(), cam, 330, 240, steps, 6)
    finally:
        api.set_launch_config("fp32", 6, 3)
    # lookups in the method's sense: a density within rounding of 0, or an optical depth
    # within rounding of the early out, may move single steps of single rays
    assert abs(count - n) <= 1e-3 * n + 6


# the edges of the rule that spreads small images over more warps (4, 8, 16 and 32 rays each):
# 9728, 38912 and 77824 pixels, ragged against every tile; the multi-view launch always has 32
@pytest.mark.parametrize("w,h", [(1, 1), (5, 3), (64, 152), (97, 101), (256, 152), (261, 151), (304, 256),
                                 (307, 257)])
@pytest.mark.parametrize("kind,precision,base_n", [("full", "fp32", 128), ("full", "bf16", 128),
                                                   ("full", "fp16", 64), ("tiny", "fp32", 64),
                                                   ("tiny", "unorm16", 32)])
@pytest.mark.parametrize("steps", [8, 21])
def test_small_images_equal_batched_views(api, w, h, kind, precision, base_n, steps):
    import torch
    vol = api.Volume(I.volume_desc(kind, seed=8, precision=precision, base_n=base_n))
    cam = I.camera((100.0, -700.0, 500.0), 210.0, 36.0, 60.0)
    view = dict(camera=cam, width=w, height=h, steps=steps, jitter_frame=5)
    for light_steps in (6, 3):
        one, count = api.render(vol, cam, I.params(), w, h, steps, light_steps, jitter_frame=5, count=True)
        batch = api.Batch(vol, I.params(), [view], light_steps)
        assert torch.equal(one, batch.render()[0])
        assert int(count.item()) >= int((one[..., 3] > 0).sum().item())


# constant density: both rules, no, one and the most light steps, the early out after a few
# steps, at once, never and off, no density at all; below, inside and above the layer
@pytest.mark.parametrize("rho0,tau_max", [(0.05, 11.5), (0.002, 0.7), (0.05, 1e-6), (1e-5, 0.0), (0.0, 11.5)])
@pytest.mark.parametrize("integration,light_steps", [("analytic", 6), ("basic", 1), ("analytic", 0), ("basic", 32)])
@pytest.mark.parametrize("height,pitch,w,h,steps", [(500.0, 20.0, 45, 31, 9), (2500.0, 0.0, 307, 257, 21),
                                                    (5200.0, -30.0, 1, 1, 130)])
def test_constant_density(api, oracle, rho0, tau_max, integration, light_steps, height, pitch, w, h, steps):
    desc, prm = I.volume_desc("constant", rho0=rho0), I.params(tau_max=tau_max)
    cam = I.camera((0.0, 0.0, height), 70.0, pitch, 60.0)
    vol, ovol = api.Volume(desc), oracle.Volume(desc)
    got, count = api.render(vol, cam, prm, w, h, steps, light_steps, jitter_frame=4, integration=integration,
                            count=True)
    rule = oracle.ANALYTIC if integration == "analytic" else oracle.BASIC
    ref, n = oracle.render(ovol, cam, prm, w, h, steps, light_steps, jitter_frame=4, integration=rule, nthreads=8)
    assert np.abs(got.cpu().numpy() - ref).max() <= TOL["fp32"]
    assert abs(int(count.item()) - n) <= 1e-3 * n + (0 if rho0 == 0.0 else 1 + light_steps)
    view = dict(camera=cam, width=w, height=h, steps=steps, jitter_frame=4)
    batch = api.Batch(vol, prm, [view, view], light_steps, integration)
    assert all(np.array_equal(o.cpu().numpy(), got.cpu().numpy()) for o in batch.render())


# Light samples of a detail tile far finer than the base tile (2^k of its periods to one of the
# base's) keep the detail tile's own precision.  Vertical one-pixel views at positions that fixed
# point holds exactly, so that only the light offsets are rounded; opaque pixels (alpha >= 0.99),
# whose colour is the sunlight of one step.  Relative tolerance: FP32 interpolation errs by at
# most 1e-6 a density (three roundings of 2^-25 and weights of 2^-23 a tile, over 1 - c), the
# optical depth of six samples of 0.04 x 37 by 9e-6, the exponential and the products by 1e-6.
# A light offset rounded to a base unit is 1/4096 of a detail texel off at 2^16, up to 2e-4 here.
@pytest.mark.parametrize("ratio", [8, 65536])
def test_light_offsets_of_a_fine_detail_tile(api, oracle, ratio):
    desc = I.volume_desc("full", seed=9, base_period=65536.0, detail_period=65536.0 / ratio,
                         detail_weight=0.6, coverage=0.25)
    prm = I.params(ambient=(0.0, 0.0, 0.0), light_step=37.0)
    rng = np.random.default_rng(12)
    views = [dict(camera=dict(pos=(x / 64.0, y / 64.0, 500.0), forward=(0.0, 0.0, 1.0),
                              right=(1.0, 0.0, 0.0), up=(0.0, 1.0, 0.0), tan_half_fovy=0.5),
                  width=1, height=1, steps=1, jitter_frame=-1)
             for x, y in rng.integers(-2 ** 21, 2 ** 21, (256, 2))]
    ovol = oracle.Volume(desc)
    got = np.array([o.cpu().numpy()[0, 0] for o in api.Batch(api.Volume(desc), prm, views).render()])
    ref = np.array([oracle.render(ovol, v["camera"], prm, 1, 1, 1, 6)[0][0, 0] for v in views])
    opaque = ref[:, 3] >= 0.99
    assert opaque.sum() >= 32
    assert np.abs(got[opaque, :3] / ref[opaque, :3] - 1.0).max() <= 1e-5


class _KernelNode(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("shared", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _grid(launch):
    """Grid (x, y) of the one kernel that launch(stream) issues, captured and not run."""
    import torch
    cu, s = ctypes.CDLL("libcuda.so.1"), torch.cuda.Stream()
    handle, graph, node, n = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_size_t(1)
    assert cu.cuStreamBeginCapture_v2(handle, 2) == 0
    try:
        launch(s)
    finally:
        assert cu.cuStreamEndCapture(handle, ctypes.byref(graph)) == 0
    got = _KernelNode()
    assert cu.cuGraphGetNodes(graph, ctypes.byref(node), ctypes.byref(n)) == 0 and n.value == 1
    assert cu.cuGraphKernelNodeGetParams_v2(node, ctypes.byref(got)) == 0
    cu.cuGraphDestroy(graph)
    return tuple(got.grid[:2])


TILES = [(16, 8), (32, 4), (32, 4), (8, 16)]  # of the four shapes


def _tiles(config, w, h):
    tw, th = TILES[config % 4]
    return (w + tw - 1) // tw, (h + th - 1) // th


# a configuration that is set reaches images of every size, the default gives small ones back
# to the rule (8x4 tiles at 203x77), and tuning on one size leaves the other in order
def test_launch_config_reaches_every_size(api):
    import torch
    vol, cam, prm = api.Volume(I.volume_desc("full", seed=3, precision="fp16")), I.orbit_camera(2, 3), I.params()
    sizes = [(203, 77), (411, 203)]
    outs = [torch.empty((h, w, 4), device="cuda") for w, h in sizes]

    def grid(k):
        return _grid(lambda s: api.render(vol, cam, prm, *sizes[k], 8, 6, jitter_frame=1, out=outs[k], stream=s))

    spread = (26, 20)
    api.set_launch_config("fp16", 6, 3)
    try:
        assert grid(0) == spread and grid(1) == _tiles(3, *sizes[1])
        for config in (0, 1, 2, 4, 5, 6, 7):
            api.set_launch_config("fp16", 6, config)
            assert api.launch_config("fp16", 6) == config
            assert [grid(0), grid(1)] == [_tiles(config, *s) for s in sizes]
        best, _ = api.autotune_render(vol, cam, prm, *sizes[1], 8, 6, jitter_frame=1, repeats=2)
        assert api.launch_config("fp16", 6) == best
        assert grid(0) == spread and grid(1) == _tiles(best, *sizes[1])
        best, _ = api.autotune_render(vol, cam, prm, *sizes[0], 8, 6, jitter_frame=1, repeats=2)
        assert api.launch_config("fp16", 6) == best and grid(1) == _tiles(best, *sizes[1])
        assert grid(0) in (spread, _tiles(best, *sizes[0]))
    finally:
        api.set_launch_config("fp16", 6, 3)
    assert grid(0) == spread


# every configuration on an image above the rule for small ones, in marches of one chunk, of
# several and of a part, for the kernels of each kind of volume
@pytest.mark.parametrize("kind,precision,over", [("full", "fp32", {}), ("full", "bf16", {}), ("tiny", "fp32", {}),
                                                 ("tiny", "unorm16", {}), ("full", "fp16", dict(base_n=64)),
                                                 ("constant", "fp32", {})])
@pytest.mark.parametrize("steps", [8, 40])
def test_every_launch_config_on_a_large_image(api, kind, precision, over, steps):
    import torch
    vol = api.Volume(I.volume_desc(kind, seed=3, precision=precision, **over))
    cam, outs = I.orbit_camera(2, 3), []
    try:
        for config in range(8):
            api.set_launch_config(precision, 6, config)
            outs.append(api.render(vol, cam, I.params(), 411, 203, steps, 6, jitter_frame=1))
    finally:
        api.set_launch_config(precision, 6, 3)
    assert outs[0][..., 3].max() > 0.1
    for config in range(1, 8):
        assert torch.equal(outs[0], outs[config]), config


# only standard volumes hold the blocked copy of the occupancy grid (2 MiB): a base tile of the
# standard size alone is 32 MiB of 16-bit records and 2 MiB of grid
def test_blocked_grid_only_where_it_is_read(api):
    import torch
    torch.cuda.synchronize()
    first = api.Volume(I.volume_desc("tiny", seed=1, precision="fp16", base_n=128))  # loads the kernels
    before = torch.cuda.mem_get_info()[0]
    more = [api.Volume(I.volume_desc("tiny", seed=k, precision="fp16", base_n=128)) for k in range(16)]
    used = (before - torch.cuda.mem_get_info()[0]) / len(more) / 2 ** 20
    assert 33.5 <= used <= 35.0
    for v in [first] + more:
        v.close()
