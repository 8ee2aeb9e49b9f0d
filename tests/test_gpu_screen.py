"""The screened passes (csrc/pcr_screen.cuh), which the exact transform runs with default tuning on LINEAR and METRIC
views, against the FP64 kernels, bit for bit: sizes at the edges of tiles, warps and blocks, dense runs on one pixel,
codes next to the stored one and to the band's edges, bands the screen leaves to k_hq_cert, keys left by another depth
mapping or another cloud."""
from __future__ import annotations

import numpy as np
import pytest

import scenes
from tests.helpers import RawView, axis_view, pack

pytestmark = pytest.mark.gpu


def _dev(points):
    import torch
    return torch.from_numpy(np.ascontiguousarray(points).view(np.int32)).cuda()


def _view(v, depth=0, scale=1000.0, transform=0):
    return RawView(np.asarray(v.view_proj), v.near, v.far, v.width, v.height, depth, scale, None, transform)


def _frames(gpu, dev, v, depth, scale, eps, before=None, accumulate=False, tuning=None):
    """Keys and sums of one frame by the exact and by the FP64 transform."""
    res = []
    for transform in (0, 1):
        fb = gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ)
        if tuning and transform == 0:
            gpu.pcr_set_tuning(fb, **tuning)
        view = _view(v, depth, scale, transform)
        if before:
            before(fb)
        if accumulate:
            gpu.pcr_hq_accumulate(fb, dev, view, *eps)
        else:
            gpu.pcr_render_hq_splat(fb, dev, view, *eps)
        keys, acc = gpu.pcr_framebuffer_keys(fb)
        res.append((keys.clone(), acc.clone()))
        assert gpu.pcr_get_device_status(fb) == gpu.PCR_OK
        fb.close()
    assert int((res[0][0] != res[1][0]).sum()) == 0
    assert int((res[0][1] != res[1][1]).sum()) == 0
    return res[0]


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 127, 129, 2047, 2048, 2049, 38911, 38913, 152 * 2048 + 1, 700001])
def test_sizes(gpu, n):
    v = scenes.lidar_1km_view(320, 180)
    keys, _ = _frames(gpu, _dev(scenes.lidar(n, 41)), v, 0, 1.0, (1, 100))
    assert int((keys != -1).sum()) > 0 or n < 64


@pytest.mark.parametrize("depth,scale", [(0, 1.0), (1, 1000.0), (1, 1e6), (1, 1e8)])
@pytest.mark.parametrize("eps", [(1, 100), (0, 1), (3, 1), (1, 1 << 20), (1 << 20, 1), (16_000_000, 1 << 20)])
def test_depth_modes_and_bands(gpu, depth, scale, eps):
    v = scenes.lidar_1km_view(160, 90)
    pts = scenes.lidar(400_001, 42)
    scenes.shuffle(pts, 3)
    _frames(gpu, _dev(pts), v, depth, scale, eps)


@pytest.mark.parametrize("spread", [0.0, 1e-7, 1e-6, 1e-4, 1e-2])
@pytest.mark.parametrize("eps", [(1, 100), (1, 1 << 20), (0, 1)])
def test_codes_next_to_the_stored_one(gpu, spread, eps):
    """Many points on few pixels in one depth sheet: codes from equal to a few units apart, in runs and shuffled."""
    rng = np.random.default_rng(7)
    n = 100_000
    w = 3.0 * (1.0 + spread * rng.random(n))
    ndc = np.repeat(rng.uniform(-0.9, 0.9, (n // 50, 2)), 50, axis=0) + rng.uniform(0, 1e-3, (n, 2))
    pts = pack(np.column_stack([ndc[:, 0] * w, ndc[:, 1] * w, -w]), rng.integers(0, 1 << 32, n, dtype=np.uint64))
    for _ in range(2):
        _frames(gpu, _dev(pts), axis_view(64, 48), 0, 1.0, eps)
        rng.shuffle(pts)


def test_one_pixel_and_every_tuned_grid(gpu):
    rng = np.random.default_rng(8)
    w = rng.uniform(1.0, 8.0, 300_000)
    pts = _dev(pack(np.column_stack([0.01 * w, 0.01 * w, -w]), np.arange(300_000, dtype=np.uint32)))
    for blocks in (1, 2, 3, 8, 32):
        _frames(gpu, pts, axis_view(64, 48), 0, 1.0, (1, 10), tuning={"blocks_per_sm": blocks})


@pytest.mark.parametrize("depth,scale", [(0, 1.0), (1, 1000.0), (1, 1e8)])
def test_keys_of_another_mapping_and_cloud(gpu, depth, scale):
    """A frame on keys that a LINEAR view and another cloud left (larger and smaller codes than the frame's own), and
    pass 2 alone on such keys (points in front of their pixel's key are outside the band) and on an empty framebuffer."""
    v = scenes.lidar_1km_view(200, 120)
    other, dev = _dev(scenes.lidar(50_000, 44)), _dev(scenes.lidar(300_000, 45))

    def before(fb):
        gpu.pcr_render_atomicmin(fb, other, _view(v, 0))

    _frames(gpu, dev, v, depth, scale, (1, 100), before)
    _frames(gpu, dev, v, depth, scale, (1, 100), before, accumulate=True)
    _frames(gpu, dev, v, depth, scale, (1, 100), accumulate=True)


def test_special_coordinates(gpu):
    pts = scenes.lidar(200_000, 46)
    f = pts[:, :3].view(np.float32)
    rng = np.random.default_rng(9)
    for value in (np.nan, np.inf, -np.inf, 3e38, -3e38, 1e20, 1e-42, 0.0, -0.0):
        f[rng.integers(0, len(pts), 800), rng.integers(0, 3, 800)] = value
    for depth, scale in ((0, 1.0), (1, 1000.0)):
        _frames(gpu, _dev(pts), scenes.lidar_1km_view(320, 180), depth, scale, (1, 100))


def test_visible_points_whose_magnitude_sum_overflows(gpu):
    """|x| + |y| + |z| is infinite in float, yet the FP64 definition draws the point: it must count once."""
    m = np.zeros((4, 4))
    m[0, 0], m[0, 1], m[1, 2], m[2, 2], m[3, 2] = 1.0, -1.0, 0.25, -1.0, -1.0
    n = 5000
    rng = np.random.default_rng(10)
    big = rng.uniform(2.0e38, 3.0e38, n).astype(np.float32)
    pts = pack(np.column_stack([big, big, -rng.uniform(1.0, 8.0, n)]), rng.integers(0, 1 << 32, n, dtype=np.uint64))
    _, acc = _frames(gpu, _dev(pts), RawView(m, 0.5, 8.5, 64, 48), 0, 1.0, (10, 1))
    assert int((acc[:, 1] >> 32).sum()) == n


@pytest.mark.parametrize("looking_away", [False, True])
def test_clouds_mostly_outside_the_view(gpu, looking_away):
    """Enough tiles a warp that pass 1 samples the cloud; a camera inside the scan has most points outside its planes."""
    n = 128 * 152 * 8 * 64 + 12345
    dev = _dev(scenes.lidar(n, 47))
    v = scenes.View.lookat((500, 500, 60), (1500, 500, 40) if looking_away else (0, 480, 0), (0, 0, 1), 60.0, 640, 360, 0.1, 300.0)
    _frames(gpu, dev, v, 0, 1.0, (1, 100), tuning={"blocks_per_sm": 1})


@pytest.mark.parametrize("n", [1, 31, 33, 63, 64, 65, 2049, 152 * 256 + 1, 500_003])
@pytest.mark.parametrize("depth", [0, 1, 2])
def test_projection_sizes(gpu, n, depth):
    """pcr_project_points by the exact transform (k_project_cert) against the FP64 kernel, point by point."""
    import torch
    dev = _dev(scenes.lidar(n, 48))
    v = scenes.lidar_1km_view(320, 180)
    ranges = np.array([[0.0, 10.0, 1e9], [10.0, 600.0, 1e6], [600.0, 5000.0, 1e3]])
    got = [gpu.pcr_project_points(dev, RawView(np.asarray(v.view_proj), v.near, v.far, 320, 180, depth, 1000.0, ranges, t))
           for t in (0, 1)]
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("depth,scale", [(0, 1.0), (1, 1000.0)])
def test_clouds_in_random_order(gpu, depth, scale):
    """Enough tiles a warp that the passes sample the cloud and, in random order, pass 1 leaves pass 2 its words: at eps up
    to 1, on a second frame, after a smaller cloud, with bands above 1 (without words), and captured."""
    import torch
    n = 97 * 152 * 8 * 64 + 4321
    pts = scenes.lidar(n, 49)
    scenes.shuffle(pts, 2)
    dev, v = _dev(pts), scenes.lidar_1km_view(400, 225)
    one = {"blocks_per_sm": 1}
    for eps in ((1, 100), (1, 1), (3, 2), (0, 1)):
        want = _frames(gpu, dev, v, depth, scale, eps, tuning=one)
        fb = gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ)
        gpu.pcr_set_tuning(fb, **one)
        view = _view(v, depth, scale)
        keys, acc = gpu.pcr_framebuffer_keys(fb)
        for points in (dev, dev[:300_001], dev):
            gpu.pcr_clear(fb)
            gpu.pcr_render_hq_splat(fb, points, view, *eps)
        assert torch.equal(keys, want[0]) and torch.equal(acc, want[1])
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            gpu.pcr_clear(fb)
            gpu.pcr_render_hq_splat(fb, dev, view, *eps)
        acc.fill_(5)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(keys, want[0]) and torch.equal(acc, want[1])
        del graph
        fb.close()


def test_words_memory_only_after_random_order(gpu):
    """The memory of pass 1's words is taken by the frame after one that found its cloud in random order, not by frames in
    scan order; the frames are the same before and after."""
    import torch
    n = 20_000_003
    pts = scenes.lidar(n, 50)
    scan = _dev(pts)
    scenes.shuffle(pts, 3)
    v, one = scenes.lidar_1km_view(400, 225), {"blocks_per_sm": 1}
    view = _view(v)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def frame(fb, points):
        gpu.pcr_clear(fb)
        gpu.pcr_render_hq_splat(fb, points, view)
        return tuple(t.clone() for t in gpu.pcr_framebuffer_keys(fb))

    for order in ("warm-up", "scan", "shuffled"):
        points = scan if order == "scan" else _dev(pts)
        want = _frames(gpu, points, v, 0, 1.0, (1, 100), tuning=one)
        fb = gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ)
        gpu.pcr_set_tuning(fb, **one)
        frame(fb, points[:100_000])  # its results' memory is taken
        left = [free()]
        for _ in range(3):
            got = frame(fb, points)
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
            left.append(free())
        if order != "warm-up":
            assert left[1] == left[0] and left[3] == left[2]
            assert (left[2] < left[1]) == (order == "shuffled")
        fb.close()


def test_words_memory_while_another_stream_is_captured(gpu):
    """A frame that takes the words' memory, on a stream of its own, leaves a capture in progress on another stream (in the
    global mode, torch's default) as it is."""
    import torch
    n = 97 * 152 * 8 * 64 + 4321
    pts = scenes.lidar(n, 49)
    scenes.shuffle(pts, 2)
    dev, v, side = _dev(pts), scenes.lidar_1km_view(400, 225), torch.cuda.Stream()
    want = _frames(gpu, dev, v, 0, 1.0, (1, 100), tuning={"blocks_per_sm": 1})
    x = torch.zeros(1000, device="cuda")
    for frames_before in (0, 1):
        fb = gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ)
        gpu.pcr_set_tuning(fb, blocks_per_sm=1)
        for _ in range(frames_before):
            gpu.pcr_render_hq_splat(fb, dev, _view(v))
        gpu.pcr_clear(fb)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            x += 1
            gpu.pcr_render_hq_splat(fb, dev, _view(v), stream=side)
            x += 1
        graph.replay()
        torch.cuda.synchronize()
        keys, acc = gpu.pcr_framebuffer_keys(fb)
        assert torch.equal(keys, want[0]) and torch.equal(acc, want[1])
        del graph
        fb.close()
    assert float(x[0]) == 4.0


@pytest.mark.parametrize("tiles", [95, 96])
@pytest.mark.parametrize("cloud", ["scan", "shuffled", "away"])
def test_sampled_loops(gpu, cloud, tiles):
    """Clouds on both sides of the sample's line, in tiles a warp of the device at hand, that every block finds in random
    order (the second frame then takes pass 1's words), mostly outside the clip planes, or neither; the restated decision
    says which loop ran."""
    import torch
    from tests.test_screen_restated import SAMPLE_TILES, sample_decisions
    blocks, warps = torch.cuda.get_device_properties(0).multi_processor_count, 8
    pts = scenes.lidar(tiles * blocks * warps * 64 + 17, 51)
    if cloud == "shuffled":
        scenes.shuffle(pts, 4)
    v = scenes.lidar_1km_view(320, 180)
    if cloud == "away":
        v = scenes.View.lookat((500, 500, 60), (1500, 500, 40), (0, 0, 1), 60.0, 320, 180, 0.1, 100.0)
    found = sample_decisions(pts, v, blocks, warps)
    assert (found is None) == (tiles < SAMPLE_TILES)
    if found is not None:
        assert found[0].all() if cloud == "away" else not found[0].any()
        assert cloud == "away" or (found[1].all() if cloud == "shuffled" else not found[1].any())
    dev, one = _dev(pts), {"blocks_per_sm": 1}
    want = _frames(gpu, dev, v, 0, 1.0, (1, 100), tuning=one)
    fb = gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ)
    gpu.pcr_set_tuning(fb, **one)
    for _ in range(3):
        gpu.pcr_clear(fb)
        gpu.pcr_render_hq_splat(fb, dev, _view(v))
        torch.cuda.synchronize()
        for a, b in zip(gpu.pcr_framebuffer_keys(fb), want):
            assert torch.equal(a, b)
    fb.close()


RANGES = {1: [[0.0, 5000.0, 2e8]], 2: [[0.0, 4.0, 1e9], [4.0, 5000.0, 1e6]],
          3: [[0.0, 2.0, 1e9], [2.0, 4.0, 1e11], [4.0, 5000.0, 1e3]],
          5: [[0.0, 1.0, 1e8], [1.0, 3.0, 1e3], [3.1, 3.2, 1e9], [3.2, 3.5, 1e11], [3.5, 5000.0, 1e4]]}


def _piecewise_keys(gpu, dev, v, ranges, before=None):
    """Keys of one pass 1 by the exact and by the FP64 transform."""
    res = []
    for transform in (0, 1):
        fb = gpu.pcr_create_framebuffer(v.width, v.height)
        if before:
            before(fb)
        gpu.pcr_render_atomicmin(fb, dev, RawView(np.asarray(v.view_proj), v.near, v.far, v.width, v.height, 2, 1000.0,
                                                  np.asarray(ranges), transform))
        res.append(gpu.pcr_framebuffer_keys(fb)[0].clone())
        fb.close()
    assert int((res[0] != res[1]).sum()) == 0
    return res[0]


@pytest.mark.parametrize("n_ranges", sorted(RANGES))
@pytest.mark.parametrize("spread", [0.0, 1e-7, 1e-4, 1.0])
def test_piecewise_codes_next_to_the_stored_one(gpu, spread, n_ranges):
    """As test_codes_next_to_the_stored_one, PIECEWISE: sheets inside a range, at a boundary and across all of them, on
    empty keys and on keys that another mapping left."""
    rng = np.random.default_rng(11)
    n = 100_000
    v = axis_view(64, 48)
    for centre in (2.9, 3.2, 4.0):
        w = centre * (1.0 + spread * (rng.random(n) - 0.5))
        ndc = np.repeat(rng.uniform(-0.9, 0.9, (n // 50, 2)), 50, axis=0) + rng.uniform(0, 1e-3, (n, 2))
        pts = pack(np.column_stack([ndc[:, 0] * w, ndc[:, 1] * w, -w]), rng.integers(0, 1 << 32, n, dtype=np.uint64))
        for _ in range(2):
            dev = _dev(pts)
            keys = _piecewise_keys(gpu, dev, v, RANGES[n_ranges])
            assert int((keys != -1).sum()) > 0
            _piecewise_keys(gpu, dev, v, RANGES[n_ranges], lambda fb: gpu.pcr_render_atomicmin(fb, dev, v))
            rng.shuffle(pts)


@pytest.mark.parametrize("n_ranges", sorted(RANGES))
def test_piecewise_special_coordinates(gpu, n_ranges):
    pts = scenes.lidar(200_000, 52)
    f = pts[:, :3].view(np.float32)
    rng = np.random.default_rng(12)
    for value in (np.nan, np.inf, -np.inf, 3e38, -3e38, 1e20, 1e-42, 0.0, -0.0):
        f[rng.integers(0, len(pts), 800), rng.integers(0, 3, 800)] = value
    scale = np.array([[250.0, 250.0, 1 / 250.0]])  # the same codes over 250 times the depth
    _piecewise_keys(gpu, _dev(pts), scenes.lidar_1km_view(320, 180), np.asarray(RANGES[n_ranges]) * scale)
