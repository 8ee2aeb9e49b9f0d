"""Work items of the batch kernel (k_batch_pass) at the edges of chunks, mask words and item sizes: every view's keys and
sums equal the single-view frame's."""
from __future__ import annotations

import pytest

import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 5 * 1024, 31 * 1024 + 7, 32 * 1024, 33 * 1024 + 1, 700_001, 2_500_003])
@pytest.mark.parametrize("slice_words", [1, 4])
def test_items(gpu, n, slice_words):
    import torch
    dev = torch.from_numpy(scenes.lidar(n, 61).view("int32")).cuda()
    views = scenes.orbit_views(6, 3, resolutions=((200, 120), (333, 95)))
    fbs = [gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ) for v in views]
    outs = [torch.zeros(v.width * v.height, dtype=torch.int32, device="cuda") for v in views]
    batch = gpu.pcr_batch_create(gpu.pcr_cloud_create(dev), fbs, outs, True, 1, 100, 0, False)
    gpu.pcr_batch_set_views(batch, views)
    gpu.pcr_batch_set_tuning(batch, {"route": 1, "slice_words": slice_words})
    gpu.pcr_batch_render(batch)
    for v, fb in zip(views, fbs):
        one = gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ)
        gpu.pcr_render_hq_splat(one, dev, v, 1, 100)
        for a, b in zip(gpu.pcr_framebuffer_keys(fb), gpu.pcr_framebuffer_keys(one)):
            assert torch.equal(a, b)
    batch.close()


def test_captured_views_of_the_screened_pass(gpu):
    """High-quality frames large enough that pass 2 runs one screened launch per view (with the view's chunk mask): a
    captured frame follows new views, other depth units, views the screen cannot take (depth codes in units of 1e26 m)
    and back, and cameras that see little of the cloud, replayed on the legacy default stream."""
    import torch
    from tests.helpers import RawView
    dev = torch.from_numpy(scenes.lidar(2_600_007, 62).view("int32")).cuda()
    sizes = ((200, 120), (333, 95))
    fbs, outs = [], []
    for i in range(6):
        w, h = sizes[i % 2]
        fbs.append(gpu.pcr_create_framebuffer(w, h, gpu.PCR_FB_HQ))
        outs.append(torch.zeros(w * h, dtype=torch.int32, device="cuda"))
    batch = gpu.pcr_batch_create(gpu.pcr_cloud_create(dev), fbs, outs, True, 1, 100, 0xFF010203, True)

    def views(seed, depth, scale, near_ground=False):
        vs = scenes.orbit_views(6, seed, resolutions=sizes)
        if near_ground:
            vs = [scenes.View.lookat((300 + 90 * i, 500, 60), (300 + 90 * i, 560, 20), (0, 0, 1), 60.0, *sizes[i % 2], 0.1, 120.0)
                  for i in range(6)]
        return [RawView(v.view_proj, v.near, v.far, v.width, v.height, depth, scale) for v in vs]

    first = True
    for vs in (views(3, 0, 1.0), views(4, 0, 1.0), views(5, 1, 1000.0), views(6, 1, 1e-26), views(7, 0, 1.0, True),
               views(8, 1, 1e8)):
        gpu.pcr_batch_set_views(batch, vs)
        if first:
            gpu.pcr_batch_capture(batch, torch.cuda.Stream())
            first = False
        for o in outs:
            o.zero_()
        gpu.pcr_batch_launch(batch, 0)
        torch.cuda.synchronize()
        for v, o in zip(vs, outs):
            one = gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ)
            want = torch.empty_like(o)
            gpu.pcr_render_hq_splat(one, dev, v, 1, 100)
            gpu.pcr_resolve(one, want, 0xFF010203, clear_after=True)
            assert torch.equal(o, want)
    batch.close()


@pytest.mark.parametrize("n", [2_499_999, 2_500_000])
def test_launches_follow_the_size_not_the_points_per_thread(gpu, n):
    """From 2.5M points on, a high-quality frame's pass 2 is one launch per view, with the default tuning, with the same
    tuning read and set again, and with two points per thread; the tuning read back is the one set."""
    import torch
    dev = torch.from_numpy(scenes.lidar(n, 63).view("int32")).cuda()
    views = scenes.orbit_views(6, 3, resolutions=((200, 120), (333, 95)))
    fbs = [gpu.pcr_create_framebuffer(v.width, v.height, gpu.PCR_FB_HQ) for v in views]
    outs = [torch.zeros(v.width * v.height, dtype=torch.int32, device="cuda") for v in views]
    batch = gpu.pcr_batch_create(gpu.pcr_cloud_create(dev), fbs, outs, True, 1, 100, 0, True)
    gpu.pcr_batch_set_views(batch, views)
    default = gpu.pcr_batch_get_tuning(batch)
    images = []
    for tuning in (None, default, {"route": 1}, {"route": 1, "points_per_thread": 2}):
        gpu.pcr_batch_set_tuning(batch, tuning)
        assert gpu.pcr_batch_get_tuning(batch) == {**default, **(tuning or {})}
        before = gpu.pcr_kernel_launch_count()
        gpu.pcr_batch_render(batch)
        # cull, tables, pass 1, pass 2, resolve
        assert gpu.pcr_kernel_launch_count() - before == 4 + (len(views) if n >= 2_500_000 else 1), tuning
        torch.cuda.synchronize()
        images.append([o.clone() for o in outs])
    for other in images[1:]:
        assert all(torch.equal(a, b) for a, b in zip(images[0], other))
    batch.close()


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 5 * 1024, 31 * 1024 + 7, 32 * 1024, 33 * 1024 + 1, 700_001])
@pytest.mark.parametrize("hq", [False, True])
@pytest.mark.parametrize("tuning", [None, {"route": 1, "points_per_thread": 2}, {"route": 1, "merge_width": 32}])
def test_items_of_other_tunings(gpu, n, hq, tuning):
    import torch
    dev = torch.from_numpy(scenes.lidar(n, 64).view("int32")).cuda()
    views = scenes.orbit_views(6, 3, resolutions=((200, 120), (333, 95)))
    flags = gpu.PCR_FB_HQ if hq else 0
    fbs = [gpu.pcr_create_framebuffer(v.width, v.height, flags) for v in views]
    outs = [torch.zeros(v.width * v.height, dtype=torch.int32, device="cuda") for v in views]
    batch = gpu.pcr_batch_create(gpu.pcr_cloud_create(dev), fbs, outs, hq, 1, 100, 0, False)
    gpu.pcr_batch_set_views(batch, views)
    if tuning:
        gpu.pcr_batch_set_tuning(batch, tuning)
    gpu.pcr_batch_render(batch)
    for v, fb in zip(views, fbs):
        one = gpu.pcr_create_framebuffer(v.width, v.height, flags)
        (gpu.pcr_render_hq_splat if hq else gpu.pcr_render_atomicmin)(one, dev, v)
        for a, b in zip(gpu.pcr_framebuffer_keys(fb), gpu.pcr_framebuffer_keys(one)):
            assert (a is None and b is None) or torch.equal(a, b)
    batch.close()
