"""The batch resolve (k_resolve_batch) against the single-view resolves, on views of mixed and odd sizes (one pixel, one
row, the edges of a block's step), basic and high-quality, with and without the clear."""
from __future__ import annotations

import pytest

import scenes

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (3, 5), (1023, 1), (1024, 1), (1025, 1), (1, 2049), (127, 33), (640, 480), (1013, 771), (2560, 1440)]


@pytest.mark.parametrize("hq", [False, True])
@pytest.mark.parametrize("clear", [False, True])
def test_mixed_sizes(gpu, hq, clear):
    import torch
    dev = torch.from_numpy(scenes.lidar(300_001, 51).view("int32")).cuda()
    views = [scenes.lidar_1km_view(w, h) for w, h in SIZES]
    flags = gpu.PCR_FB_HQ if hq else 0
    fbs = [gpu.pcr_create_framebuffer(v.width, v.height, flags) for v in views]
    # images that start 4 bytes past an aligned address
    outs = [torch.zeros(v.width * v.height + 1, dtype=torch.int32, device="cuda")[1:] for v in views]
    batch = gpu.pcr_batch_create(gpu.pcr_cloud_create(dev), fbs, outs, hq, 1, 100, 0xFF102030, clear)
    gpu.pcr_batch_set_views(batch, views)
    gpu.pcr_batch_render(batch)
    for v, fb, out in zip(views, fbs, outs):
        one = gpu.pcr_create_framebuffer(v.width, v.height, flags)
        want = torch.empty_like(out)
        (gpu.pcr_render_hq_splat if hq else gpu.pcr_render_atomicmin)(one, dev, v)
        gpu.pcr_resolve(one, want, 0xFF102030, clear_after=clear)
        assert torch.equal(out, want), (v.width, v.height)
        for a, b in zip(gpu.pcr_framebuffer_keys(fb), gpu.pcr_framebuffer_keys(one)):
            assert (a is None and b is None) or torch.equal(a, b)
        assert gpu.pcr_get_device_status(fb) == gpu.PCR_OK
    batch.close()
