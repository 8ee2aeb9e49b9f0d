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
