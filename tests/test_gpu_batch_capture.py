"""Frames of a batch recorded into graphs of the caller's (pcr_batch_render under a stream capture), beside the batch's
own captured frame, at sizes where pass 2 otherwise runs one launch per view."""
from __future__ import annotations

import pytest

import scenes

pytestmark = pytest.mark.gpu

N = 2_600_007
SIZES = ((200, 120), (333, 95))
BACKGROUND = 0xFF010203


class Setup:
    def __init__(self, gpu, hq=True, n=N, views=6):
        import torch
        self.gpu, self.hq = gpu, hq
        self.dev = torch.from_numpy(scenes.lidar(n, 71).view("int32")).cuda()
        self.fbs, self.outs = [], []
        for i in range(views):
            w, h = SIZES[i % 2]
            self.fbs.append(gpu.pcr_create_framebuffer(w, h, gpu.PCR_FB_HQ if hq else 0))
            self.outs.append(torch.zeros(w * h, dtype=torch.int32, device="cuda"))
        self.batch = gpu.pcr_batch_create(gpu.pcr_cloud_create(self.dev), self.fbs, self.outs, hq, 1, 100, BACKGROUND, True)

    def views(self, seed):
        return scenes.orbit_views(len(self.fbs), seed, resolutions=SIZES)

    def want(self, views):
        """The images of the single-view entry points."""
        import torch
        images = []
        for v, o in zip(views, self.outs):
            fb = self.gpu.pcr_create_framebuffer(v.width, v.height, self.gpu.PCR_FB_HQ if self.hq else 0)
            image = torch.empty_like(o)
            (self.gpu.pcr_render_hq_splat if self.hq else self.gpu.pcr_render_atomicmin)(fb, self.dev, v)
            self.gpu.pcr_resolve(fb, image, BACKGROUND, clear_after=True)
            images.append(image)
            fb.close()
        return images

    def check(self, views):
        import torch
        torch.cuda.synchronize()
        for k, (a, b) in enumerate(zip(self.outs, self.want(views))):
            assert torch.equal(a, b), (k, int((a != b).sum()))
        for o in self.outs:
            o.zero_()
        torch.cuda.synchronize()

    def capture(self):
        """One frame in a graph of the caller's."""
        import torch
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            self.gpu.pcr_batch_render(self.batch)
        return graph


@pytest.mark.parametrize("hq", [True, False])
def test_replays_follow_the_views(gpu, hq):
    import torch
    s = Setup(gpu, hq)
    gpu.pcr_batch_set_views(s.batch, s.views(3))
    graph = s.capture()
    for seed in (3, 4, 5):
        gpu.pcr_batch_set_views(s.batch, s.views(seed))
        graph.replay()
        s.check(s.views(seed))
    torch.cuda.synchronize()
    del graph
    s.batch.close()


def test_beside_the_batch_s_own_frame(gpu):
    """The batch's own captured frame stays its own: a capture by the caller neither replaces its nodes nor, once that
    graph is gone, leaves it any of them; un-captured frames in between."""
    import torch
    s = Setup(gpu)
    gpu.pcr_batch_set_views(s.batch, s.views(3))
    own = torch.cuda.Stream()
    gpu.pcr_batch_capture(s.batch, own)
    graph = s.capture()
    for seed in (4, 5):
        gpu.pcr_batch_set_views(s.batch, s.views(seed))
        gpu.pcr_batch_launch(s.batch, own)
        s.check(s.views(seed))
        graph.replay()
        s.check(s.views(seed))
        gpu.pcr_batch_render(s.batch)
        s.check(s.views(seed))
    torch.cuda.synchronize()
    del graph
    gpu.pcr_batch_set_views(s.batch, s.views(6))
    gpu.pcr_batch_launch(s.batch, own)
    s.check(s.views(6))
    s.batch.close()


@pytest.mark.parametrize("bad", [0, 1, 5])
def test_refused_views_leave_the_staged_frame(gpu, bad):
    """A set of views of which one is refused (near beyond far) changes nothing: un-captured frames and the batch's
    own captured frame stay those of the views before, also where the screened pass 2 cannot take those (depth codes in
    units of 1e26 m)."""
    import torch
    from tests.helpers import RawView
    s = Setup(gpu)
    own = torch.cuda.Stream()
    for k, scale in enumerate((None, 1e-26)):
        good = s.views(3 + k)
        if scale:
            good = [RawView(v.view_proj, v.near, v.far, v.width, v.height, 1, scale) for v in good]
        gpu.pcr_batch_set_views(s.batch, good)
        if not k:
            gpu.pcr_batch_capture(s.batch, own)
        refused = s.views(9)
        refused[bad] = RawView(refused[bad].view_proj, 10.0, 1.0, refused[bad].width, refused[bad].height)
        for _ in range(2):
            with pytest.raises(gpu.PcrError):
                gpu.pcr_batch_set_views(s.batch, refused)
            gpu.pcr_batch_render(s.batch)
            s.check(good)
            gpu.pcr_batch_launch(s.batch, own)
            s.check(good)
    s.batch.close()


@pytest.mark.parametrize("own", [False, True])
def test_views_wait_for_a_replay_s_copy(gpu, own):
    """pcr_batch_set_views waits until a replay that is still queued (behind 50 ms of other work) has copied its views,
    also where the graph is the caller's."""
    import torch
    s = Setup(gpu, False, 300_001)
    gpu.pcr_batch_set_views(s.batch, s.views(3))
    stream = torch.cuda.Stream()
    if own:
        gpu.pcr_batch_capture(s.batch, stream)
    else:
        graph = s.capture()
    for seed in range(3, 7):
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)
            if own:
                gpu.pcr_batch_launch(s.batch, stream)
            else:
                graph.replay()
        gpu.pcr_batch_set_views(s.batch, s.views(seed + 1))
        s.check(s.views(seed))
    s.batch.close()
