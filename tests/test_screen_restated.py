"""CPU restatement of the screened passes' tests (csrc/pcr_screen.cuh: make_screen, screen_two) against the exact
integer decisions: the float depth estimate against a stored code, with stored codes at, next to and a margin's width
around each point's own code and the band edges it makes. A point the screen drops in pass 1 must have a larger code
than the stored one (PIECEWISE: whichever range the stored code lies in); a point it accepts or rejects in pass 2 must be
in or outside the band; a point that pass 1's words leave out must be outside the band of every code that the stored one
can become. Also the sample that picks the passes' loop (sample_cloud), restated for the GPU tests."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import scenes
from tests.test_tier1_restated import F32, MAGIC, U, Tier1, add_rd, add_ru, f_down, f_up, fma32


class Screen:
    def __init__(self, t, view, eps=(0, 1)):
        far, near = float(view.far), float(view.near)
        self.S = 2.0 ** 40 / (far - near) if t.linear else float(view.metric_scale)
        off = near if t.linear else 0.0
        self.nq = int(np.floor(near * self.S)) if t.linear else 0
        self.unit1 = not t.linear and far * self.S < 4294967040.0
        unit = 1.0 if self.unit1 else 256.0
        e = eps[0] / eps[1]
        c = (unit * (1.0 + e) + 2.0) / self.S
        up = 1.0 + 2.0 ** -18
        self.k, self.k3 = f_up(7.2 * U * float(t.Mw) * up), f_up((7.2 * U * float(t.Mw3) + c) * up)
        self.a, self.b = F32(unit / self.S), F32(off + unit / self.S)
        self.lo = (self.a, F32(off))
        self.hi = (F32(unit * (1.0 + e) / self.S), F32(off + e * self.nq / self.S))

    def stored(self, qs):
        sh = np.minimum(qs, 2 ** 32 - 1) if self.unit1 else qs >> 8
        return sh.astype(np.float32)  # both round to nearest


def _view(depth, scale):
    base = scenes.lidar_1km_view(640, 360)
    v = scenes.View(base.view_proj, base.near, base.far, 640, 360)
    v.depth_mode, v.metric_scale = depth, scale
    return v


@pytest.mark.parametrize("depth,scale", [(0, 0.0), (1, 1000.0), (1, 1e6), (1, 1e8)])
@pytest.mark.parametrize("eps", [(1, 100), (0, 1), (7, 2), (1, 1 << 20)])
def test_decisions(depth, scale, eps):
    view = _view(depth, scale)
    pts = scenes.lidar(20_000, 31)
    pix, _, key = oracle.project(pts, view)
    pts, q = pts[pix >= 0], (key[pix >= 0] >> np.uint64(24)).astype(np.int64)
    t = Tier1(view)
    xyz = np.ascontiguousarray(pts[:, :3]).view(np.float32)
    x, y, z = xyz.T
    s = (np.abs(x) + np.abs(y)) + np.abs(z)
    w = fma32(t.Wr[2], z, fma32(t.Wr[1], y, fma32(t.Wr[0], x, t.Wr[3])))
    sc, sb = Screen(t, view), Screen(t, view, eps)
    m1, m2 = fma32(sc.k, s, sc.k3), fma32(sb.k, s, sb.k3)
    num, den = eps
    margin = np.maximum(1, (m1.astype(np.float64) * sc.S).astype(np.int64))
    edge = ((q.astype(object) * den - num * sb.nq) // (den + num)).astype(np.int64)  # qmin whose upper edge is near q
    sizes = {}
    for centre in (q, edge):
        for d in (0, 1, -1, 255, -256, 300, -300, *(f * margin for f in (-3.0, -1.2, -0.9, -0.3, 0.3, 0.9, 1.2, 3.0))):
            qs = np.clip(centre + np.asarray(d, np.float64).astype(np.int64), 0, 2 ** 40 - 2)
            # pass 1
            skip = (w - fma32(sc.stored(qs), sc.a, sc.b)).astype(np.float32) >= m1
            assert not (skip & (q <= qs)).any()
            # pass 2
            k = sb.stored(qs)
            dist = np.minimum((w - fma32(k, *sb.lo)).astype(np.float32), (fma32(k, *sb.hi) - w).astype(np.float32))
            band = (q >= qs) & ((q - qs).astype(object) * den <= num * (qs.astype(object) + sb.nq))
            assert not ((dist >= m2) & ~band).any()
            assert not ((dist <= -m2) & band).any()
            for name, n in (("skip", skip), ("in", dist >= m2), ("out", dist <= -m2)):
                sizes[name] = sizes.get(name, 0) + int(n.sum())
    assert sizes["skip"] > 0 and sizes["out"] > 0 and (num == 0 or eps[1] > 1000 or sizes["in"] > 0), sizes


@pytest.mark.parametrize("depth,scale", [(0, 0.0), (1, 1000.0), (1, 1e8)])
@pytest.mark.parametrize("eps", [(1, 100), (0, 1), (1, 1), (1, 1 << 20)])
def test_words(depth, scale, eps):
    """Pass 1 clears a point's bit by the key it reads; the pixel's final key is that one or smaller."""
    view = _view(depth, scale)
    pts = scenes.lidar(20_000, 32)
    pix, _, key = oracle.project(pts, view)
    pts, q = pts[pix >= 0], (key[pix >= 0] >> np.uint64(24)).astype(np.int64)
    t = Tier1(view)
    x, y, z = np.ascontiguousarray(pts[:, :3]).view(np.float32).T
    s = (np.abs(x) + np.abs(y)) + np.abs(z)
    w = fma32(t.Wr[2], z, fma32(t.Wr[1], y, fma32(t.Wr[0], x, t.Wr[3])))
    sb = Screen(t, view, eps)
    m = fma32(sb.k, s, sb.k3)
    num, den = eps
    margin = np.maximum(1, (m.astype(np.float64) * sb.S).astype(np.int64))
    edge = ((q.astype(object) * den - num * sb.nq) // (den + num)).astype(np.int64)  # qmin whose upper edge is near q
    rng, left_out = np.random.default_rng(3), 0
    for d in (0, 1, -1, 255, -256, *(f * margin for f in (-3.0, -1.2, -0.9, 0.9, 1.2, 3.0))):
        qs = np.clip(edge + np.asarray(d, np.float64).astype(np.int64), 0, 2 ** 40 - 2)
        clear = ~((fma32(sb.stored(qs), *sb.hi) - w).astype(np.float32) > -m)
        left_out += int(clear.sum())
        for smaller in (0, 1, 255, rng.integers(0, 1 << 20, len(qs)), qs):
            final = np.maximum(qs - smaller, 0)
            band = (q - final).astype(object) * den <= num * (final.astype(object) + sb.nq)
            assert not (clear & band).any()
    assert left_out > 0


class PiecewiseScreen:
    """make_screen and the windows and range starts of a PIECEWISE view (piecewise_range), restated."""

    def __init__(self, t, view):
        near, far = float(view.near), float(view.far)
        up = 1.0 + 2.0 ** -18
        self.t, self.k = t, f_up(7.2 * U * float(t.Mw) * up)
        self.a, self.b, self.k3, self.wc, self.whk, self.start, self.first, self.last = ([] for _ in range(8))
        base = 0.0
        for lo, hi, res in np.asarray(view.ranges, float):
            lo_e, hi_e = max(lo, near), min(hi, far)
            if hi_e > lo_e:
                b = lo + (256.0 - base) / res
                self.a.append(F32(256.0 / res))
                self.b.append(F32(b))
                self.k3.append(f_up((7.2 * U * float(t.Mw3) + 258.0 / res + (-4.2 * U * b if b < 0.0 else 0.0)) * up))
                nin = max(lo_e * (1.0 + 4.0 * U), (lo + 2.5 / res) * (1.0 + 4.0 * U))
                fin = min(hi_e * (1.0 - 4.0 * U), (lo + (2.0 ** 40 - 2.0 ** 25) / res) * (1.0 - 4.0 * U))
                wc = F32(0.5 * (nin + fin))
                whk = (min(float(wc) - nin, fin - float(wc)) - float(t.kw3)) / (1.0 + 2.0001 * U)
                self.wc.append(wc)
                self.whk.append(f_down(whk) if whk > 0 else F32(0.0))
                self.start.append(f_down(nin))
                self.first.append(int(base))
                self.last.append(int(base + np.ceil((hi - lo) * res)) - 1)
            base += np.ceil((hi - lo) * res)


@pytest.mark.parametrize("ranges", [
    [[0.0, 5000.0, 2e8]],                                                              # one range
    [[0.0, 10.0, 1e9], [10.0, 10010.0, 1e6]],                                          # nm, um: the second's offset is negative
    [[0.0, 700.0, 1e9], [700.0, 5000.0, 1e3]],                                         # and far below 0 (-7 * 10^8)
    [[0.0, 300.0, 1e9], [300.0, 600.0, 1e6], [600.0, 5000.0, 1e3]],
    [[0.0, 200.0, 1e8], [200.0, 400.0, 1e3], [450.0, 800.0, 1e7], [800.0, 801.0, 1e9], [801.0, 5000.0, 1e4]],
])
def test_piecewise_decisions(ranges):
    view = _view(2, 1.0)
    view.ranges = np.asarray(ranges)
    pts = scenes.lidar(30_000, 33)
    pix, _, key = oracle.project(pts, view)
    pts, q = pts[pix >= 0], (key[pix >= 0] >> np.uint64(24)).astype(np.int64)
    t = Tier1(view)
    p = PiecewiseScreen(t, view)
    x, y, z = np.ascontiguousarray(pts[:, :3]).view(np.float32).T
    s = (np.abs(x) + np.abs(y)) + np.abs(z)
    w = fma32(t.Wr[2], z, fma32(t.Wr[1], y, fma32(t.Wr[0], x, t.Wr[3])))
    r = sum((w >= start).astype(int) for start in p.start[1:]) + np.zeros(len(w), int)
    pick = lambda f: np.asarray(f, np.float32)[r]  # noqa: E731
    certain = np.abs(w - pick(p.wc)) < fma32(-t.kw, s, pick(p.whk))
    assert certain.mean() > 0.9
    # a certified point's range is the one its code lies in
    assert (q[certain] >= np.asarray(p.first)[r][certain]).all() and (q[certain] <= np.asarray(p.last)[r][certain]).all()
    m, a, b = fma32(p.k, s, pick(p.k3)), pick(p.a), pick(p.b)
    res = np.asarray([256.0 / float(v) for v in p.a])[r]
    margin = np.maximum(1, (m.astype(np.float64) * res)).astype(np.int64)
    stored = [q + d for d in (0, 1, -1, 255, -255, 256, -256, 300, -300)]
    stored += [q + (f * margin).astype(np.int64) for f in (-3.0, -1.2, -0.9, -0.3, 0.3, 0.9, 1.2, 3.0)]
    for code in (*p.first, *p.last):  # next to every range's ends, whatever the point's own range
        stored += [np.full(len(q), code + d) for d in (-300, -256, -1, 0, 1, 255, 300)]
        stored += [code + (f * margin).astype(np.int64) for f in (-1.2, -0.5, 0.5, 1.2)]
    stored += [np.zeros(len(q), np.int64), np.full(len(q), 2 ** 40 - 1)]  # the nearest code; the empty key
    dropped = np.zeros(len(p.a), int)
    for qs in stored:
        qs = np.clip(qs, 0, 2 ** 40 - 1)
        skip = certain & ((w - fma32((qs >> 8).astype(np.float32), a, b)).astype(np.float32) >= m)
        assert not (skip & (q <= qs)).any()
        dropped += np.bincount(r[skip], minlength=len(p.a))
    assert all(d > 0 for d, k in zip(dropped, range(len(p.a))) if (certain & (r == k)).any()), dropped


SAMPLE_TILES = 96


def sample_decisions(pts, view, blocks, warps):
    """Per block of a screened pass of that shape over (n, 4) uint32 points: whether it finds the cloud mostly outside the
    clip planes and in random order (sample_cloud); None where the cloud is too small to be sampled."""
    G = blocks * warps
    spread = len(pts) // 64 // G
    if spread < SAMPLE_TILES:
        return None
    t = Tier1(view)
    outside, seen, same = (np.zeros(blocks, int) for _ in range(3))
    tile = (np.arange(warps)[None, :] * blocks + np.arange(blocks)[:, None]) * spread
    for h in range(2):
        at = tile[:, :, None] * 64 + 32 * h + np.arange(32)
        x, y, z = np.moveaxis(np.ascontiguousarray(pts[at, :3]).view(np.float32), -1, 0)
        s = (np.abs(x) + np.abs(y)) + np.abs(z)
        w = fma32(t.Wr[2], z, fma32(t.Wr[1], y, fma32(t.Wr[0], x, t.Wr[3])))
        dw = fma32(t.kw, s, t.kw3)
        outside += ((s < t.xyz_max) & ((add_ru(w, dw) < t.near_o) | (add_rd(w, -dw) >= t.far_o))).sum((1, 2))
        with np.errstate(all="ignore"):
            rcp = (F32(1.0) / w).astype(np.float32)
            hE = fma32(-fma32(t.ke, s, t.ke3), rcp, t.he0)
            k, ok = [], w > 0
            for g, size in ((t.Gx, t.W), (t.Gy, t.H)):
                f = (fma32(g[2], z, fma32(g[1], y, fma32(g[0], x, g[3]))) * rcp).astype(np.float32)
                up = (f + MAGIC).astype(np.float32)
                k.append((up.view(np.int32).astype(np.int64) - 0x4B400000) & 0xFFFFFFFF)
                ok &= (k[-1] < size) & (np.abs((f - (up - MAGIC)).astype(np.float32)) < hE)
        pixel = np.where(ok, k[1] * t.W + k[0], -1 - np.arange(32))
        seen += ok.sum((1, 2))
        same += (pixel[:, :, 1:] == pixel[:, :, :-1]).sum((1, 2))
    return 2 * outside >= 32 * warps, 64 * same < seen
