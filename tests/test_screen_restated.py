"""CPU restatement of the screened passes' tests (csrc/pcr_screen.cuh: make_screen, screen_point) against the exact
integer decisions: the float depth estimate against a stored code, with stored codes at, next to and a margin's width
around each point's own code and the band edges it makes. A point the screen drops in pass 1 must have a larger code
than the stored one; a point it accepts or rejects in pass 2 must be in or outside the band."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import scenes
from tests.test_tier1_restated import F32, U, Tier1, f_up, fma32


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
