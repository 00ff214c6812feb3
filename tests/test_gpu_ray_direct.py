"""Small ray-table triangles, which setup rasterises straight into the z-buffer: bit-exact against
the oracle for rays on the layout and off it by up to a quarter pixel, triangles from a fraction
of a pixel to many pixels (direct, binned, near, across the seam, over the poles), partial tables,
odd sizes and one-row tables."""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import pytest

import cases
import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker is deselected on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1702_06813_gb300 as rm  # noqa: E402
from paper_1702_06813_gb300 import build as rmbuild  # noqa: E402

rmbuild.build()


@dataclasses.dataclass
class _Table(synth.Camera):
    """A spherical camera whose rays lie off the layout by up to `off` pixels on each axis."""
    off: float = 0.0

    def rays(self):
        r = cases.rng(self.width * 1000 + self.height)
        j, i = np.meshgrid(np.arange(self.height, dtype=float), np.arange(self.width, dtype=float), indexing="ij")
        i, j = i + r.uniform(-self.off, self.off, i.shape), j + r.uniform(-self.off, self.off, j.shape)
        az, el = self.az0 + self.az_step * (i + 0.5), self.el0 - self.el_step * j
        return np.stack([np.cos(el) * np.sin(az), -np.sin(el), np.cos(el) * np.cos(az)], axis=-1)


def _soup(r, n, px, band):
    """n triangles of about px radians around random directions of the elevation band."""
    az, el = r.uniform(-math.pi, math.pi, n), r.uniform(-band, band, n)
    d = np.stack([np.cos(el) * np.sin(az), -np.sin(el), np.cos(el) * np.cos(az)], 1)
    c = d * r.uniform(3.0, 40.0, (n, 1))
    size = np.linalg.norm(c, axis=1)[:, None, None] * px * np.exp(r.uniform(-1.0, 1.0, (n, 1, 1)))
    v = c[:, None, :] + r.normal(size=(n, 3, 3)) * size
    return v.reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


@pytest.mark.parametrize("w,h,span,az0,off", [(257, 33, 2 * math.pi, -math.pi, 0.0), (257, 33, 2 * math.pi, -math.pi, 0.24),
                                              (64, 16, 2 * math.pi, 0.3, 0.1), (61, 1, 1.4, -0.7, 0.0),
                                              (1, 40, 0.02, 0.1, 0.0), (300, 20, 2.0, -2.9, 0.05)])
@pytest.mark.parametrize("px", [0.1, 0.7, 4.0, 30.0])
def test_small_triangles_bit_exact(w, h, span, az0, off, px):
    cam = _Table("spherical", w, h, az0=az0, az_step=span / w, el0=0.35, el_step=0.7 / max(h - 1, 1), near=0.5,
                 range_min=0.5, range_max=80.0, off=off)
    r = cases.rng(int(1000 * px) + w)
    v, f = _soup(r, 6000 if px < 10 else 300, px * cam.az_step, 1.5 if px == 4.0 else 0.5)
    om = oracle.OracleMap(v, f, np.zeros(len(f), np.uint8))
    gm = rm.Map(v, f, np.zeros(len(f), np.uint8))
    intr = rm.Intrinsics.from_camera(cam)
    poses = [np.eye(4), synth.pose_from(np.array([0.4, -0.2, 0.1]), 0.5, 0.3, -0.2)]
    g = rm.render_depth(gm, np.stack(poses), intr)
    for k, P in enumerate(poses):
        o = om.render(P, cam)
        assert np.array_equal(g["tri_id"][k].cpu().numpy(), o["tri_id"]), (k, px)
        assert np.array_equal(g["depth"][k].cpu().numpy(), o["depth"], equal_nan=True), (k, px)
    gm.close()
