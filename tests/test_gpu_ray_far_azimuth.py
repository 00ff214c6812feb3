"""Full-turn ray tables whose layout starts any number of turns from zero: a tiny triangle around every
ray (a two-hundredth of a pixel) is found, bit for bit as by the oracle."""
from __future__ import annotations

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


@pytest.mark.parametrize("w,az0", [(64, 0.3), (64, 31.9), (64, 32.1), (256, 14004.976), (360, -6516.64),
                                    (360, 30207.287), (512, 7018.3208), (512, 15797.318), (1024, 7869.81)])
def test_tiny_triangles_around_every_ray(w, az0):
    h = 8
    cam = synth.Camera("spherical", w, h, az0=float(np.float32(az0)), az_step=2 * math.pi / w, el0=0.2, el_step=0.05,
                       near=0.5, range_min=0.5, range_max=80.0)
    d = cam.ray_table_f32().reshape(-1, 3).astype(np.float64)
    r = cases.rng(w)
    side = np.cross(d, [0.0, 1.0, 0.0])
    side /= np.linalg.norm(side, axis=1, keepdims=True)
    up = np.cross(side, d)
    size = 0.005 * min(cam.az_step, cam.el_step)
    ang = r.uniform(0, 2 * math.pi, (len(d), 1)) + 2 * math.pi / 3 * np.arange(3)
    v = 10.0 * (d[:, None] + size * (np.cos(ang)[..., None] * side[:, None] + np.sin(ang)[..., None] * up[:, None]))
    v, f = v.reshape(-1, 3).astype(np.float32), np.arange(3 * len(d), dtype=np.int32).reshape(-1, 3)
    lab = np.zeros(len(f), np.uint8)
    gm, om = rm.Map(v, f, lab), oracle.OracleMap(v, f, lab)
    g = rm.render_depth(gm, np.eye(4)[None], rm.Intrinsics.from_camera(cam))
    o = om.render(np.eye(4), cam)
    assert (o["tri_id"] >= 0).mean() > 0.5  # FP32 leaves some of the finest table's triangles empty
    assert np.array_equal(g["tri_id"][0].cpu().numpy(), o["tri_id"])
    assert np.array_equal(g["depth"][0].cpu().numpy(), o["depth"], equal_nan=True)
    gm.close()
