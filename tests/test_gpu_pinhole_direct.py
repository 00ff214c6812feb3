"""Small pinhole triangles, which setup rasterises straight into the z-buffer: bit-exact against the
oracle from sub-pixel slivers to triangles of many pixels (around the line between direct and
binned), across image borders, the near plane and screen tiles, at odd sizes and with exact ties;
and the z-buffer is left empty for the next call, whatever its size."""
from __future__ import annotations

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


def _soup(seed, n, px, f):
    """n camera-space triangles of about px pixels, some of them copies of another one."""
    r = cases.rng(seed)
    z = r.uniform(0.3, 6.0, n)
    c = np.stack([r.uniform(-0.8, 0.8, n) * z, r.uniform(-0.8, 0.8, n) * z, z], 1)
    size = (z * px / f)[:, None, None] * np.exp(r.uniform(-0.7, 0.7, (n, 1, 1)))
    v = c[:, None, :] + r.normal(size=(n, 3, 3)) * size * np.array([1.0, 1.0, 0.5])
    v[: n // 10] = v[n // 2 : n // 2 + n // 10]
    order = r.permutation(n)
    return v[order].reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


def _check(gm, om, cam, poses, what):
    g = rm.render_depth(gm, np.stack(poses), rm.Intrinsics.from_camera(cam))
    for k, P in enumerate(poses):
        o = om.render(P, cam)
        assert np.array_equal(g["tri_id"][k].cpu().numpy(), o["tri_id"]), (what, k)
        assert np.array_equal(g["depth"][k].cpu().numpy(), o["depth"], equal_nan=True), (what, k)


@pytest.mark.parametrize("px", [0.3, 1.0, 3.0, 6.0, 12.0, 40.0])
@pytest.mark.parametrize("w,h", [(131, 67), (64, 32), (1, 1), (333, 5)])
def test_small_triangles_bit_exact(w, h, px):
    cam = cases.small_pinhole(w=w, h=h, f=100.0, near=0.5)
    v, f = _soup(int(10 * px) + w, 5000, px, 100.0)
    lab = np.zeros(len(f), np.uint8)
    gm, om = rm.Map(v, f, lab), oracle.OracleMap(v, f, lab)
    poses = [np.eye(4), synth.pose_from(np.array([0.1, 0.0, 0.0]), 1.5, 0.1, 0.2)]
    _check(gm, om, cam, poses, (w, h, px))
    gm.close()


def test_calls_of_different_sizes_share_the_zbuffer():
    v, f = _soup(7, 8000, 3.0, 100.0)
    lab = np.zeros(len(f), np.uint8)
    gm, om = rm.Map(v, f, lab), oracle.OracleMap(v, f, lab)
    eye = np.eye(4)
    for w, h, n, wave, tile in ((160, 120, 1, 0, (0, 0)), (97, 41, 5, 2, (16, 16)), (200, 150, 3, 1, (32, 32)),
                                (33, 90, 4, 3, (32, 16)), (160, 120, 2, 0, (64, 32))):
        gm.set_tuning(tile=tile, wave_poses=wave)
        cam = cases.small_pinhole(w=w, h=h, f=100.0, near=0.5)
        poses = [eye] + [synth.perturb_fixed(eye, cases.rng(k), 0.05, 2.0) for k in range(1, n)]
        _check(gm, om, cam, poses, (w, h, n))
    gm.close()
