"""Meshification at the edges of its kernels: single rows and columns (no blocks), one CTA and a few,
and an image large enough for the separate scan of the counts; bit-exact against the oracle."""
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


@pytest.mark.parametrize("w,h,step", [(1, 5, 1), (5, 1, 1), (2, 2, 1), (16, 16, 1), (257, 2, 1), (130, 70, 3), (820, 660, 1)])
def test_meshify_sizes_bit_exact(w, h, step):
    r = cases.rng(w + h)
    y, x = np.mgrid[0:h, 0:w]
    d = (2.0 + 0.4 * np.sin(0.05 * x) + 0.3 * np.cos(0.04 * y) + r.normal(scale=0.002, size=(h, w))).astype(np.float32)
    c = (r.uniform(size=d.shape) < 0.04).astype(np.uint8) * r.integers(1, 3, d.shape).astype(np.uint8)
    cam = cases.small_pinhole(w=w, h=h, f=120.0)
    pose = synth.pose_from(np.array([0.3, -0.2, 0.1]), 0.4, 0.1, -0.2)
    g = rm.meshify(rm.Scan.make(rm.Intrinsics.from_camera(cam), d, c), pose, max_range=4.0, max_edge=0.1, step=step)
    v, f, lab = oracle.meshify(cam, d, c, pose, 4.0, 0.1, step)
    assert np.array_equal(g["vertices"].cpu().numpy().view(np.uint32), v.view(np.uint32))
    assert np.array_equal(g["faces"].cpu().numpy(), f)
    assert np.array_equal(g["labels"].cpu().numpy(), lab)
