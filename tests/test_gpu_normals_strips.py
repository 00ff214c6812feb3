"""Eq. 2 normals at the edges of the strips, chunks and radii of their kernel (62 output columns to a
strip, four rows to a step, radius 0 to 15), one image and many, against the oracle: masks exact,
smoothed depth 1e-5 relative, normals 5e-4 (the tolerances of test_gpu_normals.py)."""
from __future__ import annotations

import numpy as np
import pytest

import cases
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker is deselected on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1702_06813_gb300 as rm  # noqa: E402
from paper_1702_06813_gb300 import build as rmbuild  # noqa: E402

rmbuild.build()


@pytest.mark.parametrize("w,h,n", [(1, 3, 1), (3, 1, 2), (61, 7, 1), (62, 33, 3), (63, 34, 1), (64, 35, 2),
                                   (124, 36, 1), (125, 97, 40)])
@pytest.mark.parametrize("sigma", [0.0, 0.4, 1.5, 5.0])
def test_strips_against_oracle(w, h, n, sigma):
    r = cases.rng(w * 100 + h)
    y, x = np.mgrid[0:h, 0:w]
    d = np.stack([2.0 + 0.3 * np.sin(0.11 * x + k) + 0.2 * np.cos(0.07 * y) + r.normal(scale=0.005, size=(h, w))
                  for k in range(n)]).astype(np.float32)
    c = (r.uniform(size=d.shape) < 0.05).astype(np.uint8) * r.integers(1, 3, d.shape).astype(np.uint8)
    d[(r.uniform(size=d.shape) < 0.02)] = np.inf
    cam = cases.small_pinhole(w=w, h=h, f=100.0)
    gn, gs = rm.depth_normals(rm.Intrinsics.from_camera(cam), d, c, sigma=sigma, metric=True, want_smoothed=True)
    gn, gs = gn.cpu().numpy(), gs.cpu().numpy()
    for k in {0, n - 1}:
        on, os_ = oracle.depth_normals(d[k], c[k], sigma=sigma, metric=True, fx=cam.fx, fy=cam.fy)
        ok = ~np.isnan(os_)
        assert np.array_equal(ok, ~np.isnan(gs[k]))
        assert np.all(np.abs(gs[k][ok] - os_[ok]) <= 1e-5 * np.abs(os_[ok]))
        assert np.array_equal(np.isnan(gn[k]), np.isnan(on))
        okn = ~np.isnan(on[..., 0])
        assert np.max(np.abs(gn[k][okn] - on[okn]), initial=0.0) <= 5e-4
