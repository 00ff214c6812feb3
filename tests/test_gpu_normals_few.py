"""Eq. 2 normals, and smoothed depth of few images (tiles) and of many (strips): an image gives the
same bits alone as in a batch on the other side of the line between the two, at the edges of tiles
(64x16) and strips (62 columns), with holes and without; and the batch matches the oracle within the
tolerances of test_gpu_normals.py."""
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

LINE = 1 << 21  # pixels in all from which the strips take over


def _bits(t):
    return t.contiguous().view(torch.int32)


@pytest.mark.parametrize("w,h", [(63, 15), (64, 16), (65, 17), (62, 33), (125, 97), (640, 480), (1, 64)])
@pytest.mark.parametrize("sigma", [0.4, 1.5, 2.6, 5.0])
@pytest.mark.parametrize("holes", [False, True])
def test_alone_as_in_a_batch(w, h, sigma, holes):
    r = cases.rng(w * 1000 + h)
    y, x = np.mgrid[0:h, 0:w]
    k = np.arange(3)[:, None, None]
    d = (2.0 + 0.3 * np.sin(0.11 * x + k) + 0.2 * np.cos(0.07 * y) + r.normal(scale=0.005, size=(3, h, w))).astype(np.float32)
    c = np.zeros(d.shape, np.uint8)
    if holes:
        c[r.uniform(size=d.shape) < 0.05] = 1
        d[r.uniform(size=d.shape) < 0.02] = np.nan
    cam = cases.small_pinhole(w=w, h=h, f=100.0)
    intr = rm.Intrinsics.from_camera(cam)
    n = -(-LINE // (w * h))
    d3, c3 = torch.as_tensor(d).cuda(), torch.as_tensor(c).cuda()
    rep = torch.arange(n, device="cuda") % 3
    many = rm.depth_normals(intr, d3[rep], c3[rep], sigma=sigma, metric=True, want_smoothed=True)
    for i in range(3):
        one = rm.depth_normals(intr, d3[i], c3[i], sigma=sigma, metric=True, want_smoothed=True)
        for got, want in zip(one, many):
            assert torch.equal(torch.isnan(got), torch.isnan(want[i]))
            ok = ~torch.isnan(got)
            assert torch.equal(_bits(got[ok]), _bits(want[i][ok])), i
    on, os_ = oracle.depth_normals(d[1], c[1], sigma=sigma, metric=True, fx=cam.fx, fy=cam.fy)
    gn, gs = many[0][1].cpu().numpy(), many[1][1].cpu().numpy()
    ok = ~np.isnan(os_)
    assert np.array_equal(ok, ~np.isnan(gs))
    assert np.all(np.abs(gs[ok] - os_[ok]) <= 1e-5 * np.abs(os_[ok]))
    assert np.array_equal(np.isnan(gn), np.isnan(on))
    okn = ~np.isnan(on[..., 0])
    assert np.max(np.abs(gn[okn] - on[okn]), initial=0.0) <= 5e-4
