"""Batches of more problems than a grid has rows (65,535): plain evaluations of either camera model
equal the per-pose calls, and LM steps those of the batch's halves, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import cases
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker is deselected on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1702_06813_gb300 as rm  # noqa: E402
from paper_1702_06813_gb300 import build as rmbuild  # noqa: E402

rmbuild.build()

N = 70_000


@pytest.fixture(scope="module")
def scene():
    v, f = cases.plane_grid(4, 4, (-2.0, -2.0, 2.0), (4, 0, 0.5), (0, 4, 0.3))
    gm = rm.Map(v, f, np.zeros(len(f), np.uint8))
    r = cases.rng(71)
    poses = np.stack([synth.perturb_fixed(np.eye(4), r, 0.05, 2.0) for _ in range(16)])[np.arange(N) % 16]
    yield gm, poses
    gm.close()


def _scans(cam):
    intr = rm.Intrinsics.from_camera(cam)
    shape = (cam.height, cam.width)
    return [rm.Scan.make(intr, np.full(shape, d, np.float32), np.zeros(shape, np.uint8)) for d in (2.05, 2.2)]


@pytest.mark.parametrize("model", ["pinhole", "spherical"])
def test_plain_batch_equals_calls(scene, model):
    gm, poses = scene
    scans = _scans(cases.small_pinhole(8, 8, 8.0) if model == "pinhole" else cases.small_spherical(16, 8))
    got = rm.cost_grad_batch(gm, scans=[scans[k % 2] for k in range(N)], poses=poses)
    for k in range(2):
        want = rm.cost_grad(gm, scans[k], poses[k::2])
        assert int(want["counts"].sum()) > 0
        for key in want:
            assert torch.equal(got[key][k::2], want[key]), (k, key)


def test_align_batch_equals_its_halves(scene):
    gm, poses = scene
    scans = _scans(cases.small_pinhole(8, 8, 8.0))
    all_scans = [scans[k % 2] for k in range(N)]
    got, reps, _ = rm.align_batch(gm, scans=all_scans, poses=poses, max_iters=2)
    for part in (slice(0, N // 2), slice(N // 2, N)):
        want, wreps, _ = rm.align_batch(gm, scans=all_scans[part], poses=poses[part], max_iters=2)
        assert np.array_equal(got[part], want)
        assert reps[part] == wreps
