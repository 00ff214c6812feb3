"""The batched phases on problems that would fit one per-pose call. A plain batch of one scan runs as
the poses of rm_cost_grad; here the scan has two equal copies, so that the problems go through the
batch's own kernels and captured graph: many poses, repeated calls of one shape, per-pose calls and
larger calls in between (which reuse and reallocate the scratch), and bins that grow. Everything
equals the per-pose results bit for bit."""
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


def _copies(intr, scan):
    return [rm.Scan.make(intr, *scan) for _ in range(2)]


def _same(got, want):
    for key in want:
        assert torch.equal(got[key], want[key]), key


def _poses(gt, seed, n):
    r = cases.rng(seed)
    return np.stack([synth.perturb_fixed(gt, r, 0.1, 3.0) for _ in range(n)])


def _alternate(scans, n):
    return [scans[k % 2] for k in range(n)]


@pytest.mark.parametrize("cam,n", [(synth.cam_320x240(), 256), (synth.cam_kinect_640x480(), 65),
                                   (synth.cam_lidar_1024x64(), 40)])
def test_many_poses_equal_waves(cam, n):
    mesh = synth.room_mesh(2000, size=(10.0, 8.0, 3.0), n_boxes=120, n_slabs=12, target_fo=240_000,
                           target_fu=60_000, n_panels=250)
    r = cases.rng(2001)
    gt = synth.room_pose(r, mesh)
    scans = _copies(rm.Intrinsics.from_camera(cam), synth.synth_scan(mesh, cam, gt, r, sigma_rel=0.005))
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    poses = _poses(gt, 2002, n)
    got = rm.cost_grad_batch(gm, scans=_alternate(scans, n), poses=torch.as_tensor(poses))
    want = rm.cost_grad(gm, scans[0], poses)
    assert int(want["counts"].sum()) > 0
    _same(got, want)
    gm.close()


def test_repeated_calls_growth_and_reallocation():
    c = cases.config1(seed=1000)
    gm = rm.Map(c["mesh"].vertices, c["mesh"].faces, c["mesh"].labels)
    sph = cases.small_spherical()
    pin = _copies(rm.Intrinsics.from_camera(c["cam"]), c["scan"])
    ray = _copies(rm.Intrinsics.from_camera(sph), synth.synth_scan(c["mesh"], sph, c["gt"], cases.rng(8), sigma_abs=0.01))
    n = 24
    A, B = _poses(c["gt"], 45, n), _poses(c["gt"], 46, n)

    def calls(poses):
        for scans in (pin, ray):
            want = rm.cost_grad(gm, scans[0], poses)
            _same(rm.cost_grad_batch(gm, scans=_alternate(scans, n), poses=torch.as_tensor(poses)), want)

    calls(A)                                                        # captured
    calls(B)                                                        # replayed, a per-pose call in between
    rm.render_depth(gm, _poses(c["gt"], 47, 200), pin[0].intr)      # larger scratch: both are reallocated
    calls(A)
    gm.set_tuning(bin_capacity=4)                                   # every bin overflows and grows
    for scans in (pin, ray):
        got = rm.cost_grad_batch(gm, scans=_alternate(scans, n), poses=torch.as_tensor(A))
        _same(got, rm.cost_grad(gm, scans[0], A))
    assert gm.get_tuning()["bin_capacity"] > 4
    gm.set_tuning(bin_capacity=4)
    poses, reps, _ = rm.align_batch(gm, scans=[pin[0], ray[0], pin[1]], poses=A[:3], max_iters=9)
    gm.set_tuning()
    for k, sc in enumerate((pin[0], ray[0], pin[1])):
        one, rep = rm.align(gm, sc, A[k], max_iters=9)
        assert np.array_equal(poses[k], one) and reps[k]["e_ls_final"] == rep["e_ls_final"]
    calls(B)
    gm.close()
