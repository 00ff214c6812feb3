"""Batches over host arrays, which the library stages: scans and ray tables shared between problems and
of several sizes, and a class array that starts at the address of another scan's depth. Every
problem equals rm_cost_grad on the device bit for bit."""
from __future__ import annotations

import time

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


@pytest.fixture(scope="module")
def scene():
    c = cases.config1(seed=1000)
    gm = rm.Map(c["mesh"].vertices, c["mesh"].faces, c["mesh"].labels)
    yield c, gm
    gm.close()


def _same_as_calls(gm, probs):
    got = rm.cost_grad_batch(gm, probs)
    for k, (sc, pose) in enumerate(probs):
        rays = None if sc.intr.rays is None else sc.intr.rays.cuda()
        intr = rm.Intrinsics(**{**sc.intr.__dict__, "rays": rays})
        want = rm.cost_grad(gm, rm.Scan(intr, sc.depth.cuda(), sc.cls.cuda()), pose[None])
        assert int(want["counts"].sum()) > 0, k
        for key in want:
            assert torch.equal(got[key][k], want[key][0]), (k, key)


def test_class_array_at_the_address_of_a_depth_array(scene):
    c, gm = scene
    cam = c["cam"]
    intr = rm.Intrinsics.from_camera(cam)
    shape, n = (cam.height, cam.width), cam.width * cam.height
    shared = torch.as_tensor(np.asarray(c["scan"][0], np.float32)).nan_to_num(1.0).contiguous()
    bytes_ = shared.view(torch.uint8).reshape(-1)[:n].reshape(shape)  # classes 0 to 255: above 2 is NaN
    a = rm.Scan(intr, torch.full(shape, 2.0), bytes_)
    b = rm.Scan(intr, shared, torch.zeros(shape, dtype=torch.uint8))
    assert a.cls.data_ptr() == b.depth.data_ptr()
    for probs in ([(a, c["start"]), (b, c["gt"])], [(b, c["gt"]), (a, c["start"])]):
        _same_as_calls(gm, probs)


def test_shared_host_arrays_of_several_sizes(scene):
    c, gm = scene
    r = cases.rng(17)
    scans = []
    for cam in (c["cam"], cases.small_pinhole(97, 41, 80.0), cases.small_spherical(96, 16), cases.small_spherical(61, 9)):
        sd, sc = synth.synth_scan(c["mesh"], cam, c["gt"], r, sigma_abs=0.01)
        scans.append(rm.Scan.make(rm.Intrinsics.from_camera(cam, device="cpu"), sd, sc, device="cpu"))
    scans.append(rm.Scan(scans[2].intr, scans[2].depth * 1.01, scans[2].cls))  # its table and classes, another depth
    order = [2, 0, 1, 0, 3, 4, 2, 1, 3]
    _same_as_calls(gm, [(scans[k], synth.perturb_fixed(c["gt"], r, 0.03, 1.0)) for k in order])


def test_many_host_scans_take_time_in_proportion(scene):
    """Eight times the scans, each with its own host arrays, take about eight times as long (a search
    of the list of arrays for each of them: 31 times)."""
    c, gm = scene
    intr = rm.Intrinsics.from_camera(cases.small_pinhole(16, 16, 14.0))
    scans = [rm.Scan(intr, torch.full((16, 16), 2.0 + 1e-3 * k), torch.zeros((16, 16), dtype=torch.uint8))
             for k in range(4096)]
    poses = torch.as_tensor(c["gt"]).cuda().expand(4096, 4, 4).contiguous()

    def best(n):
        rm.cost_grad_batch(gm, scans=scans[:n], poses=poses[:n])
        took = []
        for _ in range(5):
            t = time.perf_counter()
            rm.cost_grad_batch(gm, scans=scans[:n], poses=poses[:n])
            took.append(time.perf_counter() - t)
        return min(took)

    assert best(4096) < 16 * best(512)
