"""Batches whose evaluations span several captured graphs: every problem's LM and ICP end, for
iteration counts around the graph's length, equals the single-problem call's bit for bit; with one
camera model only, both, host arrays and shared scans; and a plain mixed batch equals the per-pose
calls."""
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


@pytest.fixture(scope="module")
def scene():
    c = cases.config1(seed=1000)
    mesh = c["mesh"]
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    sph = cases.small_spherical(w=96, h=16)
    r = cases.rng(5)
    sd, sc = synth.synth_scan(mesh, sph, c["gt"], r, sigma_abs=0.01)
    scans = {"pin": rm.Scan.make(rm.Intrinsics.from_camera(c["cam"]), *c["scan"]),
             "ray": rm.Scan.make(rm.Intrinsics.from_camera(sph), sd, sc)}
    poses = [synth.perturb_fixed(c["gt"], r, 0.04, 1.5) for _ in range(3)]
    yield gm, scans, poses
    gm.close()


@pytest.mark.parametrize("kinds", ["pin", "ray", "mixed"])
@pytest.mark.parametrize("iters", [1, 7, 8, 9, 17])
def test_align_batches_equal_single_calls(scene, kinds, iters):
    gm, scans, poses = scene
    names = {"pin": ["pin"] * 3, "ray": ["ray"] * 3, "mixed": ["ray", "pin", "ray"]}[kinds]
    probs = [(scans[k], p) for k, p in zip(names, poses)]
    got, reps, _ = rm.align_batch(gm, probs, max_iters=iters)
    icp, ireps, _ = rm.icp_align_batch(gm, probs, tol=0.2, max_iters=iters)
    for k, (sc, p) in enumerate(probs):
        one, rep = rm.align(gm, sc, p, max_iters=iters)
        assert np.array_equal(got[k], one), (kinds, iters, k)
        assert {f: reps[k][f] for f in reps[k]} == {f: rep[f] for f in reps[k]}, (kinds, iters, k)
        one, rep = rm.icp_align(gm, sc, p, tol=0.2, max_iters=iters)
        assert np.array_equal(icp[k], one), (kinds, iters, k)
        assert {f: ireps[k][f] for f in ireps[k]} == {f: rep[f] for f in ireps[k]}, (kinds, iters, k)


def test_plain_mixed_batch_equals_calls(scene):
    gm, scans, poses = scene
    probs = [(scans["pin"], poses[0]), (scans["ray"], poses[1]), (scans["pin"], poses[2])]
    b = rm.cost_grad_batch(gm, probs)
    for k, (sc, p) in enumerate(probs):
        one = rm.cost_grad(gm, sc, p[None])
        for f in b:
            assert torch.equal(b[f][k], one[f][0]), (f, k)
