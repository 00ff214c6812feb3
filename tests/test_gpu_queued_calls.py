"""Calls that return before the device is done (async_status): on several streams they run one after
another, from the first call on a new map on; and a captured call, replayed between others, equals
them bit for bit."""
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
from paper_1702_06813_gb300 import _native as N  # noqa: E402
from paper_1702_06813_gb300 import build as rmbuild  # noqa: E402

rmbuild.build()


@pytest.fixture(scope="module")
def scene():
    c = cases.config1(seed=1000)
    scan = rm.Scan.make(rm.Intrinsics.from_camera(c["cam"]), *c["scan"])
    r = cases.rng(61)
    poses = torch.as_tensor(np.stack([synth.perturb_fixed(c["gt"], r, 0.1, 3.0) for _ in range(600)])).cuda()
    torch.cuda.synchronize()  # the scan and the poses are ready for every stream
    gm = rm.Map(c["mesh"].vertices, c["mesh"].faces, c["mesh"].labels)
    want = rm.cost_grad(gm, scan, poses)
    gm.close()
    return c["mesh"], scan, poses, want


def _same(got, want, sel):
    for key in want:
        assert torch.equal(got[key], want[key][sel]), key


def _finish(gm):
    N.check(N.lib().rm_status_sync(gm.handle, None))


def test_calls_on_two_streams_run_in_turn(scene):
    mesh, scan, poses, want = scene
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    gm.set_tuning(async_status=True)
    parts = [slice(0, 500), slice(500, 503), slice(100, 400), slice(503, 600)]
    for turn in range(3):  # the first on the new map
        got = []
        for k, sel in enumerate(parts):
            with torch.cuda.stream(streams[k % 2]):
                got.append(rm.cost_grad(gm, scan, poses[sel]))
        torch.cuda.synchronize()
        _finish(gm)
        for g, sel in zip(got, parts):
            _same(g, want, sel)
    gm.close()


def test_captured_call_between_others(scene):
    mesh, scan, poses, want = scene
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    gm.set_tuning(async_status=True)
    sel = slice(0, 8)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        rm.cost_grad(gm, scan, poses[sel])  # sizes the scratch
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        got = rm.cost_grad(gm, scan, poses[sel])
    for turn in range(3):
        _same(rm.cost_grad(gm, scan, poses[8:12]), want, slice(8, 12))  # the comparison waits
        torch.cuda.synchronize()
        for t in got.values():
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        _same(got, want, sel)
    _finish(gm)
    gm.close()


def test_status_waits_for_a_call_on_another_stream(scene):
    mesh, scan, poses, want = scene
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    rm.cost_grad(gm, scan, poses)  # sizes the scratch
    gm.set_tuning(async_status=True)
    s = torch.cuda.Stream()
    for turn in range(3):
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)  # about 10 ms
            got = rm.cost_grad(gm, scan, poses)
        _finish(gm)
        assert s.query()
        _same(got, want, slice(None))
    gm.close()


def test_normals_replaced_while_a_call_is_queued(scene):
    mesh, scan, poses, _ = scene
    n = np.random.Generator(np.random.PCG64(3)).normal(size=(2, len(mesh.vertices), 3)).astype(np.float32)
    normals = torch.as_tensor(n).cuda()
    gm = rm.Map(mesh.vertices, mesh.faces, mesh.labels)
    want = []
    for k in range(2):
        gm.set_vertex_normals(normals[k])
        want.append(rm.icp_terms(gm, scan, poses, tol=0.1))
    gm.set_tuning(async_status=True)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for turn in range(3):  # the map's normals are those of turn - 1 (1 at first)
        with torch.cuda.stream(s):
            torch.cuda._sleep(4_000_000)
            got = rm.icp_terms(gm, scan, poses, tol=0.1)
        gm.set_vertex_normals(normals[turn % 2])
        _finish(gm)
        _same(got, want[(turn + 1) % 2], slice(None))
    gm.close()
