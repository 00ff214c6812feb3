"""Ray tables that share an array in one batch: a crop of the first rows beside the whole table, and
one table under layouts that lie differently far from its rays. Every problem equals rm_cost_grad
bit for bit, in both orders, with the arrays on the device and on the host."""
from __future__ import annotations

import math

import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker is deselected on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1702_06813_gb300 as rm  # noqa: E402
from paper_1702_06813_gb300 import build as rmbuild  # noqa: E402

rmbuild.build()

W, H = 128, 64
AZ_STEP, EL_STEP = 2 * math.pi / W, 0.7 / (H - 1)
OFF = 0.2  # pixels off the layout, of the quarter pixel allowed


def _soup(r, n):
    """n triangles of about half a pixel around the sensor: whether one holds a ray hangs on a
    fraction of a pixel."""
    az, el = r.uniform(-math.pi, math.pi, n), r.uniform(-0.4, 0.4, n)
    d = np.stack([np.cos(el) * np.sin(az), -np.sin(el), np.cos(el) * np.cos(az)], 1)
    c = d * r.uniform(3.0, 40.0, (n, 1))
    size = np.linalg.norm(c, axis=1)[:, None, None] * 0.5 * EL_STEP
    v = c[:, None, :] + r.normal(size=(n, 3, 3)) * size
    return v.reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


def _table(off_rows):
    """The rays of the layout, rows from off_rows on OFF pixels off it on both axes."""
    j, i = np.meshgrid(np.arange(H, dtype=float), np.arange(W, dtype=float), indexing="ij")
    off = np.where(j >= off_rows, OFF, 0.0)
    az, el = -math.pi + AZ_STEP * (i + off + 0.5), 0.35 - EL_STEP * (j + off)
    return np.stack([np.cos(el) * np.sin(az), -np.sin(el), np.cos(el) * np.cos(az)], -1).astype(np.float32)


def _layouts(kind, device):
    """Two intrinsics on one array, the first exactly on its layout."""
    rays = torch.as_tensor(_table(H // 2 if kind == "rows" else H), device=device)

    def intr(h=H, az0=-math.pi, el0=0.35, az_step=AZ_STEP, el_step=EL_STEP):
        return rm.Intrinsics(rm.RM_RAYTABLE, W, h, az0=az0, az_step=az_step, el0=el0, el_step=el_step, near=0.5,
                             far=80.0, rays=rays[:h])

    other = {"rows": dict(), "az0": dict(az0=-math.pi + OFF * AZ_STEP), "el0": dict(el0=0.35 - OFF * EL_STEP),
             "el_step": dict(el_step=EL_STEP * (1 + OFF / (H - 1)))}[kind]
    return intr(h=H // 2 if kind == "rows" else H), intr(**other)


@pytest.mark.parametrize("device", ["cuda", "cpu"])
@pytest.mark.parametrize("kind", ["rows", "az0", "el0", "el_step"])
def test_layouts_on_one_table_equal_single_calls(kind, device):
    r = cases.rng(31)
    v, f = _soup(r, 30000)
    gm = rm.Map(v, f, np.zeros(len(f), np.uint8))
    exact, off = _layouts(kind, device)
    scans = []
    for intr in (exact, off):
        depth = r.uniform(3.0, 40.0, (intr.height, W)).astype(np.float32)
        scans.append(rm.Scan.make(intr, depth, np.zeros(depth.shape, np.uint8), device=device))
    eye = np.eye(4)
    want = [rm.cost_grad(gm, sc, eye[None]) for sc in scans]
    assert all(int(w["counts"].sum()) > 200 for w in want)
    for order in ((0, 1), (1, 0), (0, 1, 0, 1)):
        got = rm.cost_grad_batch(gm, [(scans[k], eye) for k in order])
        for p, k in enumerate(order):
            for key in want[k]:
                assert torch.equal(got[key][p], want[k][key][0]), (kind, order, p, key)
    gm.close()
