"""rm_cost_grad_noalloc with a ray table: setup without a z-buffer, so that every triangle goes through
the bins, equals rm_cost_grad bit for bit and matches the oracle; with rays on their layout and off it
by up to a quarter pixel.

Collected last (file name), as test_zz_no_alloc.py."""
from __future__ import annotations

import pytest

import cases
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - the gpu marker is deselected on CPU
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_ray_direct import _Table  # noqa: E402
from test_zz_no_alloc import _against_oracle, _two_calls  # noqa: E402


@pytest.mark.parametrize("w,h,off", [(96, 16, 0.0), (360, 32, 0.24), (301, 21, 0.1)])
def test_noalloc_ray_table(w, h, off):
    c = cases.config1(seed=1000)
    base = cases.small_spherical(w, h)
    cam = _Table(**{**base.__dict__, "off": off})
    scan = synth.synth_scan(c["mesh"], cam, c["gt"], cases.rng(w), sigma_abs=0.01)
    poses = [c["start"], synth.perturb_fixed(c["gt"], cases.rng(7), 0.1, 3.0)]
    res = _two_calls(c["mesh"], cam, scan, poses)
    assert res[0][0]["counts"].sum() > 0
    _against_oracle(c["mesh"], cam, scan, poses[0], res[0][0])
