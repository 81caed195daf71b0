"""Decisions by bounds against plain evaluation of every sample: settled blocks
(settle.cuh) against marching every sample (DQJ_MARCH_SAMPLES=0), and every bound
against FP32 and FP64 iteration alone (DQJ_BOUNDS=0), on frames whose tiles do
settle.  Every plane and counter equal bit for bit."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

from bounds_worker import scene_list
from paper_2303_14827_gb300 import binding
from test_gpu_bounds import probe  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _render(path, env_over):
    env = dict(os.environ, DQJ_MARCH_SPLIT="0", **env_over)  # split marches do not settle
    r = subprocess.run([sys.executable, os.path.join(HERE, "bounds_worker.py"), path], env=env,
                       cwd=os.path.dirname(HERE), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return np.load(path)


@pytest.fixture(scope="module")
def default_form(tmp_path_factory):
    return {v: _render(str(tmp_path_factory.mktemp("a") / f"{v}.npz"), {"DQJ_MARCH_VARIANT": v}) for v in ("0", "1")}


@pytest.mark.parametrize("variant", ("1", "0"))
@pytest.mark.parametrize("switch", ("DQJ_BOUNDS", "DQJ_MARCH_SAMPLES"))
def test_bounds_change_nothing(tmp_path, default_form, variant, switch):
    a, b = default_form[variant], _render(str(tmp_path / "b.npz"), {"DQJ_MARCH_VARIANT": variant, switch: "0"})
    assert sorted(a.files) == sorted(b.files)
    hits = 0
    for k in a.files:
        if k.endswith("_stats"):  # no overflow: every plane and counter is deterministic
            assert a[k][7] == 0 and b[k][7] == 0, (k, a[k][7], b[k][7])
    for k in a.files:
        assert np.array_equal(a[k], b[k], equal_nan=a[k].dtype.kind == "f"), (k, a[k].ravel()[:12], b[k].ravel()[:12])
        if k.endswith("_stats"):
            hits += int(a[k][3])
    assert hits > 5 * 10 ** 5


def test_scenes_settle(probe):  # noqa: F811
    import torch
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    settled = 0
    for s in scene_list():
        p = binding.make_params(s)
        on = ctypes.c_int32()
        n.zero_()
        assert probe.probe_settled(ctypes.byref(p), ctypes.byref(on), ctypes.c_void_p(n.data_ptr())) == 0
        assert on.value == 1, (s["width"], s["march_steps"], s["precision"])
        settled += int(n) > 0.05 * s["width"] * s["height"] * s["march_steps"] / 64
    assert settled >= 0.8 * len(scene_list())
