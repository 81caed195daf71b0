"""The FP64 re-trace of sphere tracing's recheck mode takes its pixels from lists
by the cost of their rays.  Every hit of the FP32 trace is re-traced, so wherever
the recheck frame and the FP64 frame hit, their planes come from the same FP64
trace: the escape counts are equal, the depths within one rounding to FP32 (two
compilations of one FP64 expression), and no pixel is lost or traced twice."""
import numpy as np
import pytest

from paper_2303_14827_gb300 import binding, scenes
from parity import to_numpy

pytestmark = pytest.mark.gpu

SLICE = scenes.random_slice_frame(np.random.default_rng(7))
CASES = {
    "one": dict(width=1, height=1),
    "row": dict(width=31, height=1, fov_y_deg=1.0),
    "chunk_and_one": dict(width=33, height=5),
    "all_classes": dict(width=301, height=217, max_iter=24),  # costs 20 to above 3000
    "long": dict(width=96, height=64, de_step_scale=0.25, de_epsilon=1e-4),
    "short": dict(width=96, height=64, de_max_steps=3),
    "general": dict(width=130, height=67, slice_basis=SLICE),
    "dualnum": dict(width=65, height=64, modulus_mode=scenes.MODULUS_DUALNUM, square_mode=1),
}


@pytest.fixture(scope="module")
def rdr():
    r = binding.Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("name", sorted(CASES))
def test_retraced_pixels_equal_fp64(rdr, name):
    s = scenes.default_scene(traversal=scenes.TRAVERSAL_DE, **CASES[name])
    w, h = s["width"], s["height"]
    ref = to_numpy(rdr.render(dict(s, precision=scenes.PRECISION_FP64)), w, h)
    plain = rdr.render(dict(s, precision=scenes.PRECISION_FP32))
    hits32 = binding.stats_dict(plain["stats"])["hits"]
    first = None
    for _ in range(2):
        o = rdr.render(dict(s, precision=scenes.PRECISION_FP32_RECHECK))
        g, st = to_numpy(o, w, h), binding.stats_dict(o["stats"])
        assert hits32 <= st["fixups"] <= w * h
        both = np.isfinite(g["depth"]) & np.isfinite(ref["depth"])
        assert np.array_equal(g["iter"][both], ref["iter"][both])
        d, r = g["depth"][both].astype(np.float64), ref["depth"][both].astype(np.float64)
        assert np.all(np.abs(d - r) <= 2.0 ** -23 * np.abs(r))
        if first is not None:
            assert all(np.array_equal(g[k], first[0][k]) for k in g if k != "stats") and st == first[1]
        first = (g, st)
