"""Kernel variants chosen by size, at the sizes where each can go wrong."""
import numpy as np
import pytest

from synth import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1910_01011_gb300 import api as a
    return a


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def test_short_chunks_fall_back_under_a_budget(api):
    """Where the budget does not hold the partials of short source chunks, the
    FP32 product takes the longer ones: the same bits as with that chunk
    length asked for (640 tiles: four chunks of 160)."""
    s = scenes.sphere_scene(5)
    x = scenes.smooth_trace_vector(s, 3)
    c = api.Context.from_scene(s)
    c.apply(x, precision=api.FP32)
    used = c.memory()[0]
    c.close()
    c = api.Context.from_scene(s, chunk_tiles=160)
    ref = c.apply(x, precision=api.FP32)
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used - (1 << 20))  # the short chunks' partials miss by 1 MiB
    y = c.apply(x, precision=api.FP32)
    assert np.array_equal(y, ref)
    assert c.memory()[0] < used - (1 << 28)
    c.close()
