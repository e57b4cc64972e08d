"""The ways a build takes besides its usual rounds: a chosen number of inserting warps."""
import numpy as np
import pytest

from paper_2308_06484_gb300 import workloads as W
from tests.gpu_helpers import assert_same

pytestmark = pytest.mark.gpu


def _tri(**kw):
    from paper_2308_06484_gb300 import kdt
    return kdt.Triangulation(kdt.default_config(**kw))


@pytest.mark.parametrize("warps", [1, 3, 64, 1000])
def test_build_warps(warps):
    """Level by level: every walk starts at a point of the coarser levels next to it, so it
    takes a few steps (3 to 8 on average; from the first triangle 24 to 60)."""
    xy = W.uniform_points(20000, 20, 7)
    t = _tri(domain_bits=20, build_warps=warps)
    t.build(xy)
    st = t.stats()
    assert st["walk_steps"] < 15 * len(xy)
    assert_same(t.export_triangles(), xy, "build with %d warps" % warps)
    assert t.verify() == 0


def test_build_warps_batch():
    sets = [W.uniform_points(n, 18, n) for n in (3, 4, 40, 700, 2000)]
    t = _tri(domain_bits=18, build_warps=7)
    t.build_batch(sets)
    for i, xy in enumerate(sets):
        assert_same(t.export_triangles_inst(i), xy, "instance %d" % i)
    assert t.verify() == 0
