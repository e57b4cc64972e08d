"""Steps whose moves go through rounds: what one step leaves to the next."""
import numpy as np
import pytest

from paper_2308_06484_gb300 import workloads as W
from tests.gpu_helpers import assert_same

pytestmark = pytest.mark.gpu


def _tri(**kw):
    from paper_2308_06484_gb300 import kdt
    return kdt.Triangulation(kdt.default_config(**kw))


def _shift(w, ids, seed):
    """Move the points `ids` to free places near by (positions of w follow)."""
    rng = np.random.default_rng(seed)
    xy = w.astype(np.int64)
    taken = set((xy[:, 0] << 32 | xy[:, 1]).tolist())
    out = []
    for p in ids:
        while True:
            x, y = (xy[p] + rng.integers(-9, 10, size=2)).tolist()
            if 0 <= x < 1 << 24 and 0 <= y < 1 << 24 and (x << 32 | y) not in taken:
                break
        taken.add(x << 32 | y)
        w[p] = (x, y)
        out.append((p, x, y))
    return np.array(out, dtype=np.int32)


@pytest.mark.parametrize("graph", [0, 1])
def test_large_step_makes_later_ones_no_longer(graph):
    """Steps of 2,000 moves before and after one of 40,000, one that is a rebuild and a new
    build: as many launches, and no more memory than their own."""
    import torch
    n = 150000
    xy = W.uniform_points(n, 24, 3)
    t = _tri(grid=24, domain_bits=24, use_graph=graph, rebuild_ratio=0.3)
    t.build(xy)
    rng = np.random.default_rng(1)

    def step(m, seed):
        before = t.stats()["kernel_launches"]
        t.step(_shift(xy, rng.permutation(n)[:m], seed))
        return t.stats()["kernel_launches"] - before

    def same():
        assert t.verify() == 0
        assert np.array_equal(t.export_points(), xy)

    first = step(2000, 1)
    same()
    free = torch.cuda.mem_get_info()[0]
    step(130000, 2)  # a rebuild
    assert step(2000, 3) == first
    assert free - torch.cuda.mem_get_info()[0] < 100 << 20
    many = step(40000, 4)
    same()
    assert many > first
    assert step(2000, 5) == first
    same()
    t.build(xy)
    assert step(2000, 6) == first
    assert step(32767, 7) == first and step(32768, 8) == many
    same()
    assert_same(t.export_triangles(), xy, "after steps of all sizes")


def test_steps_of_several_windows():
    """More moves than one round takes (2^18), then few, then more again."""
    n = 1200000
    xy = W.uniform_points(n, 24, 4)
    t = _tri(grid=64, domain_bits=24, rebuild_ratio=0.9)
    t.build(xy)
    rng = np.random.default_rng(2)
    for i, m in enumerate((3000, 262144, 100, 262145, 50, 600000, 3000)):
        t.step(_shift(xy, rng.permutation(n)[:m], 10 + i))
        assert t.verify() == 0
        assert np.array_equal(t.export_points(), xy)
    assert t.stats()["fallbacks"] == 0
