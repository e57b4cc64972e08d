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


def test_refused_moves_are_planned_by_32_lanes_once():
    """150 hubs of degree 20 move at once: beyond 16 lanes, which refuse a move once and not in
    every round (two refusals each counted 300 retries)."""
    k, nr, c = 20, 150, 100000
    a = 2 * np.pi * (np.arange(k) + 0.3) / k
    r = 20000.0 + 7 * (np.arange(k) % 5)
    rim = np.rint(np.stack([r * np.cos(a), r * np.sin(a)], 1)).astype(np.int64)
    i = np.arange(nr)
    at = np.stack([i % 13, i // 13], 1) * c + c // 2
    xy = np.ascontiguousarray((np.concatenate([[[0, 0]], rim])[None] + at[:, None]).reshape(-1, 2).astype(np.int32))
    t = _tri(grid=8, domain_bits=21, rebuild_ratio=2.0)
    t.build(xy)
    hubs = (k + 1) * i
    before = t.stats()
    for s in (3, -5):
        mv = np.stack([hubs, xy[hubs, 0] + s, xy[hubs, 1] + 2], 1).astype(np.int32)
        xy[hubs] = mv[:, 1:]
        t.step(mv)
        assert_same(t.export_triangles(), xy, "hubs")
    st = t.stats()
    assert st["retries"] - before["retries"] < 100
    assert st["deletes"] - before["deletes"] == 2 * nr and st["fallbacks"] == 0


def test_long_walks_are_walked_once_in_the_rounds():
    """Two rows of 9,000 points: a jump from one end to the other crosses more triangles than the
    rounds walk (4,096).  They give up once: 4,097 steps a move more than the kinetic kernel
    alone, whose walks restart at random places (12,291 where three rounds tried).  1,000
    jumps each: the walks are shorter than 1e5 steps and scatter by 1e4, their means by 450,
    so the line is 8 of these from either figure."""
    n, m = 9000, 100
    x = 200 * np.arange(n, dtype=np.int64)
    xy = np.concatenate([np.stack([x, 1000 + (x // 200) % 7], 1), np.stack([x + 90, 1300 + (x // 200) % 5], 1)])
    xy = np.ascontiguousarray(xy.astype(np.int32))
    steps = []
    for kw in (dict(), dict(kinetic_warps=m)):
        p = xy.copy()
        t = _tri(grid=4, domain_bits=21, **kw)
        t.build(p)
        ids = 40 + 9 * np.arange(m)
        before = t.stats()["walk_steps"]
        for s in range(10):
            to = 200 * (n - 60 - 7 * np.arange(m)) + 45 if s % 2 == 0 else 200 * ids + 45
            mv = np.stack([ids, to, np.full(m, 1150)], 1).astype(np.int32)
            p[ids] = mv[:, 1:]
            t.step(mv)
            assert t.verify() == 0
        assert np.array_equal(t.export_points(), p)
        assert_same(t.export_triangles(), p, "jumps")
        steps.append((t.stats()["walk_steps"] - before) / (10 * m))
    assert steps[0] - steps[1] < 8000


@pytest.mark.parametrize("graph", [0, 1])
def test_small_steps_end_at_32_moves(graph):
    """Up to two moves a warp of one block take its three launches, more the whole GPU's."""
    n = 5000
    xy = W.uniform_points(n, 24, 8)
    t = _tri(grid=4, domain_bits=24, use_graph=graph)
    t.build(xy)
    rng = np.random.default_rng(3)
    for i, m in enumerate((1, 31, 32, 33, 64, 65, 32, 16, 17)):
        before = t.stats()["kernel_launches"]
        t.step(_shift(xy, rng.permutation(n)[:m], 50 + i))
        assert (t.stats()["kernel_launches"] - before == 3) == (m <= 32)
        assert_same(t.export_triangles(), xy, "%d moves" % m)
