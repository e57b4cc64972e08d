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


def _rows(dense, sparse, bits):
    """A dense row of points facing a sparse one: the sparse points' degrees are
    dense / sparse, and each of them is inserted into a cavity of that size."""
    L = 1 << bits
    d = np.stack([np.linspace(0, L - 1, dense).astype(np.int64), np.full(dense, L // 2)], 1)
    s = np.stack([np.linspace(0, L - 1, sparse).astype(np.int64), np.full(sparse, L // 2 + L // (4 * sparse))], 1)
    return np.concatenate([d, s]).astype(np.int32)


@pytest.mark.parametrize("dense,sparse", [(2000, 20), (10000, 100), (20000, 1000)])
def test_rows_of_unlike_density(dense, sparse):
    """Points the rounds cannot take are inserted while their cavities are small: put off to
    the end they cost walks of thousands of steps (2,800 per point) and repairs of as many
    flips."""
    xy = _rows(dense, sparse, 26)
    t = _tri(domain_bits=26)
    t.build(xy)
    st = t.stats()
    assert t.verify() == 0
    assert_same(t.export_triangles(), xy, "rows %d / %d" % (dense, sparse))
    assert st["walk_steps"] < 100 * len(xy)
    assert st["fixup_flips"] < 20 * len(xy)


def test_many_refused_insertions():
    """12,000 rings of 40 points with a centre each: more insertions than 4,096 have a cavity
    beyond 16 lanes.  A build of uniform points takes some 300 launches."""
    k, nr, bits = 40, 12000, 26
    L, g = 1 << bits, 110
    c = L // g
    a = 2 * np.pi * np.arange(k) / k
    base = np.rint(np.stack([0.4 * c * np.cos(a), 0.4 * c * np.sin(a)], 1)).astype(np.int64)
    base = np.concatenate([[[0, 0]], base])
    i = np.arange(nr)
    at = np.stack([(i % g) * c + c // 2, (i // g) * c + c // 2], 1)
    xy = (base[None] + at[:, None]).reshape(-1, 2)
    xy = np.ascontiguousarray(xy[np.random.default_rng(1).permutation(len(xy))].astype(np.int32))
    t = _tri(domain_bits=bits)
    t.build(xy)
    assert t.verify() == 0
    assert t.stats()["kernel_launches"] < 1500


def test_lattice_builds():
    """A lattice (every square's corners cocircular), built often: the order in which
    insertions meet differs from build to build."""
    a = np.arange(300)
    xy = np.ascontiguousarray((np.stack(np.meshgrid(a, a), -1).reshape(-1, 2) * 7).astype(np.int32))
    t = _tri(domain_bits=20)
    for _ in range(50):
        t.build(xy)
    assert t.verify() == 0
    assert_same(t.export_triangles(), xy, "lattice")


@pytest.mark.parametrize("n", list(range(3, 35)))
def test_small_builds(n):
    """Around the sizes where a build changes from levels to rounds; a handful of points takes
    a launch a level (47 launches in rounds)."""
    t = _tri(domain_bits=16)
    for seed in range(4):
        xy = W.uniform_points(n, 16, 100 * n + seed)
        before = t.stats()["kernel_launches"]
        t.build(xy)
        launches = t.stats()["kernel_launches"] - before
        assert_same(t.export_triangles(), xy, "%d points" % n)
        if n <= 16:
            assert launches <= 20
    assert t.verify() == 0


@pytest.mark.parametrize("n,instances", [(3, 5), (4, 300), (5, 40), (8, 40), (9, 40)])
def test_small_instances(n, instances):
    sets = [W.uniform_points(n, 12, i) for i in range(instances)]
    t = _tri(domain_bits=12)
    t.build_batch(sets)
    if n <= 4:
        assert t.stats()["kernel_launches"] <= 20
    for i in range(0, instances, 7):
        assert_same(t.export_triangles_inst(i), sets[i], "instance %d" % i)
    assert t.verify() == 0


@pytest.mark.parametrize("n", [64, 40000, 52000, 1300000])
def test_boxes_of_uneven_instances(n):
    """Instances that begin and end anywhere in the runs of points a warp takes for the bounding
    boxes (runs of 32 to 1,024 points); a point out of range anywhere is refused."""
    from paper_2308_06484_gb300 import kdt
    rng = np.random.default_rng(n)
    cuts = np.unique(np.concatenate([[0, n], 3 + rng.integers(0, n - 6, size=min(300, n // 16))]))
    sizes = np.diff(cuts)
    sizes = sizes[sizes >= 3]
    sets = [W.uniform_points(int(k), 20, i) // (1 + i % 5) for i, k in enumerate(sizes)]
    sets = [np.ascontiguousarray(s[np.sort(np.unique(s, axis=0, return_index=True)[1])]) for s in sets]
    t = _tri(domain_bits=20)
    t.build_batch(sets)
    assert t.verify() == 0
    for i in range(0, len(sets), 1 + len(sets) // 5):
        if len(sets[i]) < 20000:
            assert_same(t.export_triangles_inst(i), sets[i], "instance %d" % i)
    bad = [s.copy() for s in sets]
    bad[-1][-1] = (1 << 20, 5)
    with pytest.raises(kdt.KDTError):
        t.build_batch(bad)


def test_points_left_out_in_a_batch():
    """Instances that leave points out of the rounds beside some that do not."""
    sets = [_rows(2000, 20, 26), W.uniform_points(3000, 26, 1), _rows(900, 30, 26), W.uniform_points(5, 26, 2),
            _rows(1500, 10, 26), W.uniform_points(20000, 26, 3)]
    t = _tri(domain_bits=26)
    for _ in range(3):
        t.build_batch(sets)
        assert t.verify() == 0
        for i, xy in enumerate(sets):
            assert_same(t.export_triangles_inst(i), xy, "instance %d" % i)
