"""Rounds of operations (kdt_rounds.cuh, kdt_region.cuh) where their limits lie: degrees,
cavities and borders around 16 and 32 lanes, hull points, moves that meet, more moves than
one round takes.  Exact, against the oracle (or the verifier's certificate)."""
import numpy as np
import pytest

import oracle
from paper_2308_06484_gb300 import workloads as W
from tests.gpu_helpers import assert_same

pytestmark = pytest.mark.gpu


def _tri(**kw):
    from paper_2308_06484_gb300 import kdt
    return kdt.Triangulation(kdt.default_config(**kw))


def _wheel(k):
    """A hub with k neighbours around it at nearly one distance, and a frame far out."""
    a = 2 * np.pi * (np.arange(k) + 0.3) / k
    r = 20000.0 + 7 * (np.arange(k) % 5)
    rim = np.stack([(1 << 19) + r * np.cos(a), (1 << 19) + r * np.sin(a)], 1)
    frame = np.random.default_rng(k).integers(0, 1 << 20, size=(60, 2))
    frame = frame[np.hypot(frame[:, 0] - (1 << 19), frame[:, 1] - (1 << 19)) > 150000]
    xy = np.concatenate([[[1 << 19, 1 << 19]], np.rint(rim).astype(np.int64), frame])
    return np.ascontiguousarray(xy.astype(np.int32))


@pytest.mark.parametrize("k", [3, 4, 5, 15, 16, 17, 31, 32, 33])
def test_hub_of_degree(k):
    """The hub moves inside its star, out of it and back (the cavity of its return is the
    wheel), alone and with a rim point in the same step."""
    xy = _wheel(k)
    t = _tri(grid=2, domain_bits=20)
    t.build(xy)
    c = 1 << 19
    far = (c + 90000, c + 3)
    for hub, rim in (((c + 5, c), None), (far, None), ((c, c + 1), None), (far, 1), ((c - 2, c + 9), 2)):
        mv = [(0,) + hub]
        if rim is not None:
            mv.append((rim, int(xy[rim, 0]) + 11, int(xy[rim, 1]) - 6))
        for i, x, y in mv:
            xy[i] = (x, y)
        t.step(np.array(mv, dtype=np.int32))
        assert_same(t.export_triangles(), xy, "hub of degree %d" % k)
    assert t.verify() == 0 and t.stats()["fallbacks"] == 0


@pytest.mark.parametrize("n", [5, 17, 40])
def test_hull_points_move(n):
    """Points in convex position (every one on the hull): each moves out, in, and along."""
    i = np.arange(n)
    xy = np.ascontiguousarray(np.stack([2000 + 700 * i, 3000 + 9 * i * i], 1).astype(np.int32))
    t = _tri(grid=2, domain_bits=16)
    t.build(xy)
    rng = np.random.default_rng(n)
    for s in range(12):
        ids = rng.choice(n, size=max(1, n // 4), replace=False)
        new = xy.copy()
        new[ids] += rng.integers(-400, 401, size=(ids.size, 2)).astype(np.int32)
        if np.unique(new, axis=0).shape[0] < n or new.min() < 0:
            continue
        # (a target on another mover's old place is a case of its own: see the chain test)
        if (new[ids][:, None] == xy[None]).all(2).any():
            continue
        xy = new
        t.step(np.concatenate([ids[:, None], xy[ids]], 1).astype(np.int32))
        assert_same(t.export_triangles(), xy, "hull n=%d step %d" % (n, s))
    assert t.verify() == 0


@pytest.mark.parametrize("n,frac", [(40, 1.0), (3000, 1.0), (3000, 0.3)])
def test_dense_moves(n, frac):
    """Most moves meet: many rounds, and what they leave to the warp-wide path."""
    import torch
    w = W.KineticWorkload(W.uniform_points(n, 18, n), 1, 18, (int(n * frac), int(n * frac)), (1, 3000), seed=n + 1)
    t = _tri(grid=1, domain_bits=18, rebuild_ratio=2.0)
    t.build(w.positions)
    for s in range(4):
        t.step(torch.from_numpy(w.next_moves()).cuda())
        assert_same(t.export_triangles(), w.positions, "dense n=%d step %d" % (n, s))
    assert t.verify() == 0


@pytest.mark.parametrize("side", [2, 15, 16, 17, 31, 33, 70])
def test_build_rows(side):
    """Two collinear rows: insertions that see a whole row (borders around the lanes' limits)."""
    x = np.arange(side) * 6
    xy = np.concatenate([np.stack([x, np.zeros_like(x)], 1), np.stack([x + 3, np.full_like(x, 40000)], 1)])
    xy = np.ascontiguousarray(xy[np.random.default_rng(side).permutation(2 * side)].astype(np.int32))
    t = _tri(domain_bits=16)
    t.build(xy)
    assert_same(t.export_triangles(), xy, "rows of %d" % side)
    assert t.verify() == 0


def test_more_moves_than_a_round():
    """A step of more than 2^18 moves (several windows): the verifier's certificate and the
    positions."""
    import torch
    n, m = 1_200_000, (1 << 18) + 5000
    xy = W.uniform_points(n, 24, 5)
    t = _tri(grid=68, domain_bits=24)
    t.build(xy)
    rng = np.random.default_rng(6)
    ids = rng.choice(n, size=m, replace=False)
    new = xy.copy()
    new[ids] = (new[ids].astype(np.int64) + rng.integers(-8, 9, size=(m, 2))).clip(0, (1 << 24) - 1).astype(np.int32)
    key = (new[:, 0].astype(np.int64) << 32) | new[:, 1]
    old = (xy[:, 0].astype(np.int64) << 32) | xy[:, 1]
    _, first, cnt = np.unique(np.concatenate([old, key[ids]]), return_index=True, return_counts=True)
    clash = np.isin(key, np.concatenate([old, key[ids]])[first[cnt > 1]])
    ids = ids[~clash[ids]]
    assert ids.size > 1 << 18
    xy[ids] = new[ids]
    t.step(torch.from_numpy(np.concatenate([ids[:, None], xy[ids]], 1).astype(np.int32)).cuda())
    assert np.array_equal(t.export_points(), xy)
    assert t.verify() == 0
    assert t.stats()["rebuilds"] == 1


@pytest.mark.parametrize("n,hub", [(3, 0), (15, 0), (16, 0), (17, 0), (4097, 0), (33000, 0), (600, 500), (40000, 9000)])
def test_export_buckets(n, hub):
    """The export in buckets of first ids: one bucket, its last id, several ids a bucket; and a
    bucket with more rows than its block holds (a fan of `hub` triangles around id 0), which
    is placed instead.  Into host and device memory, and with too little room."""
    import torch
    from paper_2308_06484_gb300 import kdt
    if hub:
        a = np.pi * np.arange(hub) / (hub - 1)
        rim = np.stack([(1 << 27) + 1e8 * np.cos(a), (1 << 26) + 1e8 * np.sin(a)], 1)
        rest = W.uniform_points(n - hub - 1, 20, 3)
        xy = np.concatenate([[[1 << 27, 1 << 26]], np.rint(rim), rest]).astype(np.int32)
        xy = np.concatenate([xy[:1], np.unique(xy[1:], axis=0)])
    else:
        xy = W.uniform_points(n, 24, n)
    t = _tri(domain_bits=28)
    t.build(np.ascontiguousarray(xy))
    got = t.export_triangles()
    assert_same(got, xy, "export n=%d" % n)
    out = torch.full((2 * len(xy), 3), -1, dtype=torch.int32, device="cuda")
    assert np.array_equal(t.export_triangles(out).cpu().numpy(), got)
    assert int((out[got.shape[0]:] != -1).sum()) == 0
    out.fill_(-1)
    if got.shape[0] > 1:
        with pytest.raises(kdt.KDTError) as e:
            t.export_triangles(out[:got.shape[0] - 1])
        assert e.value.name == "KDT_ERR_CAPACITY" and int((out != -1).sum()) == 0


@pytest.mark.parametrize("grid", [90, 91])
@pytest.mark.parametrize("m", [1, 2, 63, 64, 65])
def test_small_step_limits(grid, m):
    """One block's steps (up to 64 moves, up to 8192 partitions) and those just past them."""
    w = W.KineticWorkload(W.uniform_points(700, 18, m), grid, 18, (0, 0), (1, 1), seed=3)
    xy = np.array(w.positions)
    rng = np.random.default_rng(m)
    t = _tri(grid=grid, domain_bits=18, rebuild_ratio=2.0)
    t.build(xy)
    for s in range(4):
        ids = rng.choice(len(xy), size=m, replace=False)
        new = xy.copy()
        new[ids] = (new[ids] + rng.integers(-9000, 9001, size=(m, 2))).clip(0, (1 << 18) - 1)
        both = np.concatenate([xy, new[ids]])
        assert np.unique(both, axis=0).shape[0] == len(both)
        xy = new.astype(np.int32)
        t.step(np.concatenate([ids[:, None], xy[ids]], 1).astype(np.int32))
        assert_same(t.export_triangles(), xy, "grid %d m %d step %d" % (grid, m, s))
    st = t.stats()
    assert t.verify() == 0 and st["fallbacks"] == 0 and st["rebuilds"] == 1


@pytest.mark.parametrize("hubs", [255, 256, 257])
def test_leftovers_as_list_or_by_partition(hubs):
    """Hubs of degree 40 (more triangles than a round's lanes hold) all go to the kinetic
    kernel: as a list up to a quarter of the least room for moves (256), else by partition."""
    i = np.arange(17 * 17)[:hubs]
    c = np.stack([70000 + 100000 * (i % 17), 70000 + 100000 * (i // 17)], 1)
    a = 2 * np.pi * (np.arange(40) + 0.3) / 40
    r = 20000.0 + 7 * (np.arange(40) % 5)
    rim = np.rint(np.stack([r * np.cos(a), r * np.sin(a)], 1)).astype(np.int64)
    xy = np.concatenate([c, (c[:, None] + rim[None]).reshape(-1, 2)]).astype(np.int32)
    tri = oracle.delaunay(xy)
    assert (np.bincount(tri.ravel(), minlength=len(xy))[:hubs] >= 40).all()
    t = _tri(grid=4, domain_bits=21, rebuild_ratio=2.0)
    t.build(xy)
    for s in range(3):
        xy[:hubs] += np.array([3, -2], np.int32)
        t.step(np.concatenate([i[:, None], xy[:hubs]], 1).astype(np.int32))
        assert_same(t.export_triangles(), xy, "%d hubs step %d" % (hubs, s))
    assert t.verify() == 0 and t.stats()["fallbacks"] == 0


@pytest.mark.parametrize("quadtree", [0, 1, 2])
def test_arrays_kept_between_builds(quadtree):
    """One handle over point sets that fit the last one's arrays, that do not, that are far
    smaller, batches of them, and one that is refused: a step after each, exact."""
    from paper_2308_06484_gb300 import kdt
    t = _tri(domain_bits=20, points_per_partition=64, quadtree=quadtree, rebuild_ratio=2.0)
    rng = np.random.default_rng(1)

    def moved(xy):
        new = xy.copy()
        ids = rng.choice(len(xy), size=max(1, len(xy) // 20), replace=False)
        new[ids] = (new[ids] + rng.integers(-3000, 3001, size=(ids.size, 2))).clip(0, (1 << 20) - 1)
        assert np.unique(np.concatenate([xy, new[ids]]), axis=0).shape[0] == len(xy) + ids.size
        return new.astype(np.int32), np.concatenate([ids[:, None], new[ids]], 1).astype(np.int32)

    for k, sizes in enumerate([(5000,), (4000,), (1300,), (1000,), (20000,), (300, 800, 3), (900,), None, (700,),
                               (3,), (40, 50), (6000,)]):
        if sizes is None:
            dup = W.uniform_points(800, 20, 9)
            dup[5] = dup[700]
            with pytest.raises(kdt.KDTError) as e:
                t.build(dup)
            assert e.value.name == "KDT_ERR_DUPLICATE"
            continue
        xys = [W.uniform_points(n, 20, 10 * k + j) for j, n in enumerate(sizes)]
        if len(xys) == 1:
            t.build(xys[0])
            new, mv = moved(xys[0])
            t.step(mv)
            assert_same(t.export_triangles(), new, "build %d" % k)
        elif quadtree:  # (one point set only: refused, the triangulation stays as it was)
            with pytest.raises(kdt.KDTError) as e:
                t.build_batch(xys)
            assert e.value.name == "KDT_ERR_ARG"
            assert_same(t.export_triangles(), new, "build %d" % k)
        else:
            t.build_batch(xys)
            parts = [moved(x) for x in xys]
            t.step_batch(np.concatenate([p[1] for p in parts]), np.cumsum([0] + [len(p[1]) for p in parts]))
            for j, p in enumerate(parts):
                assert_same(t.export_triangles_inst(j), p[0], "build %d instance %d" % (k, j))
        assert t.verify() == 0
