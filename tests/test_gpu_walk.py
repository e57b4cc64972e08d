"""The d-calculation's walk over the stars (kdt_dcalc.cuh) at the edges of its list widths,
with and without the build's order of the points; the network's kernels (kdt_tc.cuh) with
rows that are not on a 16-byte boundary."""
import numpy as np
import pytest

from oracle import dcalc as D
from oracle import mlp_ref as M
from paper_2308_06484_gb300 import workloads as W
from tests.test_gpu_proposal import _batch, _cuda, _params

pytestmark = pytest.mark.gpu


def _tri(**kw):
    from paper_2308_06484_gb300 import kdt
    return kdt.Triangulation(kdt.default_config(**kw))


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 8, 9, 15, 16])
def test_list_widths(N):
    """Uniform points, ties (a lattice), and the least number of points a query may have;
    after a step, when the order is the old positions'."""
    g = np.stack(np.meshgrid(np.arange(13) * 8, np.arange(9) * 8), -1).reshape(-1, 2).astype(np.int32)
    for xy in (W.uniform_points(700, 20, N), g, W.uniform_points(N + 1 if N > 1 else 3, 20, N)):
        t = _tri(grid=2, domain_bits=20, rebuild_ratio=2.0)
        t.build(xy)
        for s in range(2):
            dist2 = np.empty(len(xy), np.int64)
            t.d_values(N, dist2)
            assert np.array_equal(dist2, D.nth_nn_dist2(xy, N))
            xy = xy.copy()
            ids = np.arange(0, len(xy), 3)
            xy[ids, 0] += 3  # (the lattice's steps are 8: no two points meet)
            if np.unique(xy, axis=0).shape[0] < len(xy):
                break
            t.step(np.concatenate([ids[:, None], xy[ids]], 1).astype(np.int32))


@pytest.mark.parametrize("batch_build", [0, 1])
@pytest.mark.parametrize("N", [1, 3, 9])
def test_batch_with_and_without_the_order(batch_build, N):
    """Instances built one at a time leave no order over all points."""
    parts = [W.uniform_points(n, 20, n) for n in (40, 333, 1200)]
    t = _tri(domain_bits=20, batch_build=batch_build)
    t.build_batch(parts)
    dist2 = np.empty(sum(len(p) for p in parts), np.int64)
    t.d_values(N, dist2)
    assert np.array_equal(dist2, np.concatenate([D.nth_nn_dist2(p, N) for p in parts]))


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("rows", [1, 127, 129, 1000])
def test_rows_off_the_boundary(rows, off):
    """The same values 4, 8 and 12 bytes off a 16-byte boundary: the same bits."""
    import torch
    t = _tri(domain_bits=24)
    _, bits = _params(3)
    w = _cuda(bits.view(np.int16))
    X, y = _batch(rows, 4)
    x = _cuda(X)
    buf = torch.zeros(rows * 32 + 4, dtype=torch.float32, device="cuda")
    xo = buf[off:off + rows * 32].view(rows, 32)
    xo.copy_(x)
    assert xo.data_ptr() % 16 == 4 * off
    out = [torch.full((rows, 18), float("nan"), device="cuda") for _ in range(2)]
    grad = [torch.zeros(M.N_PARAMS, device="cuda") for _ in range(2)]
    loss = [torch.zeros(1, device="cuda") for _ in range(2)]
    for i, v in enumerate((x, xo)):
        t.mlp_forward_tc(w, v, out[i])
        t.mlp_loss_grad(w, v, _cuda(y), grad[i], loss[i], tensor_cores=True)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(out[0]).all()) and bool(torch.isfinite(grad[0]).all())
    assert torch.equal(out[0], out[1]) and torch.equal(grad[0], grad[1]) and torch.equal(loss[0], loss[1])
    assert t.stats()["tensor_timeouts"] == 0
