"""The triangle list where a bucket of first ids holds many rows."""
import numpy as np
import pytest

from tests.gpu_helpers import assert_same

pytestmark = pytest.mark.gpu


def _hubs(degrees, spread=1):
    """Rings with their centres, the centres having the lowest ids."""
    centres, rims = [], []
    for i, k in enumerate(degrees):
        a = 2 * np.pi * (np.arange(k) + 0.3) / k
        at = np.array([(i % 8) * 8000000 + 4000000, (i // 8) * 8000000 + 4000000])
        r = 3000000.0 + 7 * (np.arange(k) % 5)
        centres.append(at[None])
        rims.append(np.rint(np.stack([r * np.cos(a), r * np.sin(a)], 1)).astype(np.int64) + at)
    return np.ascontiguousarray(np.concatenate(centres + rims).astype(np.int32))


@pytest.mark.parametrize("degrees,buckets", [([40] * 16, True), ([40] * 40, True), ([700, 30, 600], True),
                                             ([1400], True), ([1700], False)])
def test_rows_of_large_stars(degrees, buckets):
    """Up to 1,536 rows a bucket the list takes its four launches, beyond it is placed."""
    import torch
    from paper_2308_06484_gb300 import kdt
    xy = _hubs(degrees)
    t = kdt.Triangulation(kdt.default_config(domain_bits=27))
    t.build(xy)
    out = torch.zeros((2 * len(xy), 3), dtype=torch.int32, device="cuda")
    before = t.stats()["kernel_launches"]
    got = t.export_triangles(out).cpu().numpy()
    assert (t.stats()["kernel_launches"] - before == 4) == buckets
    assert_same(got, xy, "stars of %s" % degrees)
    assert_same(t.export_triangles(), xy, "stars of %s, host" % degrees)
