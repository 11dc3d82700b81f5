"""Plans of small meshes (no GPU): a mesh built without a partition places its
node rows by sums, without the scan over the groups, whose lookback words such
a build does not clear."""
import itertools

import pytest

from paper_1604_04689_gb300 import nn

FAKE = 1 << 20  # 16-byte aligned, never read
TYPES = ((nn.TRI, 3), (nn.QUAD, 4), (nn.TET, 4), (nn.HEX, 8), (nn.MIXED, 6))


@pytest.fixture(scope="module")
def h():
    from paper_1604_04689_gb300 import build
    build.build()
    handle = nn.nn_create_offline()
    yield handle
    nn.nn_destroy(handle)


def struct(etype, n_nodes, n_elems, npe):
    tables = FAKE if etype == nn.MIXED else None
    return nn.NNMesh(etype, n_nodes, n_elems, n_elems * npe, FAKE, tables, tables)


@pytest.mark.parametrize("sb", [None] + list(range(4, 12)))
def test_direct_plans_have_no_scan(h, sb):
    """Kernels of a direct build: initialization, buckets, placement.  A
    partitioned one has at least five."""
    nn.nn_set_tuning(h, dict(sb=sb) if sb else None)
    seen = set()
    try:
        for (etype, npe), n_nodes, n_elems in itertools.product(
                TYPES, (1, 500, 4000, 16641, 38912, 131072, 140000, 155648, 311296), (1, 60, 5000, 8192)):
            for want, most in ((nn.WANT_NODES, 3), (nn.WANT_ELEMS, 2), (nn.WANT_BOTH, 3)):
                k = nn.nn_plan_info(h, struct(etype, n_nodes, n_elems, npe), want)["kernels"]
                assert k == most or k >= 5, (etype, n_nodes, n_elems, want, k)
                seen.add(k == most)
    finally:
        nn.nn_set_tuning(h, None)
    assert seen == {True, False}
