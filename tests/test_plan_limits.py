"""Sizes a plan has to take (no GPU): as many nodes as 32-bit ids allow, with
every result and type, as long as a record's fields fit 128 bits."""
import pytest

from paper_1604_04689_gb300 import nn

FAKE = 1 << 20  # 16-byte aligned, never read


@pytest.fixture(scope="module")
def h():
    from paper_1604_04689_gb300 import build
    build.build()
    handle = nn.nn_create_offline()
    yield handle
    nn.nn_destroy(handle)


@pytest.mark.parametrize("n_nodes", [1 << 28, (1 << 28) + 1, 1 << 30, (1 << 30) + 1, 1500000000, (1 << 31) - 2])
@pytest.mark.parametrize("etype,npe", [(nn.TRI, 3), (nn.QUAD, 4), (nn.TET, 4), (nn.HEX, 8), (nn.MIXED, 6)])
@pytest.mark.parametrize("want", [nn.WANT_NODES, nn.WANT_ELEMS, nn.WANT_BOTH])
@pytest.mark.parametrize("share", [0.0, 0.01, 0.2])
def test_very_many_nodes(h, n_nodes, etype, npe, want, share):
    n = int(n_nodes * share / npe)
    tables = FAKE if etype == nn.MIXED else None
    m = nn.NNMesh(etype, n_nodes, n, n * npe, FAKE if n else None, tables, tables)
    k = (2 if etype in (nn.TRI, nn.QUAD) else 3) if want & nn.WANT_NODES else 0
    fixed = k * n_nodes.bit_length() + (1 + max(1, (n - 1).bit_length()) if want & nn.WANT_ELEMS else 0)
    if fixed + 11 > 128:  # the widest place in a bucket does not fit beside the ids
        pytest.skip("no record format")
    nn.nn_query(h, m, want)
    info = nn.nn_plan_info(h, m, want)
    assert info["n_buckets"] <= 1 << 20 and info["n_buckets"] << info["sb"] >= n_nodes
