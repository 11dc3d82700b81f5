"""Small meshes, built without a partition: every type and result, sizes around
the bucket edges and the limit of the rule, nodes of very many records (the
queue emptied several times, buckets built by the whole CTA), repeated nodes
and refused meshes.  Bit for bit against the oracle, on the direct path and on
the partitioned one."""
import numpy as np
import pytest

import oracle
from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn
from tests.gpu_util import assert_same, check_against_oracle, env, gpu_build

pytestmark = pytest.mark.gpu

LIMIT = 1 << 16  # incidences up to which a mesh is built directly


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1604_04689_gb300 import build
    build.build()


def cut(mesh, n_elems):
    return mg.Mesh(mesh.etype, mesh.n_nodes, mesh.conn[: n_elems * mg.NPE[mesh.etype]].copy())


def fan(n, extra=0):
    """n triangles around node 0, over n + 1 nodes and `extra` unused ones."""
    k = np.arange(n, dtype=np.int32)
    conn = np.stack((np.zeros(n, np.int32), 1 + k, 1 + (k + 1) % n), 1)
    return mg.Mesh(mg.TRI, n + 1 + extra, np.ascontiguousarray(conn.reshape(-1)))


def hub_tets(n, nodes, seed):
    """n tets that share node 0, the other nodes at random (some repeat)."""
    rng = np.random.default_rng(seed)
    conn = rng.integers(0, nodes, (n, 4)).astype(np.int32)
    conn[:, 0] = 0
    return mg.Mesh(mg.TET, nodes, np.ascontiguousarray(conn.reshape(-1)))


MESHES = {
    "tri2": lambda: mg.tri_grid(2, 1), "tri33": lambda: mg.tri_grid(33, 2), "tri64": lambda: mg.tri_grid(64, 3),
    "tri104": lambda: mg.tri_grid(104, 4),
    "quad91": lambda: mg.quad_grid(91, 5), "tet5": lambda: mg.tet_grid(5, 6), "tet14": lambda: mg.tet_grid(14, 7),
    "hex9": lambda: mg.hex_grid(9, 8), "hex21": lambda: mg.hex_grid(21, 9), "mixed6": lambda: mg.mixed_grid(6, 10),
    "mixed14": lambda: mg.mixed_grid(14, 11), "holes": lambda: mg.tri_grid(100, 12, holes=0.2),
    "limit": lambda: cut(mg.tri_grid(106, 13), LIMIT // 3), "over": lambda: cut(mg.tri_grid(106, 13), LIMIT // 3 + 1),
    "fan": lambda: fan(700, 5), "fan_long": lambda: fan(21000), "hub": lambda: hub_tets(9000, 500, 14),
    "hub_few": lambda: hub_tets(60, 40, 15), "no_elements": lambda: mg.Mesh(mg.HEX, 100, np.zeros(0, np.int32)),
}


@pytest.mark.parametrize("name", MESHES)
@pytest.mark.parametrize("want", [nn.WANT_BOTH, nn.WANT_NODES, nn.WANT_ELEMS])
def test_both_paths_match_oracle(name, want):
    mesh = MESHES[name]()
    res = check_against_oracle(mesh, want)
    with env(NN_PART="sorted"):
        assert_same(gpu_build(mesh, want, nn.Builder()), dict(res, status=0), want)


def test_large_node_numbers_of_few_elements():
    # many nodes, few elements: buckets of 256 nodes for one SM each, and more than that
    for n_nodes in (38911, 38912, 38913, 65536, 65537, 200000):
        m = mg.tet_grid(8, 16)
        conn = (m.conn.astype(np.int64) * (n_nodes // m.n_nodes)).astype(np.int32)
        check_against_oracle(mg.Mesh(mg.TET, n_nodes, conn))


@pytest.mark.parametrize("bad", [-1, 1089])
def test_node_out_of_range_is_reported(bad):
    m = mg.tri_grid(33, 2)
    conn = m.conn.copy()
    conn[77] = bad
    assert gpu_build(mg.Mesh(mg.TRI, m.n_nodes, conn))["status"] == oracle.neighbors(
        mg.Mesh(mg.TRI, m.n_nodes, conn))["status"] != 0


def test_overlapping_mixed_elements_are_reported():
    # every element starts at the same place: more incidences than connectivity
    m = mg.mixed_grid(6, 10)
    ptr = m.elem_ptr.copy()
    etype = np.full(m.n_elems, mg.HEX, np.uint8)
    ptr[:] = np.where(np.arange(ptr.size) % 2, 8, 0)
    bad = mg.Mesh(mg.MIXED, m.n_nodes, m.conn, ptr, etype)
    assert gpu_build(bad)["status"] != 0


def test_workspace_of_the_minimum_size():
    # no spill area: an ordinary mesh builds, a hub whose bucket needs one is refused on the device
    b = nn.Builder()
    for mesh, ok in ((mg.tet_grid(12, 17), True), (fan(5000), False)):
        dm = nn.DeviceMesh.from_host(mesh)
        out = b.alloc_outputs(dm, nn.WANT_BOTH)
        n = nn.nn_plan_info(b.h, dm.struct(), nn.WANT_BOTH)["ws_min"]
        assert b.launch(dm, nn.WANT_BOTH, out, ws=b.workspace(n), ws_bytes=n) == 0
        assert (int(b.status.item()) == 0) == ok
