"""Element face adjacency of one-type meshes, matched node by node: small
groups of elements over few shared nodes, so that faces border several
elements, lie in an element without being one of its faces, or repeat a
node; node rows below, at and above the lanes of a group and past the longest
matched row.  Bit for bit against the oracle, with and without room for the
matching pass in the workspace."""
import numpy as np
import pytest

import oracle
from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1604_04689_gb300 import build
    build.build()


def groups(etype, n_groups, nodes, elems, repeat, seed):
    """n_groups disjoint groups of `elems` random elements over `nodes` nodes; a share `repeat` of them repeats a node."""
    rng = np.random.default_rng(seed)
    el = []
    for g in range(n_groups):
        for _ in range(elems):
            nd = rng.permutation(nodes)[: mg.NPE[etype]]
            if rng.random() < repeat:
                nd[rng.integers(0, nd.size)] = nd[rng.integers(0, nd.size)]
            el.append((etype, tuple(int(x) for x in nd + g * nodes)))
    order = rng.permutation(len(el))
    return mg.from_elements([el[i] for i in order], n_groups * nodes)


CASES = [(t, n, e, r) for t, extra in ((mg.TRI, 2), (mg.QUAD, 1), (mg.TET, 2), (mg.HEX, 2))
         for n in (mg.NPE[t], mg.NPE[t] + extra) for e, r in ((2, 0.0), (6, 0.0), (9, 0.05), (33, 0.02), (70, 0.0))]


@pytest.mark.parametrize("etype,nodes,elems,repeat", CASES)
def test_groups_match_oracle(etype, nodes, elems, repeat):
    import torch
    mesh = groups(etype, 41, nodes, elems, repeat, 1000 * etype + 10 * nodes + elems)
    ref = oracle.element_adjacency(mesh)["adj"]
    b = nn.Builder()
    dm = nn.DeviceMesh.from_host(mesh)
    res = b.build(dm, nn.WANT_ELEMS)
    assert res["status"] == 0
    rp, col = b.element_neighbors(dm, res["elems"])
    np.testing.assert_array_equal(rp.cpu().numpy(), ref[0])
    np.testing.assert_array_equal(col.cpu().numpy(), ref[1])
    # a workspace with the counts and the scan alone: the merge of every element's node rows
    T, up = mesh.n_elems, lambda x: -(-x // 256) * 256
    ws_bytes = up(4 * T) + up(8 * ((T + 127) // 128 + 1)) + 256
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    rp2, col2 = torch.empty_like(rp), torch.empty(max(len(ref[1]), 1), dtype=torch.int32, device="cuda")
    ne_rp, ne_col = res["elems"]
    assert nn.nn_element_neighbors(b.h, dm.struct(), nn.NNCSR(ne_rp.data_ptr(), ne_col.data_ptr(), ne_col.numel()),
                                   nn.NNCSR(rp2.data_ptr(), col2.data_ptr(), col2.numel()), ws.data_ptr(), ws_bytes,
                                   b.status.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(b.status.item()) == 0
    np.testing.assert_array_equal(rp2.cpu().numpy(), ref[0])
    np.testing.assert_array_equal(col2.cpu().numpy()[: len(ref[1])], ref[1])


def test_boundary_cases_of_the_grids():
    # grids of every type whose last blocks and groups are partly filled
    for mesh in (mg.tri_grid(17, 3), mg.quad_grid(18, 4), mg.tet_grid(7, 5), mg.hex_grid(7, 6), mg.tri_grid(2, 1),
                 mg.hex_grid(2, 1)):
        b = nn.Builder()
        dm = nn.DeviceMesh.from_host(mesh)
        rp, col = b.element_neighbors(dm, b.build(dm, nn.WANT_ELEMS)["elems"])
        ref = oracle.element_adjacency(mesh)["adj"]
        np.testing.assert_array_equal(rp.cpu().numpy(), ref[0])
        np.testing.assert_array_equal(col.cpu().numpy(), ref[1])


@pytest.mark.parametrize("T", [1, 255, 1023, 1024, 1025, 2049])
def test_row_pass_tile_edges(T):
    # element counts around the row pass's tiles (1024 elements), every type
    for grid in (mg.tri_grid(41, 3), mg.quad_grid(60, 4), mg.tet_grid(9, 5), mg.hex_grid(15, 6)):
        mesh = mg.Mesh(grid.etype, grid.n_nodes, grid.conn[: T * mg.NPE[grid.etype]].copy())
        assert mesh.n_elems == T
        b = nn.Builder()
        dm = nn.DeviceMesh.from_host(mesh)
        rp, col = b.element_neighbors(dm, b.build(dm, nn.WANT_ELEMS)["elems"])
        ref = oracle.element_adjacency(mesh)["adj"]
        np.testing.assert_array_equal(rp.cpu().numpy(), ref[0])
        np.testing.assert_array_equal(col.cpu().numpy(), ref[1])
