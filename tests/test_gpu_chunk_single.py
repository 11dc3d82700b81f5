"""A chunked build whose only chunk is the whole mesh: small meshes, which are
built without a partition, with more than 512 groups of 32 nodes, so that a scan
over the groups would have several tiles.  The workspace starts out full of
set bits and is used again for another mesh of the same shape.  Bit for bit
against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn
from tests.gpu_util import assert_same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1604_04689_gb300 import build
    build.build()


def apart(etype, n, nodes, seed):
    """n elements that share no node, over `nodes` nodes."""
    k = n * mg.NPE[etype]
    assert k <= nodes
    return mg.Mesh(etype, nodes, np.random.default_rng(seed).permutation(nodes)[:k].astype(np.int32))


def few(etype, n, nodes, seed):
    return mg.Mesh(etype, nodes, np.random.default_rng(seed).integers(0, nodes, n * mg.NPE[etype]).astype(np.int32))


SHAPES = {
    "quads": lambda s: mg.quad_grid(129, s),   # 521 groups
    "triangles_apart": lambda s: apart(mg.TRI, 10000, 30000, s),
    "tets": lambda s: few(mg.TET, 10000, 20000, s),
    "sparse": lambda s: few(mg.TRI, 5000, 38912, s),
    "grid": lambda s: mg.tri_grid(64, s),            # one tile
    "partitioned": lambda s: mg.tri_grid(200, s),    # beyond the direct builds
}


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("want", [nn.WANT_BOTH, nn.WANT_NODES, nn.WANT_ELEMS])
def test_one_chunk_in_a_used_workspace(shape, want):
    import torch
    b = nn.Builder()
    meshes = [SHAPES[shape](seed) for seed in (1, 2)]
    whole = b.query(nn.DeviceMesh.from_host(meshes[0]), want)[0] + 256
    ws = torch.full((whole,), 0xA5, dtype=torch.uint8, device="cuda")
    for m in meshes:
        dm = nn.DeviceMesh.from_host(m)
        out = b.alloc_outputs(dm, want)
        assert b.launch_chunked(dm, want, out, [(0, m.n_nodes, m.conn.size)], ws, whole) == 0
        torch.cuda.synchronize()
        res = {"status": int(b.status.item())}
        for k, (rp, col) in out.items():
            res[k] = (rp.cpu().numpy(), col.cpu().numpy()[: int(rp[-1])])
        assert_same(res, oracle.neighbors(m, want), want)


@pytest.mark.parametrize("records", [9999, 15000])  # partitioned (fewer than elements), direct
def test_one_chunk_of_too_few_records_is_reported(records):
    import torch
    b, m = nn.Builder(), SHAPES["triangles_apart"](3)
    dm = nn.DeviceMesh.from_host(m)
    ws = torch.full((b.query(dm, nn.WANT_BOTH)[0] + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    out = b.alloc_outputs(dm, nn.WANT_BOTH)
    assert b.launch_chunked(dm, nn.WANT_BOTH, out, [(0, m.n_nodes, records)], ws, ws.numel()) == 0
    torch.cuda.synchronize()
    assert int(b.status.item()) == 2
