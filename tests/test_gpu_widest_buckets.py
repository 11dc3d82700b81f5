"""Buckets of 2048 nodes, four slots each (what meshes of more than 2^30 nodes
are built with): every type and result on ordinary meshes, against the oracle;
and one mesh of more than 2^30 nodes, whose results are known in closed form."""
import numpy as np
import pytest

from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn
from tests.gpu_util import check_against_oracle

pytestmark = pytest.mark.gpu

MESHES = {
    "tri": lambda: mg.tri_grid(130, 1), "tri_holes": lambda: mg.tri_grid(201, 2, holes=0.2),
    "quad": lambda: mg.quad_grid(129, 3), "tet": lambda: mg.tet_grid(20, 4), "hex": lambda: mg.hex_grid(25, 5),
    "mixed": lambda: mg.mixed_grid(15, 6),
    "pairs": lambda: mg.Mesh(mg.TRI, 40000, np.random.default_rng(7).integers(0, 40000, 30000).astype(np.int32)),
}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1604_04689_gb300 import build
    build.build()


@pytest.mark.parametrize("name", MESHES)
@pytest.mark.parametrize("want", [nn.WANT_BOTH, nn.WANT_NODES, nn.WANT_ELEMS])
def test_widest_buckets(name, want):
    b = nn.Builder()
    nn.nn_set_tuning(b.h, dict(sb=11))
    m = MESHES[name]()
    assert nn.nn_plan_info(b.h, nn.DeviceMesh.from_host(m).struct(), want)["sb"] == 11
    check_against_oracle(m, want, b)


def test_more_than_2_30_nodes():
    import torch
    N = (1 << 30) + 5
    if torch.cuda.mem_get_info()[0] < 64 << 30:
        pytest.skip("needs 64 GB of device memory")
    # 100,000 triangles (a, a + 1, a + 2) apart from each other, up to the last node
    T, step = 100000, (N - 3) // 99999
    a = torch.arange(T, device="cuda", dtype=torch.int64) * step
    a[-1] = N - 3
    conn = torch.stack((a, a + 1, a + 2), 1).reshape(-1).to(torch.int32)
    b, dm = nn.Builder(), nn.DeviceMesh(nn.TRI, N, conn, None, None)
    res = b.build(dm, nn.WANT_BOTH)
    assert res["status"] == 0
    b.ws = None
    for key, per in (("nodes", 2), ("elems", 1)):
        rp, col = res[key]
        deg = rp[1:] - rp[:-1]
        assert int(rp[0]) == 0 and int(rp[-1]) == 3 * T * per == col.numel()
        assert torch.equal(torch.nonzero(deg)[:, 0], conn.long()) and bool((deg[conn.long()] == per).all())
        del deg
        v = torch.stack((a, a + 1, a + 2), 1)
        want = torch.stack((v[:, [1, 2]], v[:, [0, 2]], v[:, [0, 1]]), 1).reshape(-1) if key == "nodes" else \
            torch.arange(T, device="cuda").repeat_interleave(3)
        assert torch.equal(col.long(), want)
