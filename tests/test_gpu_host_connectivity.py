"""Small meshes whose connectivity stays in pinned host memory, built as one
chunk: results against the oracle, in the planned workspace and in the smallest
one, and the time against that of the same mesh on the device, partitioned."""
import numpy as np
import pytest

import oracle
from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn
from tests.gpu_util import assert_same, env

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1604_04689_gb300 import build
    build.build()


MESHES = {"tri": lambda: mg.tri_grid(64, 1), "tri_large": lambda: mg.tri_grid(104, 2), "quad": lambda: mg.quad_grid(129, 3),
          "tet": lambda: mg.tet_grid(13, 4), "hex": lambda: mg.hex_grid(20, 5), "mixed": lambda: mg.mixed_grid(13, 6)}


def pinned(m):
    import torch
    t = [None if x is None else torch.from_numpy(x).pin_memory() for x in (m.conn, m.elem_ptr, m.elem_type)]
    return nn.DeviceMesh(int(m.etype), m.n_nodes, *t)


def launcher(b, dm, out, ws, m):
    chunks = [(0, m.n_nodes, m.conn.size)]
    return lambda: b.launch_chunked(dm, nn.WANT_BOTH, out, chunks, ws, ws.numel())


@pytest.mark.parametrize("spill", [True, False])
@pytest.mark.parametrize("name", MESHES)
def test_pinned_connectivity_in_one_chunk(name, spill):
    import torch
    m, b = MESHES[name](), nn.Builder()
    dm = pinned(m)
    out = b.alloc_outputs(nn.DeviceMesh.from_host(m), nn.WANT_BOTH)
    n = b.query(dm, nn.WANT_BOTH)[0] if spill else nn.nn_plan_info(b.h, dm.struct(), nn.WANT_BOTH)["ws_min"]
    ws = torch.full((n + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        assert launcher(b, dm, out, ws, m)() == 0
    torch.cuda.synchronize()
    res = {"status": int(b.status.item())}
    for k, (rp, col) in out.items():
        res[k] = (rp.cpu().numpy(), col.cpu().numpy()[: int(rp[-1])])
    assert_same(res, oracle.neighbors(m))


@pytest.mark.parametrize("name", ["tri_large", "hex"])
def test_pinned_connectivity_is_not_read_by_every_bucket(name):
    """6,859 hexes took five times the partitioned build's time so."""
    import torch
    m, times = MESHES[name](), []
    for part, where in (("auto", pinned), ("sorted", nn.DeviceMesh.from_host)):
        with env(NN_PART=part):
            b = nn.Builder()
        dm = where(m)
        out = b.alloc_outputs(nn.DeviceMesh.from_host(m), nn.WANT_BOTH)
        ws = torch.empty(b.query(dm, nn.WANT_BOTH)[0] + 256, dtype=torch.uint8, device="cuda")
        f = launcher(b, dm, out, ws, m)
        t = []
        for _ in range(8):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                assert f() == 0
            z.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(z))
        times.append(min(t))
    assert times[0] < 2 * times[1], times
