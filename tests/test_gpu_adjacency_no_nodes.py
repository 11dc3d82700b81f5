"""Element neighbours of meshes without nodes: every element is invalid, so all
rows are empty and the call succeeds."""
import pytest

from paper_1604_04689_gb300 import nn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("etype,npe", [(nn.TRI, 3), (nn.QUAD, 4), (nn.TET, 4), (nn.HEX, 8), (nn.MIXED, 8)])
@pytest.mark.parametrize("n", [1, 1500])
def test_elements_without_nodes(etype, npe, n):
    import torch
    from paper_1604_04689_gb300 import build
    build.build()
    b = nn.Builder()
    tables = (torch.arange(n + 1, device="cuda") * 8, torch.full((n,), nn.HEX, dtype=torch.uint8, device="cuda")) \
        if etype == nn.MIXED else (None, None)
    dm = nn.DeviceMesh(etype, 0, torch.zeros(npe * n, dtype=torch.int32, device="cuda"), *tables)
    ne_rp = torch.zeros(1, dtype=torch.int64, device="cuda")
    ne_col = torch.zeros(4, dtype=torch.int32, device="cuda")
    ws_bytes, _ = nn.nn_element_neighbors_query(b.h, dm.struct())
    ws = torch.full((ws_bytes,), 0xA5, dtype=torch.uint8, device="cuda")
    rp = torch.full((n + 1,), -1, dtype=torch.int64, device="cuda")
    col = torch.zeros(16, dtype=torch.int32, device="cuda")
    assert nn.nn_element_neighbors(b.h, dm.struct(), nn.NNCSR(ne_rp.data_ptr(), ne_col.data_ptr(), 4),
                                   nn.NNCSR(rp.data_ptr(), col.data_ptr(), 16), ws.data_ptr(), ws_bytes,
                                   b.status.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(b.status.item()) == 0 and bool((rp == 0).all()) and bool((col == 0).all())
