"""Few elements over very many nodes with a tuning of wide buckets: more groups
of 32 nodes than the placement sums up, in a workspace full of set bits.  Bit
for bit against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn
from tests.gpu_util import assert_same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("want", [nn.WANT_NODES, nn.WANT_BOTH])
@pytest.mark.parametrize("n_nodes", [131072, 131073, 140000, 155648])
def test_wide_buckets_of_few_elements(n_nodes, want):
    import torch
    from paper_1604_04689_gb300 import build
    build.build()
    b = nn.Builder()
    nn.nn_set_tuning(b.h, dict(sb=10))
    ws = None
    for seed in (1, 2):
        m = mg.Mesh(mg.TRI, n_nodes, np.random.default_rng(seed).integers(0, n_nodes, 15000).astype(np.int32))
        dm = nn.DeviceMesh.from_host(m)
        out = b.alloc_outputs(dm, want)
        if ws is None:
            ws = torch.full((b.query(dm, want)[0],), 0xA5, dtype=torch.uint8, device="cuda")
        assert b.launch(dm, want, out, ws=ws, ws_bytes=ws.numel()) == 0
        torch.cuda.synchronize()
        res = {"status": int(b.status.item())}
        for k, (rp, col) in out.items():
            res[k] = (rp.cpu().numpy(), col.cpu().numpy()[: int(rp[-1])])
        assert_same(res, oracle.neighbors(m, want), want)
