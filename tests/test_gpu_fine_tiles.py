"""The fine partition pass by buckets per coarse region: below 512 (256
threads), 512 and above (512 threads, several digits a thread), with records of
8 and 16 bytes.  Few elements over many node ids, so that regions are small and
tiles are partly filled, and one dense mesh of several tiles a region."""
import numpy as np
import pytest

from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn
from tests.gpu_util import check_against_oracle, env

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1604_04689_gb300 import build
    build.build()


@pytest.mark.parametrize("want", [nn.WANT_BOTH, nn.WANT_ELEMS])
@pytest.mark.parametrize("shift", [1, 6, 8, 9, 10])
def test_regions_of_every_width(shift, want):
    # buckets of 16 nodes, 200 regions of 2^shift buckets; every region's first and last bucket is used
    n_nodes = 16 * 200 << shift
    rng = np.random.default_rng(shift)
    conn = rng.integers(0, n_nodes, (6000, 4)).astype(np.int32)
    conn[:200, 0] = (16 << shift) * np.arange(200)
    conn[:200, 1] = (16 << shift) * np.arange(1, 201) - 1
    mesh = mg.Mesh(mg.TET, n_nodes, np.ascontiguousarray(conn.reshape(-1)))
    with env(NN_SB=4, NN_PART="sorted"):
        b = nn.Builder()
        dm = nn.DeviceMesh.from_host(mesh)
        plan = nn.nn_plan_info(b.h, dm.struct(), want)
        assert plan["partition"] == shift and plan["record_bytes"] == (16 if want == nn.WANT_BOTH and shift > 1 else 8)
        check_against_oracle(mesh, want, b)


def test_several_tiles_a_region():
    # 2,197 nodes of a tet grid in the middle of 2 M: their region's records fill more than one tile
    m = mg.tet_grid(13, 3)
    mesh = mg.Mesh(mg.TET, 1 << 21, (m.conn + 1000000).astype(np.int32))
    with env(NN_SB=4, NN_PART="sorted"):
        b = nn.Builder()
        assert nn.nn_plan_info(b.h, nn.DeviceMesh.from_host(mesh).struct(), nn.WANT_BOTH)["partition"] == 9
        check_against_oracle(mesh, nn.WANT_BOTH, b)
