"""The bucket pass at the edges of its slots, its list and its registers:
nodes whose record count lies just below, at and above the places a node has
in the shared-memory table, above the register arrays, and beyond what a
bucket's list holds; node counts off the group and bucket widths; every
selection of results.  Bit for bit against the oracle."""
import numpy as np
import pytest

from paper_1604_04689_gb300 import meshgen as mg
from paper_1604_04689_gb300 import nn
from tests.gpu_util import check_against_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1604_04689_gb300 import build
    build.build()


def joined(parts, seed):
    """Disjoint union of (type, element array) parts of one type, nodes and elements shuffled."""
    rng = np.random.default_rng(seed)
    el, base = [], 0
    for p in parts:
        el.append(p + base)
        base += int(p.max()) + 1
    el = np.concatenate(el)
    perm = rng.permutation(base)
    return perm[el][rng.permutation(len(el))].astype(np.int32), base


def fan(n):        # n triangles around node 0: n records, n neighbours
    k = np.arange(n)
    return np.stack([0 * k, 1 + k, 1 + (k + 1) % n], 1)


def cone(n):       # n quads at node 0, sharing edges: n records, n neighbours
    k = np.arange(n)
    return np.stack([0 * k, 1 + k, 1 + n + k, 1 + (k + 1) % n], 1)


def spindle(n):    # n tets around the edge 0-1: n records, n + 1 neighbours
    k = np.arange(n)
    return np.stack([0 * k, 0 * k + 1, 2 + k, 2 + (k + 1) % n], 1)


def tets(n):       # Kuhn grid: 24 records at inner nodes, so that the mean asks for many slots
    return mg.tet_grid(n, 0, permute_nodes=False, permute_elems=False).conn.reshape(-1, 4).astype(np.int64)


def hexes(n):      # unrelated hexes at node 0: n records, 3 n neighbours
    k = np.arange(n)[:, None]
    return np.concatenate([0 * k, 1 + 7 * k + np.arange(7)[None, :]], 1)


CASES = {
    # slots 8, registers 24 (22 neighbours fit a triangle's column)
    "fans_7_10": (mg.TRI, lambda: [fan(n) for n in (7, 8, 9, 10)] * 40),
    "fans_20_26": (mg.TRI, lambda: [fan(n) for n in (20, 21, 22, 23, 24, 25, 26)] * 7),
    "fans_40_400": (mg.TRI, lambda: [fan(n) for n in (40, 100, 400)] * 3),
    "fans_all_listed": (mg.TRI, lambda: [fan(16)] * 300),           # more listed records than a bucket's list holds
    "quads": (mg.QUAD, lambda: [cone(n) for n in (3, 4, 8, 9, 13, 22, 23, 24, 25)] * 9),
    "hexes": (mg.HEX, lambda: [hexes(n) for n in (6, 7, 8, 9, 10, 24, 25)] * 5),
    # slots 24, registers 64
    "tets_23_26": (mg.TET, lambda: [tets(9)] * 5 + [spindle(n) for n in (23, 24, 25, 26)] * 3),
    "tets_31_66": (mg.TET, lambda: [tets(9)] * 9 + [spindle(n) for n in (31, 32, 33, 48, 63, 64, 65, 66)]),
    "tets_200": (mg.TET, lambda: [tets(9)] * 9 + [spindle(200)]),
    # scattered valences
    "tri_soup": (mg.TRI, lambda: [np.random.default_rng(1).integers(0, 2003, (4000, 3))]),
    "tet_soup_20": (mg.TET, lambda: [np.random.default_rng(2).integers(0, 1501, (7500, 4))]),
    "tet_soup_9": (mg.TET, lambda: [np.random.default_rng(3).integers(0, 1501, (3400, 4))]),
    "hex_soup_12": (mg.HEX, lambda: [np.random.default_rng(4).integers(0, 1501, (2250, 8))]),
}


@pytest.mark.parametrize("want", [nn.WANT_BOTH, nn.WANT_NODES, nn.WANT_ELEMS])
@pytest.mark.parametrize("name", list(CASES))
def test_slots_lists_and_registers(name, want):
    etype, parts = CASES[name]
    conn, n = joined(parts(), len(name))
    check_against_oracle(mg.Mesh(etype, n + 5, conn.reshape(-1)), want, ws_extra=64 * conn.size)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 4097])
def test_node_counts_off_the_group_and_bucket_widths(n):
    k = np.arange(n + 1)
    conn = np.stack([k[:-1], k[1:] % n, (k[:-1] + 2) % n], 1).astype(np.int32)
    check_against_oracle(mg.Mesh(mg.TRI, n, conn.reshape(-1)), nn.WANT_BOTH)
