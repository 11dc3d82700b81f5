"""Mixed meshes whose offsets are wrong in such a way that the valid elements
overlap and have more incidences than the connectivity has entries, which is
what records, scratch and results are sized by.  The build reports them and
writes nothing outside its buffers: canaries after the outputs and after the
workspace, in the ordinary and the bounds-checked library, without and with a
partition."""
import ctypes as C

import numpy as np
import pytest

from paper_1604_04689_gb300 import nn
from tests.gpu_util import env

pytestmark = pytest.mark.gpu

CANARY = 0x5A5A5A5A
TAIL = 256  # canary words after each buffer
MESHES = {  # connectivity entries, elements, nodes, distance of the hexes' starts (0: anywhere)
    "one_hex": (16, 16, 40, 0), "few": (1528, 1500, 337, 0), "same_place": (4000, 4000, 200, 8000),
    "windows": (6000, 6000, 5000, 1), "limit": (1 << 15, 1 << 15, 20000, 0),
}


@pytest.fixture(scope="module", params=["ordinary", "checked"])
def lib(request):
    from paper_1604_04689_gb300 import build
    path = build.build(checked=request.param == "checked")
    L = C.CDLL(path)
    P = C.c_void_p
    L.nn_create.argtypes = [C.POINTER(P)]
    L.nn_destroy.argtypes = [P]
    L.nn_query.argtypes = [P, P, C.c_int, C.POINTER(C.c_size_t), C.POINTER(C.c_int64), C.POINTER(C.c_int64)]
    L.nn_neighbors_both.argtypes = [P, P, P, P, P, C.c_size_t, P, P]
    return L


def overlapping(n_conn, n_elems, n_nodes, step):
    """Every other element is a hex at some place, the ones between run backwards."""
    rng = np.random.default_rng(n_conn + step)
    k = n_elems // 2 + 1
    at = rng.integers(0, n_conn - 7, k) if step == 0 else (np.arange(k) * step) % (n_conn - 7)
    ptr = np.stack((at, at + 8), 1).reshape(-1)[: n_elems + 1].astype(np.int64)
    valid = int((ptr[1:] - ptr[:-1] == 8).sum())
    assert 8 * valid > n_conn, "the valid elements have to have more incidences than the connectivity"
    return rng.integers(0, n_nodes, n_conn).astype(np.int32), ptr, np.full(n_elems, nn.HEX, np.uint8)


@pytest.mark.parametrize("name", MESHES)
@pytest.mark.parametrize("part", ["auto", "sorted"])
def test_overlapping_elements_stay_in_bounds(lib, name, part):
    import torch
    n_conn, n_elems, n_nodes, _ = MESHES[name]
    conn, ptr, etype = (torch.from_numpy(x).cuda() for x in overlapping(*MESHES[name]))
    ms = nn.NNMesh(nn.MIXED, n_nodes, n_elems, n_conn, conn.data_ptr(), ptr.data_ptr(), etype.data_ptr())
    h = C.c_void_p()
    with env(NN_PART=part):
        assert lib.nn_create(C.byref(h)) == 0
    try:
        ws_bytes, ncap, ecap = C.c_size_t(), C.c_int64(), C.c_int64()
        assert lib.nn_query(h, C.byref(ms), nn.WANT_BOTH, C.byref(ws_bytes), C.byref(ncap), C.byref(ecap)) == 0
        words = {"ws": (ws_bytes.value + 3) // 4, "rp_n": 2 * (n_nodes + 1), "col_n": ncap.value,
                 "rp_e": 2 * (n_nodes + 1), "col_e": ecap.value}
        buf = {k: torch.full((n + TAIL,), CANARY, dtype=torch.int32, device="cuda") for k, n in words.items()}
        nodes = nn.NNCSR(buf["rp_n"].data_ptr(), buf["col_n"].data_ptr(), ncap.value)
        elems = nn.NNCSR(buf["rp_e"].data_ptr(), buf["col_e"].data_ptr(), ecap.value)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        assert lib.nn_neighbors_both(h, C.byref(ms), C.byref(nodes), C.byref(elems), buf["ws"].data_ptr(),
                                     ws_bytes.value, status.data_ptr(), None) == 0
        torch.cuda.synchronize()
        assert int(status.item()) in (2, 5)  # workspace too small for the records, offsets inconsistent
        for k, n in words.items():
            assert bool((buf[k][n:] == CANARY).all()), k
    finally:
        lib.nn_destroy(h)
