"""Timed workloads of the library: what a mesh program has it do, through its public entry points.

A case is one call on seeded synthetic grids (the mesh families of the
repository's generator: triangle grids with a random diagonal per quad, quad,
Kuhn-split tet, hex and hex/tet mixed grids), made on the GPU from the seed
alone.  ``op`` names the call:

* ``launch``  Builder.launch: a program that keeps its workspace and its
  output buffers (sized by the library's own bounds) and builds again and again;
* ``build``   Builder.build: the one-call form, which allocates, waits and trims;
* ``chunked`` Builder.launch_chunked: a workspace of a fraction of the whole
  build's, the chunks planned beforehand;
* ``adj``     Builder.element_neighbors: face neighbours of every element;
* ``batch``   nn_batch_submit: many uneven meshes in one call.

``order`` is the numbering: ``random`` relabels the nodes by a random
permutation (and reorders the elements, except for hex and mixed grids, which
keep their cell order), ``natural`` keeps the row-by-row numbering of a
structured mesh; node ids and element lists that keep their order start at a
random place of it.  ``holes`` deletes that share of
the triangles, at random places.
"""
import math

import torch

from paper_1604_04689_gb300 import nn

TYPE = {"tri": nn.TRI, "quad": nn.QUAD, "tet": nn.TET, "hex": nn.HEX, "mixed": nn.MIXED}
WANT = {"nodes": nn.WANT_NODES, "elems": nn.WANT_ELEMS, "both": nn.WANT_BOTH}
NPE = {"tri": 3, "quad": 4, "tet": 4, "hex": 8}
SPLIT = 0.30  # share of a mixed grid's cells that are split into six tets
# Kuhn split of a VTK-ordered hex: six tets around the 0-6 diagonal
KUHN = ((0, 1, 2, 6), (0, 1, 5, 6), (0, 3, 2, 6), (0, 3, 7, 6), (0, 4, 5, 6), (0, 4, 7, 6))
# edge neighbours of each local node, for exact() alone
NBRS = {"tri": ((1, 2), (2, 0), (0, 1)),
        "quad": ((1, 3), (2, 0), (3, 1), (0, 2)),
        "tet": ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2)),
        "hex": ((1, 3, 4), (0, 2, 5), (1, 3, 6), (0, 2, 7), (0, 5, 7), (1, 4, 6), (2, 5, 7), (3, 4, 6))}
FACES = {"tri": ((0, 1), (1, 2), (2, 0)),
         "quad": ((0, 1), (1, 2), (2, 3), (3, 0)),
         "tet": ((0, 1, 2), (0, 1, 3), (0, 2, 3), (1, 2, 3)),
         "hex": ((0, 1, 2, 3), (4, 5, 6, 7), (0, 1, 5, 4), (1, 2, 6, 5), (2, 3, 7, 6), (3, 0, 4, 7))}


def _case(op, mesh, n, want="both", order="random", **more):
    return dict(op=op, mesh=mesh, n=n, want=want, order=order, **more)


def listed():
    return [
        # the smallest configured mesh (7,938 triangles): launches and latency are all of it
        dict(_case("launch", "tri", 64), name="tri64"),
        # a small one-off request, as a script makes it: buffers allocated, result waited for and trimmed
        dict(_case("build", "hex", 21), name="hex21_build"),
        # a scanned surface of the usual size (1.76 M triangles, the paper's largest scan)
        dict(_case("launch", "tri", 939), name="tri939"),
        # node rows alone, of a structured quad mesh in its natural numbering (odd sides)
        dict(_case("launch", "quad", 1001, want="nodes", order="natural"), name="quad1001_nodes_natural"),
        # the large surface with holes: ragged valences, a triangle count that is no multiple of anything
        dict(_case("launch", "tri", 2048, holes=0.05), name="tri2048_holes"),
        # element rows alone (a vertex-to-cell map for finite elements), 6 M tets
        dict(_case("launch", "tet", 101, want="elems"), name="tet101_elems"),
        # a large tet volume, 24.6 M tets: long rows, many repeated neighbours
        dict(_case("launch", "tet", 161), name="tet161"),
        # the headline workload: 16.8 M hexes, both results
        dict(_case("launch", "hex", 257), name="hex257"),
        # the largest call: hexes and tets in one mesh, per-element types and offsets
        dict(_case("launch", "mixed", 257), name="mixed257"),
        # a workspace capped at a quarter of the whole build's
        dict(_case("chunked", "tet", 101, frac=0.25), name="tet101_chunked"),
        # the dual graph of a tet mesh, as partitioners and flux loops want it
        dict(_case("adj", "tet", 101), name="tet101_adj"),
        # a serving batch: 24 uneven requests (1e3 to 5e5 elements, tri / tet / hex) in one call
        dict(op="batch", meshes=24, lo=1e3, hi=5e5, want="both", order="random", name="batch24"),
    ]


def _side(mesh, elems):
    """Nodes per side of the grid whose element count is nearest to `elems` (2 at least)."""
    m = {"tri": (elems / 2) ** 0.5, "quad": elems ** 0.5, "tet": (elems / 6) ** (1 / 3), "hex": elems ** (1 / 3),
         "mixed": (elems / 2.5) ** (1 / 3)}[mesh]
    return max(2, int(round(m)) + 1)


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    op = rng.choices(("launch", "build", "chunked", "adj", "batch"), (10, 3, 1, 2, 2))[0]
    if op == "batch":
        return dict(op="batch", meshes=rng.randint(3, 40), lo=1e3, hi=log(1e4, 5e5),
                    want=rng.choice(("both", "both", "nodes", "elems")), order="random")
    # (the trimmed results of mixed grids and of grids with holes are of no size known beforehand)
    trimmed = op in ("build", "adj")
    mesh = rng.choice(("tri", "tri", "quad", "tet", "tet", "hex", "hex") + ((), ("mixed",))[not trimmed])
    want = "elems" if op == "adj" else rng.choice(("both", "both", "both", "nodes", "elems"))
    order = rng.choice(("random", "random", "random", "natural"))
    # up to the listed sizes of each family; adjacency and chunked builds up to 6 M tets' work
    most = {"tri": 8.3e6, "quad": 8.3e6, "tet": 2.4e7, "hex": 1.6e7, "mixed": 4.1e7}
    if op != "launch":
        most = {"tri": 8.3e6, "quad": 4e6, "tet": 5.9e6, "hex": 2e6, "mixed": 2e6}
    lo = 1e6 if op == "chunked" else 1e3  # (a fraction of a small workspace is below its fixed part)
    case = _case(op, mesh, _side(mesh, log(lo, most[mesh])), want, order)
    if mesh == "tri" and not trimmed and rng.random() < 0.5:
        case["holes"] = round(rng.uniform(0.01, 0.3), 3)
    if op == "chunked":
        case["frac"] = rng.choice((0.25, 0.5))
    return draw(rng) if any(dict(case, name=c["name"]) == c for c in listed()) else case


# ------------------------------------------------------------------ inputs

def _cells(n):
    """VTK-ordered cells of an n^3 node grid, cell by cell (node (i, j, k) is i + n j + n n k)."""
    r = torch.arange(n - 1, device="cuda")
    base = (r[None, None, :] + n * r[None, :, None] + n * n * r[:, None, None]).reshape(-1, 1)
    return base + torch.tensor([0, 1, 1 + n, n, n * n, n * n + 1, n * n + 1 + n, n * n + n], device="cuda")


def _mesh(mesh, n, order, holes, g):
    """(number of nodes, {type: (element ids, nodes [.., npe])}, conn, elem_ptr, elem_type) of one grid."""
    if mesh in ("tri", "quad"):
        N, r = n * n, torch.arange(n - 1, device="cuda")
        a = (r[None, :] + n * r[:, None]).reshape(-1)
        b, c, d = a + 1, a + 1 + n, a + n
        if mesh == "quad":
            el = torch.stack((a, b, c, d), 1)
        else:
            bit = torch.rand(a.numel(), device="cuda", generator=g) < 0.5
            el = torch.stack((torch.stack((a, b, torch.where(bit, d, c)), 1),
                              torch.stack((torch.where(bit, b, a), c, d), 1)), 1).reshape(-1, 3)
            if holes:
                T = el.shape[0]
                el = el[torch.randperm(T, device="cuda", generator=g)[int(T * holes):].sort().values]
    else:
        N, el = n ** 3, _cells(n)
        if mesh == "tet":
            el = el[:, torch.tensor(KUHN, device="cuda")].reshape(-1, 4)
    if order == "natural":
        el = (el + torch.randint(N, (1,), device="cuda", generator=g)) % N
    else:
        pi = torch.randperm(N, device="cuda", generator=g)
        el = pi[el]
    if order == "random" and mesh in ("tri", "quad", "tet"):
        el = el[torch.randperm(el.shape[0], device="cuda", generator=g)]
    else:
        el = el.roll(int(torch.randint(el.shape[0], (1,), device="cuda", generator=g)), 0)
    el = el.to(torch.int32)
    if mesh != "mixed":
        return N, {mesh: (None, el)}, el.reshape(-1), None, None
    split = torch.zeros(el.shape[0], dtype=torch.bool, device="cuda")
    split[torch.randperm(el.shape[0], device="cuda", generator=g)[: int(el.shape[0] * SPLIT)]] = True
    first = torch.cumsum(torch.where(split, 6, 1), 0)  # elements up to and including each cell
    T = int(first[-1])
    first = first - torch.where(split, 6, 1)
    etype = torch.full((T,), nn.HEX, dtype=torch.uint8, device="cuda")
    tid = (first[split][:, None] + torch.arange(6, device="cuda")).reshape(-1)
    hid = first[~split]
    etype[tid] = nn.TET
    ptr = torch.zeros(T + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.where(etype == nn.TET, 4, 8), 0, out=ptr[1:])
    conn = torch.empty(int(ptr[-1]), dtype=torch.int32, device="cuda")
    hexes = el[~split]
    tets = el[split][:, torch.tensor(KUHN, device="cuda")].reshape(-1, 4)
    conn[(ptr[hid][:, None] + torch.arange(8, device="cuda")).reshape(-1)] = hexes.reshape(-1)
    conn[(ptr[tid][:, None] + torch.arange(4, device="cuda")).reshape(-1)] = tets.reshape(-1)
    return N, {"hex": (hid, hexes), "tet": (tid, tets)}, conn, ptr, etype


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _batch_specs(case):
    """(mesh, n) of the meshes of a batch: element counts spread evenly over the logarithm, types in turn."""
    q = case["hi"] / case["lo"]
    return [(m, _side(m, case["lo"] * q ** ((i + 0.5) / case["meshes"])))
            for i, m in ((i, ("tri", "tet", "hex")[i % 3]) for i in range(case["meshes"]))]


def _device_mesh(mesh, N, conn, ptr, etype):
    return nn.DeviceMesh(TYPE[mesh], N, conn.clone(), ptr, etype)


def _cap(mesh, n_conn, key):
    """The library's bound on a result's entries: the edge ends (or the incidences) of all elements."""
    return n_conn if key == "elems" else (2 if mesh in ("tri", "quad") else 3) * n_conn


def _pool(n):
    """Entries that a row takes in a batch's output pool (256-byte steps)."""
    return -(-n // 64) * 64


def _zeroed(out):
    for rp, col in out.values():
        rp.zero_()
        col.zero_()
    return out


def prepare(case, seed):
    g = _generator(seed)
    b, want = nn.Builder(), WANT[case["want"]]
    s = dict(case=case, b=b, want=want)
    if case["op"] == "batch":
        s["dms"] = [_device_mesh(m, *[x for i, x in enumerate(_mesh(m, n, case["order"], 0.0, g)) if i != 1])
                    for m, n in _batch_specs(case)]
        k = len(s["dms"])
        s["meshes"] = (nn.NNMesh * k)(*[d.struct() for d in s["dms"]])
        s["out"] = {}
        for key, flag in (("nodes", nn.WANT_NODES), ("elems", nn.WANT_ELEMS)):
            s[key] = None
            if want & flag:
                # one pool each for all meshes' row pointers and columns
                sizes = [(d.n_nodes + 1, _cap(m, d.n_conn, key)) for d, (m, _) in zip(s["dms"], _batch_specs(case))]
                rp, col = (torch.zeros(sum(_pool(z[i]) for z in sizes), dtype=t, device="cuda")
                           for i, t in ((0, torch.int64), (1, torch.int32)))
                s["out"][key], csrs, a, c = (rp, col), [], 0, 0
                for r, n in sizes:
                    csrs.append(nn.NNCSR(rp[a:].data_ptr(), col[c:].data_ptr(), n))
                    a, c = a + _pool(r), c + _pool(n)
                s[key] = (nn.NNCSR * k)(*csrs)
        s["ws_bytes"] = nn.nn_batch_submit_query(b.h, s["meshes"], k, want)
        s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda")
        s["status"] = torch.zeros(k, dtype=torch.int32, device="cuda")
        return s
    N, _, conn, ptr, etype = _mesh(case["mesh"], case["n"], case["order"], case.get("holes", 0.0), g)
    dm = s["dm"] = _device_mesh(case["mesh"], N, conn, ptr, etype)
    if case["op"] == "adj":
        s["node_elems"] = b.build(dm, nn.WANT_ELEMS)["elems"]
        b.ws = None  # the build's workspace is not needed any more
    elif case["op"] != "build":
        s["out"] = _zeroed(b.alloc_outputs(dm, want))
        s["ws_bytes"] = b.query(dm, want)[0]
        if case["op"] == "chunked":
            s["ws_bytes"] = int(s["ws_bytes"] * case["frac"])
            s["chunks"] = b.plan_chunks(dm, want, s["ws_bytes"])
        s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda")
    return s


def run(state):
    s, b = state, state["b"]
    op = s["case"]["op"]
    if op == "build":
        res = b.build(s["dm"], s["want"])
        return {k: res[k] for k in ("nodes", "elems") if k in res}
    if op == "adj":
        return b.element_neighbors(s["dm"], s["node_elems"])
    if op == "batch":
        st = nn.nn_batch_submit(b.h, s["meshes"], s["nodes"], s["elems"], len(s["dms"]), s["ws"].data_ptr(),
                                s["ws_bytes"], s["status"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        out = s["out"]
    elif op == "chunked":
        st = b.launch_chunked(s["dm"], s["want"], s["out"], s["chunks"], s["ws"], s["ws_bytes"])
        out = s["out"]
    else:
        st = b.launch(s["dm"], s["want"], s["out"], ws=s["ws"], ws_bytes=s["ws_bytes"])
        out = s["out"]
    if st:
        raise RuntimeError("status %d" % st)
    return out


# ------------------------------------------------------------------- work

def _sizes(mesh, n, holes=0.0):
    """(nodes, elements, incidences, node-row entries, face-neighbour entries), expected values where the seed decides."""
    m = n - 1
    if mesh == "tri":
        keep = 1 - holes
        inner, rim = 2 * m * (m - 1) + m * m, 4 * m
        T = 2 * m * m - int(2 * m * m * holes)
        return n * n, T, 3 * T, 2 * (inner * (1 - holes ** 2) + rim * keep), 2 * inner * keep ** 2
    if mesh == "quad":
        return n * n, m * m, 4 * m * m, 4 * m * n, 4 * m * (m - 1)
    if mesh == "tet":
        T = 6 * m ** 3
        return n ** 3, T, 4 * T, 2 * (3 * m * n * n + 3 * m * m * n + m ** 3), 4 * T - 12 * m * m
    if mesh == "hex":
        return n ** 3, m ** 3, 8 * m ** 3, 6 * m * n * n, 6 * m * m * (m - 1)
    inner, rim, s = 3 * m * m * (m - 1), 6 * m * m, SPLIT
    edges = 3 * m * n * n + inner * (1 - (1 - s) ** 2) + rim * s + s * m ** 3
    T = m ** 3 * (1 + 5 * s)
    adj = s * m ** 3 * 12 + 2 * inner * ((1 - s) ** 2 + 2 * s * s + 4 * s * (1 - s))
    return n ** 3, T, m ** 3 * (8 * (1 - s) + 24 * s), 2 * edges, adj


def work(case):
    """Connectivity read once, each wanted CSR written once (adjacency: the node-to-element CSR read too)."""
    if case["op"] == "batch":
        grids = [_sizes(m, n) for m, n in _batch_specs(case)]
    else:
        grids = [_sizes(case["mesh"], case["n"], case.get("holes", 0.0))]
    total = 0.0
    for N, T, C, nnz, adj in grids:
        total += 4 * C
        if case.get("mesh") == "mixed":
            total += 9 * T
        if case["op"] == "adj":
            total += 8 * (N + 1) + 4 * C + 8 * (T + 1) + 4 * adj
            continue
        if case["want"] != "elems":
            total += 8 * (N + 1) + 4 * nnz
        if case["want"] != "nodes":
            total += 8 * (N + 1) + 4 * C
    return {"bytes": float(total), "flops": 0.0}


# ------------------------------------------------------------------ exact

def _csr(rows, cols, n_rows, n_cols, cap=None):
    """Canonical CSR of the pairs: rows ascending, without repeats; col filled up with zeros to `cap`."""
    key = torch.unique(rows * n_cols + cols)
    rp = torch.zeros(n_rows + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(torch.div(key, n_cols, rounding_mode="floor"), minlength=n_rows), 0, out=rp[1:])
    col = torch.zeros(key.numel() if cap is None else max(cap, 1), dtype=torch.int32, device="cuda")
    col[: key.numel()] = (key % n_cols).to(torch.int32)
    return rp, col


def _parts(groups):
    """(type, element ids, nodes as 64-bit) of every type group of a mesh."""
    for t, (ids, el) in groups.items():
        yield t, torch.arange(el.shape[0], device="cuda") if ids is None else ids, el.long()


def _exact_build(mesh, N, groups, conn, want, trimmed):
    C, out = conn.numel(), {}
    T = sum(el.shape[0] for _, el in groups.values())
    if want != "elems":
        v = torch.cat([el[:, i] for t, _, el in _parts(groups) for i in range(NPE[t]) for _ in NBRS[t][i]])
        w = torch.cat([el[:, j] for t, _, el in _parts(groups) for i in range(NPE[t]) for j in NBRS[t][i]])
        out["nodes"] = _csr(v, w, N, N, None if trimmed else _cap(mesh, C, "nodes"))
        del v, w
    if want != "nodes":
        v = torch.cat([el.reshape(-1) for _, _, el in _parts(groups)])
        e = torch.cat([ids.repeat_interleave(NPE[t]) for t, ids, _ in _parts(groups)])
        out["elems"] = _csr(v, e, N, T, None if trimmed else C)
    return out


def _exact_adj(mesh, N, el):
    """Elements that share a face, by sorting the faces: a face of these conforming grids is known by its
    nodes, a hex face already by its smallest node and the one across from it."""
    faces, T = FACES[mesh], el.shape[0]
    f = el[:, torch.tensor(faces, device="cuda")].reshape(T * len(faces), -1)
    if mesh == "hex":
        lo, at = f.min(1)
        key = lo * N + f.gather(1, ((at + 2) % 4)[:, None])[:, 0]
    else:
        f = f.sort(1).values
        key = f[:, 0]
        for i in range(1, f.shape[1]):
            key = key * N + f[:, i]
    key, at = key.sort()
    e = torch.div(at, len(faces), rounding_mode="floor")
    same = key[1:] == key[:-1]
    a, b = e[:-1][same], e[1:][same]
    return _csr(torch.cat((a, b)), torch.cat((b, a)), T, T)


def exact(case, seed):
    g = _generator(seed)
    if case["op"] == "batch":
        all_ = []
        for m, n in _batch_specs(case):
            N, groups, conn, _, _ = _mesh(m, n, case["order"], 0.0, g)
            all_.append(_exact_build(m, N, groups, conn, case["want"], False))
        return {k: [torch.cat([torch.nn.functional.pad(x[k][i], (0, -x[k][i].numel() % 64)) for x in all_])
                    for i in (0, 1)] for k in all_[0]}
    mesh = case["mesh"]
    N, groups, conn, _, _ = _mesh(mesh, case["n"], case["order"], case.get("holes", 0.0), g)
    if case["op"] == "adj":
        if mesh == "tet" and N ** 3 >= 2 ** 63:  # a face's three nodes have to fit one 64-bit key
            return None
        return _exact_adj(mesh, N, groups[mesh][1].long())
    return _exact_build(mesh, N, groups, conn, case["want"], case["op"] == "build")
