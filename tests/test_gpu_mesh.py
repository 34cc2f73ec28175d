"""The grouped build of the edge list and of L's structure at the sizes where
its paths change: one tet, groups around a warp's 32 and its 64 shared-memory
entries, a node with thousands of edges (radix sorts) as the smallest and as
the largest id, and node numberings without locality.  Integers: bit-exact
against the oracle."""
import numpy as np
import pytest

import oracle as O
from dec_inputs import canonical_tets, make_workload

pytestmark = pytest.mark.gpu


def sphere(rings, segments, centre_last):
    """Tets joining a closed triangulated sphere to its centre."""
    th = np.pi * (np.arange(rings) + 1) / (rings + 1)
    ph = 2 * np.pi * np.arange(segments) / segments
    pts = np.stack([np.sin(th)[:, None] * np.cos(ph), np.sin(th)[:, None] * np.sin(ph),
                    np.broadcast_to(np.cos(th)[:, None], (rings, segments))], -1).reshape(-1, 3)
    i, j = np.meshgrid(np.arange(rings - 1), np.arange(segments), indexing="ij")
    a, b = i * segments + j, i * segments + (j + 1) % segments
    c, d = a + segments, b + segments
    tri = np.concatenate([np.stack([a, b, c], -1).reshape(-1, 3),
                          np.stack([b, d, c], -1).reshape(-1, 3)])
    n = rings * segments                       # then the poles and the centre
    j = np.arange(segments)
    k = (j + 1) % segments
    top = np.stack([np.full(segments, n), j, k], -1)
    bottom = np.stack([np.full(segments, n + 1), k + n - segments, j + n - segments], -1)
    tri = np.concatenate([tri, top, bottom])
    pts = np.concatenate([pts, [[0, 0, 1], [0, 0, -1], [0, 0, 0]]])
    tets = np.concatenate([tri, np.full((len(tri), 1), n + 2)], 1)
    if not centre_last:                        # rotate the ids: the centre becomes 0
        tets = (tets + 1) % (n + 3)
        pts = np.roll(pts, 1, axis=0)
    return np.ascontiguousarray(pts), canonical_tets(tets, pts)


def renumbered(N, seed):
    wl = make_workload("lognormal64", N=N)
    new = np.random.default_rng(seed).permutation(wl.n)
    xyz = np.empty_like(wl.xyz)
    xyz[new] = wl.xyz
    return xyz, canonical_tets(new[wl.tets], xyz)


MESHES = {
    "one tet": lambda: (np.array([[0., 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]]),
                        np.array([[0, 1, 2, 3]], dtype=np.int32)),
    "hub 30": lambda: sphere(2, 3, False),      # 36 entries at node 0
    "hub 64": lambda: sphere(3, 4, False),      # 72
    "hub first": lambda: sphere(28, 30, False),   # 5,040 entries at node 0
    "hub last": lambda: sphere(66, 64, True),     # 4,226 lower neighbours
    "shuffled 7": lambda: renumbered(7, 1),
    "shuffled 20": lambda: renumbered(20, 2),
    "far away": lambda: (renumbered(6, 3)[0] + 1e7, renumbered(6, 3)[1]),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_edges_and_structure(name):
    from paper_2104_05999_gb300 import abi
    xyz, tets = MESHES[name]()
    tags = np.zeros(len(xyz), dtype=np.uint8)
    E, t2e = O.edge_list(tets)
    with abi.Context(device=0) as ctx:
        ctx.dec_mesh_upload(np.ascontiguousarray(xyz), tets, tags)
        Eg, t2eg = ctx.dec_get_edges()
        rowptr, col, _, _ = ctx.dec_get_csr(values=False)
        # an inverted tet is still refused, wherever the mesh lies
        bad = tets.copy()
        bad[-1, [0, 1]] = bad[-1, [1, 0]]
        with pytest.raises(abi.DecError) as e:
            ctx.dec_mesh_upload(np.ascontiguousarray(xyz), bad, tags)
        assert e.value.status == abi.DEC_ERR_MESH
    assert np.array_equal(E, Eg) and np.array_equal(t2e, t2eg)
    n = len(xyz)
    both = np.concatenate([E, E[:, ::-1], np.stack([np.arange(n)] * 2, 1)]).astype(np.int64)
    order = np.lexsort((both[:, 1], both[:, 0]))
    assert np.array_equal(col, both[order, 1])
    assert np.array_equal(rowptr, np.searchsorted(both[order, 0], np.arange(n + 1)))
