"""The grouped build of the edge list and of L's structure for nodes with many
edges: on both sides of the lines between a warp's, a block's and the radix
sorts (256 and 16,384 entries or lower neighbours), with the hub as the first,
the last and a middle node, and with many hubs at once.  Integers: bit-exact
against the oracle."""
import numpy as np
import pytest

import test_gpu_mesh as mesh
from dec_inputs import canonical_tets

pytestmark = pytest.mark.gpu


def rotated(xyz, tets, shift):
    xyz = np.roll(xyz, shift, axis=0)
    return xyz, canonical_tets((tets + shift) % len(xyz), xyz)


def copies(xyz, tets, count):
    n = len(xyz)
    return (np.concatenate([xyz + 3.0 * i for i in range(count)]),
            np.concatenate([tets + n * i for i in range(count)]).astype(np.int32))


MESHES = {   # sphere(rings, segments): 6 r s entries at a first hub, r s + 2 neighbours
    "first 252": lambda: mesh.sphere(1, 42, False),
    "first 258": lambda: mesh.sphere(1, 43, False),
    "first 1020": lambda: mesh.sphere(10, 17, False),
    "first 4092": lambda: mesh.sphere(22, 31, False),
    "first 16380": lambda: mesh.sphere(42, 65, False),
    "first 16386": lambda: mesh.sphere(1, 2731, False),
    "last 256": lambda: mesh.sphere(2, 127, True),
    "last 257": lambda: mesh.sphere(15, 17, True),
    "last 4096": lambda: mesh.sphere(46, 89, True),
    "last 16384": lambda: mesh.sphere(2, 8191, True),
    "last 16385": lambda: mesh.sphere(127, 129, True),
    "middle": lambda: rotated(*mesh.sphere(24, 30, True), 300),
    "forty first": lambda: copies(*mesh.sphere(9, 12, False), 40),
    "forty last": lambda: copies(*mesh.sphere(15, 20, True), 40),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_edges_and_structure_with_hubs(name, monkeypatch):
    monkeypatch.setitem(mesh.MESHES, name, MESHES[name])
    mesh.test_edges_and_structure(name)
