"""The FP32 sub-triangle test of the crack states where its bounds decide
little or nothing: thin tets, coordinates far from the origin, planes through
mesh nodes (corners exactly on the plane), many states, one far disc.  The
states are the oracle's FP64 ones, edge by edge."""
import numpy as np
import pytest

import oracle as O
from dec_inputs import crack_scales, make_workload, penny_discs

pytestmark = pytest.mark.gpu


def case(name):
    wl = make_workload("lognormal64", N=7)
    xyz, scales = wl.xyz.copy(), None
    discs = penny_discs(14, 0.1, 0.5, np.random.default_rng(5))
    if name == "thin":
        xyz[:, 0] *= 1e-3
        discs[:, 0] *= 1e-3
    elif name == "flat tets":
        xyz[:, 2] *= 1e-5
        discs[:, 2] *= 1e-5
    elif name == "far":
        xyz += 300.0
        discs[:, :3] += 300.0
    elif name == "states":
        scales = crack_scales(40, 0.02, 1.5)
    elif name == "through nodes":
        wl = make_workload("kuhn9", N=5)
        xyz = wl.xyz.copy()
        discs = np.array([[0.5, 0.5, 0.5, 0, 0, 1, 0.3], [0.25, 0.5, 0.5, 1, 0, 0, 0.4],
                          [0.5, 0.75, 0.3, 0, 1, 0, 0.2]])
    elif name == "miss":
        discs[:, :3] += 9.0
    return np.ascontiguousarray(xyz), wl.tets, discs, scales


@pytest.mark.parametrize("geom", [0, 1])
@pytest.mark.parametrize("name", ["plain", "thin", "flat tets", "far", "states", "through nodes",
                                  "miss"])
def test_states_match_oracle(name, geom):
    from paper_2104_05999_gb300 import abi
    xyz, tets, discs, scales = case(name)
    E, t2e = O.edge_list(tets)
    want = O.edge_crack_state(xyz, tets, E, t2e, discs, scales)
    with abi.Context(device=0) as ctx:
        ctx.dec_set_geom_precision(geom)
        ctx.dec_mesh_upload(xyz, tets, np.zeros(len(xyz), dtype=np.uint8))
        ctx.dec_hodge_assemble(None, discs, scales)
        _, got = ctx.dec_get_hodge()
    assert np.array_equal(got.astype(np.int64), want)
