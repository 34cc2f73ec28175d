"""Crack states of meshes of thin tets, whose sub-triangles are tested in FP64
disc by disc: many discs and states per tet, circumballs that hold the whole
mesh, so that rejected, one-sided and cut pairs all occur.  The states are the
oracle's."""
import numpy as np
import pytest

import oracle as O
from dec_inputs import crack_scales, make_workload, penny_discs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom", [0, 1])
@pytest.mark.parametrize("axis,factor", [(2, 1e-2), (2, 1e-3), (0, 1e-4), (1, 1e-6)])
def test_states_of_thin_tets(axis, factor, geom):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    wl = make_workload("lognormal64", N=6)
    xyz = wl.xyz.copy()
    xyz[:, axis] *= factor
    discs = penny_discs(60, 0.02, 0.15, np.random.default_rng(7))
    discs[:, axis] *= factor
    scales = crack_scales(6, 0.1, 1.0)
    E, t2e = O.edge_list(wl.tets)
    want = O.edge_crack_state(xyz, wl.tets, E, t2e, discs, scales)
    assert len(np.unique(want)) > 3
    with abi.Context(device=0) as ctx:
        ctx.dec_set_geom_precision(geom)
        ctx.dec_mesh_upload(xyz, wl.tets, wl.tags)
        ctx.dec_hodge_assemble(None, discs, scales)
        got = ctx.dec_get_hodge()[1]
    assert np.array_equal(got.astype(np.int64), want)
