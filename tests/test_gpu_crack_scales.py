"""Crack states of meshes in small and large units: mesh and discs multiplied
by a power of two, so that every product of the FP64 test scales exactly and
the states are those of the unscaled mesh (the oracle's), while single
precision would underflow or overflow in the fifth powers of lengths that
circumcentres need.  The last cases mix sizes: a fine mesh among coarse discs,
radii and scales at the ends of the FP32 range."""
import numpy as np
import pytest

import oracle as O
from dec_inputs import crack_scales, make_workload, penny_discs

pytestmark = pytest.mark.gpu

POWERS = [-120, -60, -40, -30, -27, -24, -20, 24, 26, 30, 40, 60, 120]


def states(xyz, tets, discs, scales, geom=0):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    with abi.Context(device=0) as ctx:
        ctx.dec_set_geom_precision(geom)
        ctx.dec_mesh_upload(np.ascontiguousarray(xyz), tets, np.zeros(len(xyz), dtype=np.uint8))
        ctx.dec_hodge_assemble(None, np.ascontiguousarray(discs), scales)
        return ctx.dec_get_hodge()[1].astype(np.int64)


def oracle_states(xyz, tets, discs, scales):
    E, t2e = O.edge_list(tets)
    return O.edge_crack_state(xyz, tets, E, t2e, discs, scales)


@pytest.fixture(scope="module")
def cube():
    wl = make_workload("lognormal64", N=7)
    discs = penny_discs(14, 0.1, 0.5, np.random.default_rng(5))
    scales = crack_scales(5, 0.1, 1.2)
    return wl.xyz, wl.tets, discs, scales, oracle_states(wl.xyz, wl.tets, discs, scales)


def scaled(xyz, discs, f):
    d = discs.copy()
    d[:, :3] *= f
    d[:, 6] *= f
    return xyz * f, d


@pytest.mark.parametrize("power", POWERS)
def test_states_do_not_depend_on_the_unit(cube, power):
    xyz, tets, discs, scales, want = cube
    x, d = scaled(xyz, discs, 2.0 ** power)
    assert 0 < (want < 5).sum() < want.size
    assert np.array_equal(states(x, tets, d, scales), want)


@pytest.mark.parametrize("name", ["fine mesh", "small radii", "large radii", "small scales",
                                  "large scales"])
def test_states_of_unlike_sizes(cube, name):
    xyz, tets, discs, scales, _ = cube
    discs = discs.copy()
    if name == "fine mesh":                # 2^-28 of the cube, at a disc's rim
        axis = np.cross(discs[0, 3:6], [0.3, -0.5, 0.8])
        discs[:, :3] -= discs[0, :3] + discs[0, 6] * axis / np.linalg.norm(axis)
        discs[:, 6] *= 1.0 + 1e-9
        xyz = (xyz - 0.5) * 2.0 ** -28
        scales = np.array([1.0])
    elif name == "small radii":            # r = 1e-41 to 1e-39, scales that undo it
        discs[:, 6] *= 2.0 ** -130
        scales = scales * 2.0 ** 130
    elif name == "large radii":
        discs[:, 6] *= 2.0 ** 140
        scales = scales * 2.0 ** -140
    elif name == "small scales":
        scales = scales * 1e-42
    elif name == "large scales":
        scales = scales * 1e39
    want = oracle_states(xyz, tets, discs, scales)
    assert np.array_equal(states(xyz, tets, discs, scales), want)


@pytest.mark.parametrize("power", POWERS)
def test_fp32_geometry_in_any_unit(cube, power):
    """DEC_GEOM_MIXED: the same states, and *1 within the 2e-6 of the largest
    weight that FP32 geometry is held to at unit scale."""
    xyz, tets, discs, scales, want = cube
    x, d = scaled(xyz, discs, 2.0 ** power)
    assert np.array_equal(states(x, tets, d, scales, geom=1), want)
    from paper_2104_05999_gb300 import abi
    E, t2e = O.edge_list(tets)
    w = O.hodge_star1(xyz, tets, E, t2e) * 2.0 ** power
    with abi.Context(device=0) as ctx:
        ctx.dec_set_geom_precision(abi.DEC_GEOM_MIXED)
        ctx.dec_mesh_upload(np.ascontiguousarray(x), tets, np.zeros(len(x), dtype=np.uint8))
        ctx.dec_hodge_assemble(None)
        got = ctx.dec_get_hodge()[0]
    assert np.abs(got - w).max() <= 2e-6 * np.abs(w).max()
