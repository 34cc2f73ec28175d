"""Dirichlet sets, crack states and conductivity fields solved after one
another on one context, mesh and instance stride: each kind has its own
kernels, so each tunes its launch variant itself (the staged variants exist
for sets only) and keeps its choice when the others come in between."""
import numpy as np
import pytest

from dec_inputs import crack_scales, make_fields, make_workload

pytestmark = pytest.mark.gpu


def test_each_kind_of_instances_has_its_own_variant():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    wl = make_workload("hetero192", N=9)
    scales = crack_scales(8)
    fields = make_fields(wl, 8)
    sets = wl.T0

    def solve(ctx, kind):
        """temperatures, launches of the solve, variant"""
        if kind == "fields":
            ctx.dec_hodge_assemble_fields(fields, None)
        else:
            ctx.dec_hodge_assemble(wl.k, wl.discs, scales if kind == "states" else None)
        ctx.dec_laplacian_build(sets if kind == "sets" else sets[:1],
                                abi.DEC_PRECOND_FSAI_SHARED)
        T = np.zeros((8, wl.n))
        before = ctx.dec_get_launch_count()
        ctx.dec_solve(1e-10, 20000, abi.DEC_MODE_MIXED_BATCHED, T)
        return T, ctx.dec_get_launch_count() - before, ctx.dec_get_batch_variant()
    kinds = ("sets", "states", "fields")
    assert len(sets) == 8
    alone = {}
    for kind in kinds:
        with abi.Context(device=0) as ctx:
            ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags)
            alone[kind] = solve(ctx, kind)
    with abi.Context(device=0) as ctx:
        ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags)
        first = {kind: solve(ctx, kind) for kind in kinds}
        again = {kind: solve(ctx, kind) for kind in kinds}
    for kind in kinds:
        assert np.array_equal(first[kind][0], alone[kind][0])
        assert np.array_equal(again[kind][0], alone[kind][0])
        assert first[kind][1] == alone[kind][1]            # tuned for this kind
        assert again[kind][1] < first[kind][1]             # and remembered
        assert again[kind][2] == first[kind][2]
        assert kind == "sets" or first[kind][2] in (2, 4, 12, 114, 106)
