"""Batched solves with more windows than SMs, where a block goes from window to
window (the small meshes of the other tests spread their slices over all SMs):
8 Dirichlet sets in windows of 512 rows, 16 fields of 256, 40 crack states of
64, the last window ragged.  Every launch variant gives the same bits, and the
temperatures are those of FP64 solves of the single instances by the kernels
per phase, to the 1e-8 that this library's solves are held to (residuals of
1e-11 here)."""
import numpy as np
import pytest

from dec_inputs import crack_scales, make_fields, make_workload

pytestmark = pytest.mark.gpu

VARIANTS = {"sets": (2, 4, 12, 114, 106, 1004, 2004, 2002, 2512),
            "fields": (2, 4, 12, 114, 106), "states": (2, 4, 12, 114, 106)}
SIZE = {"sets": (44, 512), "fields": (34, 256), "states": (22, 64)}


@pytest.mark.parametrize("kind", list(SIZE))
def test_variants_over_several_windows_per_block(kind):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    N, rows = SIZE[kind]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wl = make_workload("hetero192" if kind == "sets" else "growth96", N=N)
    assert wl.n > rows * sms and wl.n % rows
    T0 = wl.T0[:8] if kind == "sets" else wl.T0[:1]
    with abi.Context(device=0) as ctx:
        ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags)
        if kind == "fields":
            ctx.dec_hodge_assemble_fields(make_fields(wl, 16), None)
        else:
            ctx.dec_hodge_assemble(wl.k, wl.discs, crack_scales(40) if kind == "states" else None)
        ctx.dec_laplacian_build(T0, abi.DEC_PRECOND_FSAI)
        B = ctx.sizes()[4]
        assert B == {"sets": 8, "fields": 16, "states": 40}[kind]
        want = np.zeros((B, wl.n))
        ctx.dec_solve(1e-11, 20000, abi.DEC_MODE_FP64, want)
        ctx.dec_laplacian_build(T0, abi.DEC_PRECOND_FSAI_SHARED)
        base = None
        for v in VARIANTS[kind]:
            ctx.dec_set_batch_variant(v)
            T = np.zeros((B, wl.n))
            _, iters, relres = ctx.dec_solve(1e-11, 20000, abi.DEC_MODE_MIXED_BATCHED, T)
            assert (relres <= 1e-11).all()
            if base is None:
                base = T, iters
                for b in range(B):
                    assert np.linalg.norm(T[b] - want[b]) <= 1e-8 * np.linalg.norm(want[b])
            else:
                assert np.array_equal(T, base[0]) and np.array_equal(iters, base[1]), v
