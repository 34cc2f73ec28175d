"""dec_get_launch_count counts the kernels that ran: step by step the number the
profiler records, for meshes below and above the sizes where prefix sums take
one launch or three, with discs, hubs, thin tets, every solve mode and crack
growth."""
import numpy as np
import pytest

from dec_inputs import crack_scales, make_fields, make_workload
from test_gpu_mesh import sphere

pytestmark = pytest.mark.gpu


def kernels(f):
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        f()
        torch.cuda.synchronize()
    return sum(e.device_type == torch.autograd.DeviceType.CUDA and "dec::" in e.name
               for e in p.events())


@pytest.mark.parametrize("N", [5, 13, 23])
def test_counted_launches_are_those_the_profiler_sees(N):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    wl = make_workload("hetero192", N=N)
    thin = wl.xyz * np.array([1.0, 1.0, 1e-4])
    hub_xyz, hub_tets = sphere(20, 30, N > 5)
    scales = crack_scales(9)
    with abi.Context(device=0) as ctx:
        ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags)
        if not any(kernels(lambda: ctx.dec_hodge_assemble(None)) for _ in range(3)):
            pytest.skip("the profiler records no kernels here")
        steps = [lambda: ctx.dec_mesh_upload(hub_xyz, hub_tets,
                                             np.zeros(len(hub_xyz), dtype=np.uint8)),
                 lambda: ctx.dec_mesh_upload(thin, wl.tets, wl.tags),
                 lambda: ctx.dec_hodge_assemble(None, wl.discs, scales),
                 lambda: ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags),
                 lambda: ctx.dec_hodge_assemble(wl.k, wl.discs),
                 lambda: ctx.dec_laplacian_build(wl.T0[:1], abi.DEC_PRECOND_JACOBI),
                 lambda: ctx.dec_solve(1e-8, 5000, abi.DEC_MODE_FP64),
                 lambda: ctx.dec_laplacian_build(wl.T0[:2], abi.DEC_PRECOND_FSAI)]
        steps += 2 * [lambda m=m: ctx.dec_solve(1e-8, 5000, m)
                      for m in (abi.DEC_MODE_FP64, abi.DEC_MODE_MIXED, abi.DEC_MODE_MIXED_PHASED)]
        steps += [lambda: ctx.dec_k_eff(),
                  lambda: ctx.dec_laplacian_build(wl.T0, abi.DEC_PRECOND_FSAI_SHARED),
                  lambda: ctx.dec_solve(1e-8, 5000, abi.DEC_MODE_MIXED_BATCHED),
                  lambda: ctx.dec_k_eff(),
                  lambda: ctx.dec_hodge_assemble_fields(make_fields(wl, 3), wl.discs),
                  lambda: ctx.dec_laplacian_build(wl.T0[:1], abi.DEC_PRECOND_FSAI_SHARED),
                  lambda: ctx.dec_hodge_assemble(wl.k),
                  lambda: ctx.dec_laplacian_build(wl.T0[:1], abi.DEC_PRECOND_FSAI),
                  lambda: ctx.dec_crack_evolve(abi.DEC_CRACK_MAX_FLUX, 2, rtol=1e-8),
                  lambda: ctx.dec_tet_solve(wl.T0[0], rtol=1e-8),
                  lambda: ctx.dec_tet_solve(wl.T0[0], rtol=1e-8)]
        for i, step in enumerate(steps):
            before = ctx.dec_get_launch_count()
            seen = kernels(step)
            assert ctx.dec_get_launch_count() - before == seen, i
