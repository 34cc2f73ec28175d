"""A Dirichlet value that makes the right-hand side NaN, or its norm overflow:
an FP64 solve reports DEC_ERR_BREAKDOWN, as include/dec.h says, in the cluster
launch of small systems and in the kernels of larger ones (forced here by a
SELL launch shape) alike.  A right-hand side of 0 still needs no iteration, and
the context solves the next system."""
import numpy as np
import pytest

from dec_inputs import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", ["fsai", "jacobi"])
@pytest.mark.parametrize("forced", [False, True])
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e160])
def test_right_hand_side_that_is_not_finite_breaks_down(bad, forced, precond):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    wl = make_workload("lognormal64", N=6)
    hot = wl.T0[0] != 0.0
    T0 = wl.T0[:1].copy()
    if np.isfinite(bad):
        T0[:, hot] *= bad
    else:
        T0[0, np.flatnonzero(hot)[0]] = bad
    pc = {"fsai": abi.DEC_PRECOND_FSAI, "jacobi": abi.DEC_PRECOND_JACOBI}[precond]
    with abi.Context(device=0) as ctx:
        if forced:
            ctx.dec_set_sell_variant(408, 14)
        ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags)
        ctx.dec_hodge_assemble(wl.k)
        ctx.dec_laplacian_build(T0, pc)
        st, iters, relres = ctx.dec_solve(1e-10, 500, abi.DEC_MODE_FP64, raise_on_error=False)
        assert st == abi.DEC_ERR_BREAKDOWN
        st, steps, _ = ctx.dec_crack_evolve(abi.DEC_CRACK_MAX_FLUX, 3, raise_on_error=False)
        assert st == abi.DEC_ERR_BREAKDOWN and len(steps) == 0
        ctx.dec_laplacian_build(np.zeros_like(T0), pc)
        st, iters, relres = ctx.dec_solve(1e-10, 500, abi.DEC_MODE_FP64)
        assert iters[0] == 0 and relres[0] == 0.0
        ctx.dec_laplacian_build(wl.T0[:1], pc)
        st, iters, relres = ctx.dec_solve(1e-10, 500, abi.DEC_MODE_FP64)
        assert iters[0] > 0 and relres[0] <= 1e-10
        # rtol >= 1 still takes an iteration
        st, iters, relres = ctx.dec_solve(2.0, 500, abi.DEC_MODE_FP64)
        assert iters[0] == 1
