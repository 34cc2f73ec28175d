"""FP64 solves of small systems in one cluster launch against the kernels that
larger systems take (a forced SELL launch shape keeps those): one slice, the
edges of a 512-row window, about a slice per warp, and a hub whose rows do not
fit in shared memory, so that one block of the cluster reads them from global
memory.  Both end below a residual of 1e-12, and the condition numbers here
are below 1e4, so temperatures agree to 1e-8; iteration counts differ by the
order of the sums only."""
import numpy as np
import pytest

from dec_inputs import make_workload
from test_gpu_mesh import sphere

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    c = abi.Context(device=0)
    yield c
    c.close()


def inputs(name):
    if name == "hub":
        xyz, tets = sphere(28, 30, False)
        tags = np.zeros(len(xyz), dtype=np.uint8)
        T0 = np.zeros(len(xyz))
        hot, cold = xyz[:, 2] > 0.9, xyz[:, 2] < -0.9
        tags[hot | cold] = 1
        T0[hot] = 1.0
        return xyz, tets, tags, T0, None
    wl = make_workload("lognormal64", N=int(name))
    return wl.xyz, wl.tets, wl.tags, wl.T0, wl.k


@pytest.mark.parametrize("precond", ["fsai", "jacobi"])
@pytest.mark.parametrize("name", ["3", "8", "9", "18", "hub"])
def test_cluster_solve_matches_the_general_kernels(ctx, name, precond):
    from paper_2104_05999_gb300 import abi, run
    xyz, tets, tags, T0, k = inputs(name)
    assert abi.DEC_NODE_DIRICHLET == 1
    T0 = np.reshape(T0, (-1, len(xyz)))[:1]
    sets = np.concatenate([T0, 0.0 * T0, T0[:, ::-1] * (tags == 1)])

    def solve(max_iter=100000):
        return run.run_path(ctx, xyz, tets, tags, sets, k=k, precond=precond, mode="fp64",
                            rtol=1e-12, max_iter=max_iter, raise_on_error=False)
    got, short = solve(), solve(3)
    ctx.dec_set_sell_variant(408, 14)
    try:
        want, want_short = solve(), solve(3)
    finally:
        ctx.dec_set_sell_variant(0, 0)
    assert got.status == want.status == 0
    assert (got.relres <= 1e-12).all()
    assert got.iters[1] == 0 and not got.T[1].any()
    for b in (0, 2):
        assert np.linalg.norm(got.T[b] - want.T[b]) <= 1e-8 * np.linalg.norm(want.T[b])
        assert abs(int(got.iters[b]) - int(want.iters[b])) <= 3
    np.testing.assert_allclose(got.energy, want.energy, rtol=1e-8, atol=1e-14)
    assert short.status == want_short.status
    assert np.array_equal(short.iters, want_short.iters)
