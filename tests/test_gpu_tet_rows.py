"""The tet-centred solve where a block goes through its rows more than once
(more tets than 152 blocks of 1,024 threads) and where the last block is
ragged: a linear field is reproduced at every circumcentre.  The smaller
lattices of the other tests hold 1e-10 at N = 7; the condition number grows
with N^2, so (32 / 7)^2 times that is allowed here."""
import numpy as np
import pytest

from dec_inputs import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [6, 32])
def test_linear_field_over_several_rows_per_thread(N):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    wl = make_workload("lognormal64", N=N)
    m = len(wl.tets)
    assert m % 1024 and (N < 32 or m > 152 * 1024)
    ctx = abi.Context(device=0)
    try:
        ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags)
        res = ctx.dec_tet_solve(wl.T0[0], limiter=1e-8, rtol=1e-11)
    finally:
        ctx.close()
    P = wl.xyz[wl.tets]
    d = P[:, 1:] - P[:, :1]
    centre = P[:, 0] + np.linalg.solve(2.0 * d, (d * d).sum(-1)[..., None])[..., 0]
    assert res["limited"] == 0
    np.testing.assert_allclose(res["alpha"], 1.0 - centre[:, 0], atol=2.1e-9)
    assert res["q_in"] == pytest.approx(1.0, rel=2.1e-9)
    assert res["q_out"] == pytest.approx(1.0, rel=2.1e-9)
