"""The tet-centred solve on both sides of the line between its block sizes
(256 threads per block up to 6 rows a thread: 233,472 tets on 152 SMs): a
linear field is reproduced at every circumcentre.  The smaller lattices of the
other tests hold 1e-10 at N = 7; the condition number grows with N^2, so
(35 / 7)^2 times that is allowed here."""
import numpy as np
import pytest

from dec_inputs import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,small", [(4, True), (33, True), (35, False)])
def test_linear_field_with_either_block_size(N, small):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    wl = make_workload("lognormal64", N=N)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (len(wl.tets) <= 6 * 256 * sms) == small
    with abi.Context(device=0) as ctx:
        ctx.dec_mesh_upload(wl.xyz, wl.tets, wl.tags)
        res = ctx.dec_tet_solve(wl.T0[0], limiter=1e-8, rtol=1e-11)
        again = ctx.dec_tet_solve(wl.T0[0], limiter=1e-8, rtol=1e-11)
    assert np.array_equal(res["alpha"], again["alpha"])
    P = wl.xyz[wl.tets]
    d = P[:, 1:] - P[:, :1]
    centre = P[:, 0] + np.linalg.solve(2.0 * d, (d * d).sum(-1)[..., None])[..., 0]
    assert res["limited"] == 0
    np.testing.assert_allclose(res["alpha"], 1.0 - centre[:, 0], atol=2.5e-9)
    assert res["q_in"] == pytest.approx(1.0, rel=2.5e-9)
