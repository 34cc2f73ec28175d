"""Orientation of tets whose FP32 determinant underflows: edges of about 2e-15
at coordinates of about 2e-12, where a product of three edges has no bits left
in FP32.  Tets are picked on the CPU whose determinant, in FP32 as the first
test of the upload computes it, comes out positive by rounding although the
tet is inverted; each is refused, and accepted once two nodes are swapped."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def truncated(v):
    return ((v.view(np.uint64) >> np.uint64(29)) << np.uint64(29)).view(np.float64).astype(
        np.float32)


def inverted_tets(count):
    rng = np.random.default_rng(1)
    k = 300000
    size = 10 ** rng.uniform(-12, -11.5, k)
    edge = 10 ** rng.uniform(-15.5, -14.5, k)
    base = rng.uniform(-1, 1, (k, 1, 3)) * size[:, None, None]
    base[:, 0, 0] = 1.05 * size
    x = base + rng.uniform(-1, 1, (k, 4, 3)) * edge[:, None, None]
    det = np.linalg.det((x[:, 1:] - x[:, :1]) * 1e14)
    x[det > 0] = x[det > 0][:, [0, 2, 1, 3]]
    d = (x[:, 1:] - x[:, :1]) * 1e14
    c = truncated(x.reshape(-1)).reshape(x.shape)
    a, b, e = np.moveaxis(c[:, 1:] - c[:, :1], 1, 0)
    det32 = (a[:, 0] * (b[:, 1] * e[:, 2] - b[:, 2] * e[:, 1]) +
             a[:, 1] * (b[:, 2] * e[:, 0] - b[:, 0] * e[:, 2]) +
             a[:, 2] * (b[:, 0] * e[:, 1] - b[:, 1] * e[:, 0]))
    clear = np.linalg.det(d) < -1e-3 * np.abs(d).max((1, 2)) ** 3
    pick = np.flatnonzero((det32 > 0) & clear)
    assert len(pick) >= count
    return x[pick[:count]]


def test_inverted_tets_of_tiny_meshes_are_refused():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi
    _build.build()
    abi.load()
    tets = np.array([[0, 1, 2, 3]], dtype=np.int32)
    tags = np.zeros(4, dtype=np.uint8)
    accepted = 0
    with abi.Context(device=0) as ctx:
        for x in inverted_tets(100):
            try:
                ctx.dec_mesh_upload(np.ascontiguousarray(x), tets, tags)
                accepted += 1
            except abi.DecError as e:
                assert e.status == abi.DEC_ERR_MESH
            ctx.dec_mesh_upload(np.ascontiguousarray(x[[0, 2, 1, 3]]), tets, tags)
    assert accepted == 0
