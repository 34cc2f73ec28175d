"""Small FP64 solves where the device cannot place a cluster of 16 blocks: a
child process runs with a stand-in for the two runtime calls concerned, which
reports room for no cluster and refuses cluster launches.  The solves then take
the kernels per phase and give what those give."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = """
static int launches;
int cudaOccupancyMaxActiveClusters(int *n, const void *f, const void *c) { *n = 0; return 0; }
int cudaLaunchKernelExC(const void *c, const void *f, void **a) { ++launches; return 701; }
int fake_cluster_launches(void) { return launches; }
"""
CHILD = """
import ctypes, sys
import numpy as np
from dec_inputs import make_workload
from paper_2104_05999_gb300 import abi, run
wl = make_workload("lognormal64", N=9)
for precond in ("fsai", "jacobi"):
    res, grown = [], []
    for shapes in ((0, 0), (408, 14)):
        with abi.Context(device=0) as ctx:
            ctx.dec_set_sell_variant(*shapes)
            res.append(run.run_path(ctx, wl.xyz, wl.tets, wl.tags, wl.T0, k=wl.k,
                                    precond=precond, mode="fp64", rtol=1e-11))
            grown.append(ctx.dec_crack_evolve(abi.DEC_CRACK_MAX_FLUX, 4, rtol=1e-11))
    assert res[0].relres[0] <= 1e-11
    assert np.array_equal(res[0].T, res[1].T) and np.array_equal(res[0].iters, res[1].iters)
    assert np.array_equal(grown[0][1], grown[1][1]) and np.array_equal(grown[0][2], grown[1][2])
assert ctypes.CDLL(sys.argv[1]).fake_cluster_launches() == 0
print("fallback ok")
"""


def test_solves_without_room_for_a_cluster(tmp_path):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build
    _build.build()
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler")
    src, lib = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.run([cc, "-shared", "-fPIC", "-o", str(lib), str(src)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "fallback ok" in r.stdout, r.stdout + r.stderr
