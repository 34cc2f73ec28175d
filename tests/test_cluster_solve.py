"""The cluster solve of small FP64 systems beside other work.

A block may store into the shared memory of another block of its cluster only
once that block runs, so a cluster barrier has to end before the first sum is
exchanged; the source is read for that.  On the GPU, contexts in several
threads solve while a third stream keeps the SMs busy, so that the blocks of a
cluster wait for room: the temperatures are those of a solve alone, bit for
bit (every sum has a fixed order).
"""
import os
import re
import threading

import numpy as np
import pytest

from dec_inputs import make_workload

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2104_05999_gb300", "csrc")


def test_every_block_has_started_before_the_first_remote_store():
    with open(os.path.join(CSRC, "dec_persist.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    body = src[src.index("pcg_cluster_kernel(ClusterArgs a) {"):]
    body = body[:body.index("\ndec_status ")]
    arrive = body.index("cluster.barrier_arrive()")
    wait = body.index("cluster.barrier_wait(")
    # the stores stand in sum2, which only run() calls
    calls = [m.start() for m in re.finditer(r"\brun\(std::", body)]
    store, solve = body.index("store_cluster("), body.index("auto run = ")
    assert len(calls) == 2 and arrive < wait < min(calls)
    assert store < solve and not re.search(r"\bsum2\(", body[:solve].split("auto sum2", 1)[0])
    assert not re.search(r"\bsum2\(", body[store:solve])


@pytest.mark.gpu
@pytest.mark.parametrize("precond", ["fsai", "jacobi"])
def test_concurrent_solves_are_those_of_a_solve_alone(precond):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_2104_05999_gb300 import _build, abi, run
    _build.build()
    abi.load()
    sizes = (5, 9, 13, 17)
    wls = [make_workload("lognormal64", N=N) for N in sizes]

    def solve(ctx, wl):
        return run.run_path(ctx, wl.xyz, wl.tets, wl.tags, wl.T0, k=wl.k, precond=precond,
                            mode="fp64", rtol=1e-11)
    alone = []
    for wl in wls:
        with abi.Context(device=0) as ctx:
            alone.append(solve(ctx, wl))
    got, errors = [[] for _ in wls], []

    def work(i):
        try:
            with abi.Context(device=0) as ctx:
                for _ in range(6):
                    got[i].append(solve(ctx, wls[i]))
        except Exception as e:       # reported by the main thread
            errors.append(e)
    side = torch.cuda.Stream()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(wls))]
    for t in threads:
        t.start()
    with torch.cuda.stream(side):
        a = torch.ones(4096, 4096, device="cuda")
        while any(t.is_alive() for t in threads):
            for _ in range(4):
                a = (a @ a) * 2.0 ** -12
            side.synchronize()
    for t in threads:
        t.join()
    assert not errors, errors
    for want, res in zip(alone, got):
        assert len(res) == 6
        for r in res:
            assert np.array_equal(r.T, want.T) and np.array_equal(r.iters, want.iters)
