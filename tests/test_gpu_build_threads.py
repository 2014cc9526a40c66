"""Handles built by several threads at once, small and large ones in turn: the limits that a kernel
is given are the process's, and one thread's sizes must not show in another's build."""
import threading

import pytest
import torch

import workloads as W
from helpers import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["dense", "csr"])
def test_threads_build_handles_of_different_sizes(lsq, kind):
    if kind == "dense":     # both by one kernel instance: four columns of the operator per CTA
        mats = [W.gaussian_dense(2000, 460, 1), W.gaussian_dense(6000, 1900, 2)]
    else:
        mats = [W.sparse_random(6000, 100, 8, 1), W.sparse_random(200000, 4000, 8, 2)]
    jobs, want, fails = [], [], []
    for i, mat in enumerate(mats):
        Mx, keep, seen = to_device(lsq, mat)
        o = lsq.opts(seed=i)
        idx, p, d = lsq.lsq_sample_rows(Mx, o)
        R = torch.arange(1, Mx.n + 1, dtype=torch.float64, device="cuda")
        jobs.append((Mx, keep, o, idx, p, d, R))
        want.append(lsq.lsq_build_precond(Mx, idx, p, d, o).apply(R))
    torch.cuda.synchronize()

    def work(i):
        Mx, keep, o, idx, p, d, R = jobs[i]
        st = torch.cuda.Stream()
        try:
            with torch.cuda.stream(st):
                for _ in range(20):
                    if not torch.equal(lsq.lsq_build_precond(Mx, idx, p, d, o, stream=st).apply(R, stream=st), want[i]):
                        fails.append((i, "another result"))
        except Exception as ex:
            fails.append((i, str(ex)))

    threads = [threading.Thread(target=work, args=(i % 2,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not fails, fails
