"""GPU: host threads that solve on different plans at the same time, each on its own stream.  What one plan's launch needs of
a kernel's shared-memory limit must not depend on the plan another thread solves with."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle

pytestmark = pytest.mark.gpu

NOT_CONVERGED = 8


def test_small_and_large_partitions_at_once():
    import paper_2204_06666_gb300 as eh
    # two FP64 vectors of a partition: less than 100 KB, and more
    jobs = []
    for N, rows in ((20, 53), (37, 6500)):
        A = gen.tet_lap3d(N=N)
        P = eh.Plan(A, slice_rows=rows, block_threads=1024)
        M = eh.Fsai(P, A)
        b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 3))).cuda()
        x = torch.zeros_like(b)
        assert P.pcg(M, b, x, max_iter=2)[0] == NOT_CONVERGED
        jobs.append((P, M, b, x.clone()))
    torch.cuda.synchronize()
    bad = []
    start = threading.Barrier(len(jobs))

    def solve(P, M, b, ref):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            x = torch.empty_like(b)
            start.wait()
            for i in range(300):  # two iterations each: the solves are mostly launches
                x.zero_()
                try:
                    st, info = P.pcg(M, b, x, max_iter=2, stream=s)
                except eh.EhybError as e:
                    bad.append((b.numel(), i, str(e)))
                    return
                if st != NOT_CONVERGED or not torch.equal(x, ref):
                    bad.append((b.numel(), i, st, "bits"))
                    return

    threads = [threading.Thread(target=solve, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
    assert all(P.check() == 0 for P, *_ in jobs)
