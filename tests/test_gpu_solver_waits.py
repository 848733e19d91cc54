"""GPU: the waits of the solvers' cooperative kernels.  With one arrival missing (a counter that starts one too low) the
first wait runs out after wait_timeout_ns, every block leaves and the call reports it; the context stays usable.  The same
hook shows which form a plan's iterations take: separate launches have no such wait."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle
from test_gpu_persistent_solvers import CASES, _matrix

pytestmark = pytest.mark.gpu

LIMIT = 100_000_000  # the least with which solvers iterate persistently


def _timed_out(eh, call):
    t = time.perf_counter()
    try:
        call()
    except eh.EhybError as e:
        assert e.status == eh.EHYB_ERR_TIMEOUT
        assert time.perf_counter() - t < 1.5  # the limit is 0.1 s
        return True
    return False


@pytest.mark.parametrize("inject", (2, 3))
def test_wait_that_runs_out(inject):
    import paper_2204_06666_gb300 as eh
    A = gen.tet_lap3d(N=20)
    b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 3))).cuda()
    P = eh.Plan(A, lowp=1, inject_wait_fault=inject, wait_timeout_ns=LIMIT)
    Ms = [eh.Fsai(P, A, lowp=low) for low in (0, 2)]
    calls = [lambda x, r=r: P.cg(b, x, refine=r) for r in (0, 1, 3)]
    calls += [lambda x, M=M: P.pcg(M, b, x) for M in Ms] + [lambda x: P.pcg_refined(Ms[1], b, x)]
    for call in calls:
        x = torch.full_like(b, 0.5)
        assert _timed_out(eh, lambda: call(x))
        assert torch.all(x == 0.5)              # nothing is written
        assert P.check() == eh.EHYB_ERR_TIMEOUT and P.check() == 0
    # the products of the same plan, and another plan's solves
    y = torch.empty_like(b)
    P.spmv(b, y)
    assert np.allclose(y.cpu().numpy(), oracle.spmv(A, b.cpu().numpy()), rtol=1e-12, atol=1e-12)
    Q = eh.Plan(A, lowp=1)
    x = torch.zeros_like(b)
    assert Q.cg(b, x)[0] == 0 and Q.check() == 0


# a few large partitions (or more than the SMs) are left to the separate launches, and so is every plan with a shorter limit
SEPARATE = ("x in memory", "q, r and x in memory", "more partitions than SMs")


@pytest.mark.parametrize("name", list(CASES))
def test_form_of_each_case(name):
    import paper_2204_06666_gb300 as eh
    A, opts = _matrix(name)
    b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 3))).cuda()
    for limit, persistent in ((LIMIT, name not in SEPARATE), (LIMIT - 1, False)):
        P = eh.Plan(A, inject_wait_fault=2, wait_timeout_ns=limit, **opts)
        assert _timed_out(eh, lambda: P.cg(b, torch.zeros_like(b))) == persistent


# four FP64 vectors of a partition: x, r and x, and all but p too large for the shared memory
@pytest.mark.parametrize("N,rows", [(33, 3000), (33, 3600), (105, 0)])
def test_cg_bits_at_each_placement(N, rows):
    import paper_2204_06666_gb300 as eh
    A = gen.tet_lap3d(N=N)
    A = gen.shifted(A, 0.1 * float(np.abs(A.val).max()))
    b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 3))).cuda()
    runs = []
    for kw in ({}, {"wait_timeout_ns": LIMIT - 1}, {"wait_timeout_ns": LIMIT, "inject_wait_fault": 2}):
        P = eh.Plan(A, slice_rows=rows, block_threads=1024, **kw)
        x = torch.zeros_like(b)
        if "inject_wait_fault" in kw:
            assert _timed_out(eh, lambda: P.cg(b, x))
            break
        st, info = P.cg(b, x, rtol=1e-10)
        assert st == 0
        runs.append((x.cpu().numpy(), info["iterations"], P.cg_history()))
    assert runs[0][1] == runs[1][1] and all(np.array_equal(runs[0][k], runs[1][k]) for k in (0, 2))


# the forms against each other where the plans of G and G^T have many warps
@pytest.mark.parametrize("kind,N,opts", [("hexe", 24, {}), ("tet", 45, {}), ("tet", 33, {"ell_tpr": 2}),
                                         ("tet", 36, {"slice_rows": 5700})])
def test_bits_with_and_without_cooperative_kernels(kind, N, opts):
    import paper_2204_06666_gb300 as eh
    A = gen.tet_lap3d(N=N) if kind == "tet" else gen.hex_elast3d(N=N)
    A = gen.shifted(A, 0.1 * float(np.abs(A.val).max()))
    b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 3))).cuda()
    plans = [eh.Plan(A, lowp=1, wait_timeout_ns=w, **opts) for w in (0, LIMIT - 1)]
    for low in (0, 1, 2):
        Ms = [eh.Fsai(P, A, lowp=low) for P in plans]
        for refined in ((False, True) if low else (False,)):
            xs = []
            for P, M in zip(plans, Ms):
                x = torch.zeros_like(b)
                st, info = P.pcg_refined(M, b, x, rtol=1e-9) if refined else P.pcg(M, b, x, rtol=1e-9)
                assert st == 0, (low, refined, info)
                xs.append((x.cpu().numpy(), info["iterations"], M.history()))
            assert xs[0][1] == xs[1][1] and all(np.array_equal(xs[0][k], xs[1][k]) for k in (0, 2)), (low, refined)
