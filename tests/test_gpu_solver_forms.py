"""GPU: a solve's bits do not depend on the form its iterations take.  The same partitions behind 192 empty ones are
more than the SMs, so those plans iterate in separate launches; 192 zero partials leave the lanes of every sum as they
are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle

pytestmark = pytest.mark.gpu

EMPTY = 192  # a multiple of 32, above the SMs


def _spd(A):
    return gen.shifted(A, 0.1 * float(np.abs(A.val).max()))


def _plans(A, threads, **opts):
    """(the plan of the default partition, the same one behind empty partitions)"""
    import paper_2204_06666_gb300 as eh
    ex = eh.Plan(A, host_only=1, num_sms=152, **{k: v for k, v in opts.items() if k == "slice_rows"}).export()
    pv = np.empty(A.n, np.int32)
    pv[ex["new_to_old"]] = np.repeat(np.arange(ex["nparts"]), np.diff(ex["part_ptr"]))
    opts = {"slice_rows": int(np.diff(ex["part_ptr"]).max()), **opts}
    P, Q = (eh.Plan(A, part_vec=pv + s, block_threads=threads, **opts) for s in (0, EMPTY))
    assert P.info()["nparts"] <= 152 < Q.info()["nparts"]
    return P, Q


def _same(runs):
    (x0, i0, h0), (x1, i1, h1) = runs
    assert i0["iterations"] == i1["iterations"] > 3 and i0["refinements"] == i1["refinements"]
    assert np.array_equal(h0, h1) and np.array_equal(x0, x1)


# rows of FP64 vectors: less than a vector kernel's grid, and (tet 69) more, with a last odd element
@pytest.mark.parametrize("kind,N,threads,opts", [
    ("tet", 69, 1024, {}), ("tet", 33, 256, {}), ("tet", 20, 32, {}), ("tet", 20, 96, {"ell_tpr": 2}),
    ("tet", 20, 352, {"er_layout": 2}), ("hexs", 9, 768, {"slice_rows": 729}), ("hexe", 16, 512, {}),
    ("tet", 5, 128, {}),
])
def test_cg_bits_of_both_forms(kind, N, threads, opts):
    make = {"tet": gen.tet_lap3d, "hexs": gen.hex_lap3d, "hexe": gen.hex_elast3d}
    A = _spd(make[kind](N))
    b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 3))).cuda()
    for low, refines in ((1, (0, 1, 3, 5)), (2, (4,))):
        plans = _plans(A, threads, lowp=low, **opts)
        for refine in refines:
            runs = []
            for P in plans:
                x = torch.zeros_like(b)
                st, info = P.cg(b, x, rtol=1e-9, refine=refine)
                assert st == 0, (refine, info)
                runs.append((x.cpu().numpy(), info, P.cg_history()))
            _same(runs)
        assert all(P.check() == 0 for P in plans)


# four slices a partition at most: the plans of G and G^T get 128 threads in both
@pytest.mark.parametrize("kind,N,opts", [("tet", 26, {}), ("hexs", 13, {"slice_rows": 77}),
                                         ("tet", 20, {"ell_tpr": 2})])
def test_pcg_bits_of_both_forms(kind, N, opts):
    import paper_2204_06666_gb300 as eh
    A = _spd(gen.tet_lap3d(N=N) if kind == "tet" else gen.hex_lap3d(N))
    b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 3))).cuda()
    plans = _plans(A, 256, lowp=1, **opts)
    for low in (0, 1, 2):
        Ms = [eh.Fsai(P, A, lowp=low) for P in plans]
        for refined in ((False, True) if low else (False,)):
            runs = []
            for P, M in zip(plans, Ms):
                x = torch.zeros_like(b)
                st, info = P.pcg_refined(M, b, x, rtol=1e-9) if refined else P.pcg(M, b, x, rtol=1e-9)
                assert st == 0, (low, refined, info)
                runs.append((x.cpu().numpy(), info, M.history()))
            _same(runs)
    assert all(P.check() == 0 for P in plans)
