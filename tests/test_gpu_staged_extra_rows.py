"""GPU: FP32 / BF16 products whose extra rows read x staged at their columns (plans in which a column serves many
slots), bit for bit against the column-major copies, which gather; at the rule's edge and in the solvers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle

pytestmark = pytest.mark.gpu


def _slots_per_column(eh, A, **kw):
    e = eh.Plan(A, host_only=1, num_sms=152, smem_budget=231424, lowp=1, **kw).export()
    ptr = e["er_slice_pos"][e["slice_ptr"]]
    cols = sum(np.unique(e["er_scol"][a:b]).size for a, b in zip(ptr[:-1], ptr[1:]))
    return ptr[-1] / max(1, cols)


# partitions of more than 32 slices (fewer take the one-slice-per-warp kernel); slots per column on either side of 10
CASES = [("hexe", 20, 1500, 1), ("hexe", 20, 1031, 1), ("hexe", 24, 3300, 1), ("hexe", 20, 1500, 2), ("hexs", 36, 1500, 1)]


@pytest.mark.parametrize("kind,N,rows,tpr", CASES)
def test_staged_equals_gathered(kind, N, rows, tpr):
    import paper_2204_06666_gb300 as eh
    A = gen.hex_elast3d(N=N) if kind == "hexe" else gen.hex_lap3d(N)
    shared = _slots_per_column(eh, A, slice_rows=rows, ell_tpr=tpr)
    assert (shared >= 10) == (kind == "hexe"), shared
    x = torch.from_numpy(gen.uniform(A.n, 5)).cuda().float()
    for low in (1, 2):
        out = {}
        for group in (1, 4):
            P = eh.Plan(A, slice_rows=rows, lowp=low, lowp_group=group, ell_tpr=tpr)
            y = torch.full_like(x, np.nan)
            P.spmv_lowp(x, y)
            buf, buf2 = torch.full((A.n + 1,), np.nan, device="cuda"), torch.empty(A.n + 1, device="cuda")
            buf2[1:] = x                                 # x and y at an odd 4-byte offset
            P.spmv_lowp(buf2[1:], buf[1:])
            out[group] = y.cpu().numpy()
            assert np.array_equal(out[group], buf[1:].cpu().numpy()) and P.check() == 0
        assert np.array_equal(out[1], out[4]), low


def test_solvers_with_staged_extra_rows():
    import paper_2204_06666_gb300 as eh
    A = gen.hex_elast3d(N=20, clamp_minz=True)
    A = gen.shifted(A, 0.05 * float(np.abs(A.val).max()))
    b_np = oracle.spmv(A, gen.uniform(A.n, 3))
    b = torch.from_numpy(b_np).cuda()
    assert _slots_per_column(eh, A, slice_rows=1500) >= 10
    its = {}
    for group in (1, 4):                                 # gathered, staged
        P = eh.Plan(A, slice_rows=1500, lowp=1, lowp_group=group)
        for refine in (1, 3, 5):
            x = torch.zeros_like(b)
            st, info = P.cg(b, x, rtol=1e-10, refine=refine)
            assert st == 0
            r = oracle.spmv(A, x.cpu().numpy()) - b_np
            assert np.linalg.norm(r) <= 3e-10 * np.linalg.norm(b_np)
            its[group, refine] = (info["iterations"], x.cpu().numpy())
    for refine in (1, 3, 5):                             # the same products, summed in the same order
        assert its[1, refine][0] == its[4, refine][0] and np.array_equal(its[1, refine][1], its[4, refine][1])
    P = eh.Plan(A, slice_rows=1500, lowp=1)
    for low in (1, 2):
        M = eh.Fsai(P, A, lowp=low)
        for refined in (False, True):
            xs = []
            for _ in range(2):
                x = torch.zeros_like(b)
                st, info = P.pcg_refined(M, b, x, rtol=1e-10) if refined else P.pcg(M, b, x, rtol=1e-10)
                assert st == 0, (low, refined, info)
                xs.append(x.cpu().numpy())
            r = oracle.spmv(A, xs[0]) - b_np
            assert np.array_equal(xs[0], xs[1]) and np.linalg.norm(r) <= 3e-10 * np.linalg.norm(b_np)
