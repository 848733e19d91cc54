"""GPU: er_layout 2, where a slice holds both parts of its rows: slices wider than one chunk (96 slots) whose rows have no
part above it, in a plan that has a wide row elsewhere.  Such a slice is one chain at its full width."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle

pytestmark = pytest.mark.gpu

PAIRS = ((49, 49), (60, 60), (96, 1), (96, 96), (1, 96), (64, 33))
N, PART = 900, 300


def _matrix(integers):
    """Three partitions of short rows; in each 64 rows of PAIRS' slab / extra counts and, in the first, one row over 96."""
    rng = np.random.default_rng(11)
    lens = rng.integers(0, 6, (N, 2))
    for p in range(3):
        pick = p * PART + rng.choice(PART, 65, replace=False)
        lens[pick[:64]] = [PAIRS[i % len(PAIRS)] for i in range(64)]
        if p == 0:
            lens[pick[64]] = (280, 300)
    rows, cols = [], []
    for i in range(N):
        p = i // PART
        own = p * PART + rng.integers(0, PART, lens[i, 0])
        other = (p * PART + PART + rng.integers(0, N - PART, lens[i, 1])) % N
        rows.append(np.full(lens[i].sum(), i))
        cols.append(np.concatenate([own, other]))
    r, c = np.concatenate(rows), np.concatenate(cols)
    v = rng.integers(-8, 9, r.size).astype(np.float64) if integers else rng.uniform(-1, 1, r.size)
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=N))]).astype(np.int64)
    return gen.CSR(N, rp, c.astype(np.int32), v, "halo wide"), (np.arange(N) // PART).astype(np.int32)


def _unflagged_wide_slices(P):
    ex = P.export()
    cin, cer = ex["row_ell_count"], ex["row_er_count"]
    found = 0
    for p in range(ex["nparts"]):
        for r0 in range(int(ex["part_ptr"][p]), int(ex["part_ptr"][p + 1]), 32):
            r = slice(r0, min(r0 + 32, int(ex["part_ptr"][p + 1])))
            found += max(cin[r].max(), cer[r].max()) <= 96 < (cin[r] + cer[r]).max()
    return found


@pytest.mark.parametrize("integers", (True, False))
@pytest.mark.parametrize("group", (1, 4))
def test_unflagged_wide_slices(integers, group):
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(integers)
    x = gen.int_vector(N, 5) if integers else gen.uniform(N, 6)
    xd = torch.from_numpy(x).cuda()
    ys = {}
    for lay in (0, 2):
        for low in (1, 2):
            P = eh.Plan(A, part_vec=pv, slice_rows=PART, er_layout=lay, lowp=low, lowp_group=group, keep_host=1)
            if lay == 2:
                assert _unflagged_wide_slices(P) > 0
            y32 = torch.full_like(xd.float(), np.nan)
            P.spmv_lowp(xd.float(), y32)
            ys[lay, "low%d" % low] = y32.cpu().numpy()
        y, xp, yp, yn = (torch.full_like(xd, np.nan) for _ in range(4))
        P.spmv(xd, y)
        P.permute(True, xd, xp)
        P.spmv_permuted(xp, yp)
        P.permute(False, yp, yn)
        ys[lay, "spmv"], ys[lay, "permuted"] = y.cpu().numpy(), yn.cpu().numpy()
        assert P.check() == 0
    for (lay, name), y in ys.items():
        if integers:  # sums of small integers: exact in every precision
            assert np.array_equal(y.astype(np.float64), oracle.spmv(A, x)), (lay, name)
        assert np.array_equal(y, ys[0, name]), (lay, name)


def test_cg_on_unflagged_wide_slices():
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(False)
    rows = np.repeat(np.arange(N), np.diff(A.row_ptr))
    # symmetric and diagonally dominant: A + A^T with the absolute row sums on the diagonal
    r, c, v = np.concatenate([rows, A.col, np.arange(N)]), np.concatenate([A.col, rows, np.arange(N)]), None
    s = np.bincount(rows, np.abs(A.val), N) + np.bincount(A.col, np.abs(A.val), N)
    v = np.concatenate([A.val, A.val, s + 1.0])
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=N))]).astype(np.int64)
    S = gen.CSR(N, rp, c[o].astype(np.int32), v[o], "spd")
    b = torch.from_numpy(oracle.spmv(S, gen.uniform(N, 3))).cuda()
    P = eh.Plan(S, part_vec=pv, slice_rows=PART, er_layout=2, keep_host=1)
    assert _unflagged_wide_slices(P) > 0
    x = torch.zeros_like(b)
    st, info = P.cg(b, x, rtol=1e-10)
    assert st == 0 and info["relres"] <= 3e-10
    r = oracle.spmv(S, x.cpu().numpy()) - b.cpu().numpy()
    assert np.linalg.norm(r) <= 3e-10 * np.linalg.norm(b.cpu().numpy())
