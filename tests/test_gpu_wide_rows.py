"""GPU: rows longer than one chunk of a lane's slots (96) in the slab, in the extra rows and in both, at the edges
of the chunks.  Integer data are exact in every precision, so each path must equal the oracle; on real data every
path sums in one order, so their results must agree bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle

pytestmark = pytest.mark.gpu

EDGES = (1, 95, 96, 97, 100, 191, 192, 193, 288, 289, 500)


def _matrix(seed, integers, n=900, part=300):
    """Rows in three partitions of `part` consecutive rows; every pair of EDGES is one row's slab / extra count."""
    rng = np.random.default_rng(seed)
    lens = np.zeros((n, 2), np.int64)
    lens[:] = rng.integers(0, 6, (n, 2))
    pairs = [(a, b) for a in EDGES for b in EDGES + (0,)] + [(0, b) for b in EDGES]
    lens[rng.choice(n, len(pairs), replace=False)] = pairs
    rows, cols = [], []
    for i in range(n):
        p = i // part
        own = p * part + rng.integers(0, part, lens[i, 0])
        other = (p * part + part + rng.integers(0, n - part, lens[i, 1])) % n
        c = np.concatenate([own, other])
        rng.shuffle(c)
        rows.append(np.full(c.size, i))
        cols.append(c)
    r, c = np.concatenate(rows), np.concatenate(cols)
    v = rng.integers(-8, 9, r.size).astype(np.float64) if integers else rng.uniform(-1, 1, r.size)
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int64)
    A = gen.CSR(n, rp, c.astype(np.int32), v, "wide")
    return A, (np.arange(n) // part).astype(np.int32)


def _run(eh, A, pv, x, tpr=1, lay=0, group=0, threads=0):
    out = {}
    xd = torch.from_numpy(x).cuda()
    for low in (1, 2):
        P = eh.Plan(A, part_vec=pv, slice_rows=300, ell_tpr=tpr, er_layout=lay, lowp=low, lowp_group=group,
                    block_threads=threads)
        y32 = torch.full_like(xd.float(), np.nan)
        P.spmv_lowp(xd.float(), y32)
        out["low%d" % low] = y32.cpu().numpy()
    y, xp, yp, yn = (torch.full_like(xd, np.nan) for _ in range(4))
    P.spmv(xd, y)
    P.permute(True, xd, xp)
    P.spmv_permuted(xp, yp)
    P.permute(False, yp, yn)
    out["spmv"], out["permuted"] = y.cpu().numpy(), yn.cpu().numpy()
    P.spmv_noalloc(xd, yn)
    out["noalloc"] = yn.cpu().numpy()
    if lay == 0:
        for k in (1, 3, 8):
            X = torch.zeros(A.n, k, dtype=torch.float64, device="cuda")
            X[:, k - 1] = xd
            Y = torch.full_like(X, np.nan)
            P.spmm(X, Y)
            out["spmm%d" % k] = Y[:, k - 1].contiguous().cpu().numpy()
        y2 = [torch.full_like(xd, np.nan) for _ in range(3)]
        eh.Batch([P, P, P]).spmv([xd, 2 * xd, xd], y2)     # one plan three times: each entry its own sums
        out["batch0"], out["batch2"] = y2[0].cpu().numpy(), y2[2].cpu().numpy()
        out["batch1"] = (y2[1] / 2).cpu().numpy()
        for world in (1, 2):
            parts = []
            for r in range(world):
                S = eh.Shard(P, world, r)
                ext = torch.empty(S.n_local + S.n_halo, dtype=torch.float64, device="cuda")
                ext[:S.n_local] = xp[S.row_begin:S.row_end]
                ext[S.n_local:] = xp[torch.from_numpy(S.lists()["halo_rows"].astype(np.int64)).cuda()]
                yl = torch.full((S.n_local,), np.nan, dtype=torch.float64, device="cuda")
                S.spmv(ext, yl)
                parts.append(yl)
            P.permute(False, torch.cat(parts), yn)
            out["shard%d" % world] = yn.cpu().numpy()
    torch.cuda.synchronize()
    assert P.check() == 0
    return out


@pytest.mark.parametrize("tpr,lay,group,threads", [(1, 0, 4, 0), (1, 0, 1, 64), (2, 0, 4, 1024), (8, 0, 4, 0),
                                                   (32, 0, 1, 0), (1, 2, 4, 0), (1, 2, 1, 96)])
def test_integer_rows_exact(tpr, lay, group, threads):
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(3, True)
    x = gen.int_vector(A.n, 5)
    ref = oracle.spmv(A, x)
    for name, y in _run(eh, A, pv, x, tpr, lay, group, threads).items():
        assert np.array_equal(y.astype(np.float64), ref), name


def test_real_rows_one_order_on_every_path():
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(4, False)
    x = gen.uniform(A.n, 6)
    base = _run(eh, A, pv, x, group=4)
    for kw in ({"group": 1}, {"lay": 2, "group": 4}, {"lay": 2, "group": 1}, {"threads": 32}, {"threads": 1024}):
        for name, y in _run(eh, A, pv, x, **kw).items():
            ref = base[name] if name.startswith("low") else base["spmv"]
            assert np.array_equal(y, ref), (kw, name)
    for name, y in base.items():
        if not name.startswith("low"):
            assert np.array_equal(y, base["spmv"]), name
    k = np.diff(A.row_ptr)
    assert np.all(np.abs(base["spmv"] - oracle.spmv(A, x)) <= 2 * oracle.gamma(k + 6) * oracle.abs_spmv(A, x))


def test_solvers_on_a_power_law_matrix():
    # the fused dot products p.q (CG) and t.t (FSAI) over rows whose sums come from several chunks
    import paper_2204_06666_gb300 as eh
    A = gen.powerlaw_csr(6000, 9, 2.2, max_len=1500)
    b = torch.from_numpy(oracle.spmv(A, gen.uniform(A.n, 8))).cuda()
    P = eh.Plan(A)
    M = eh.Fsai(P, A)
    for solve in (lambda x: P.cg(b, x), lambda x: P.pcg(M, b, x)):
        xs = []
        for _ in range(2):
            x = torch.zeros_like(b)
            st, info = solve(x)
            assert st == 0 and info["relres"] <= 1e-9
            xs.append(x.cpu().numpy())
        assert np.array_equal(xs[0], xs[1])      # bit-reproducible
        r = oracle.spmv(A, xs[0]) - b.cpu().numpy()
        assert np.linalg.norm(r) <= 1e-9 * np.linalg.norm(b.cpu().numpy())
