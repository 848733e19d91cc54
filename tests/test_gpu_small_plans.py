"""GPU: the one-slice-per-warp kernel against the general one (a plan held to 32 threads takes it), bit for bit, and
against the oracle on integers, at the edges of what a lane holds before its loops (8, 16 and 32 slab slots, 4
extra-row slots) and of the rule (8, 16, 32 and 33 slices in a partition)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle

pytestmark = pytest.mark.gpu


def _matrix(n, part, seed, integers, width=0, extra=0):
    """Partitions of `part` consecutive rows; with width / extra every row up to that many own / foreign entries."""
    rng = np.random.default_rng(seed)
    own_n = rng.integers(max(0, width - 2), width + 1, n) if width else rng.integers(0, 40, n)
    ext_n = rng.integers(max(0, extra - 1), extra + 1, n) if extra else rng.integers(0, 12, n)
    if n <= part:
        ext_n[:] = 0
    r, c = [], []
    for i in range(n):
        p0 = i // part * part
        m = min(part, n - p0)
        own = p0 + rng.integers(0, m, own_n[i])
        ext = (p0 + m + rng.integers(0, max(1, n - m), ext_n[i])) % n
        r.append(np.full(own.size + ext.size, i))
        c.append(np.concatenate([own, ext]))
    r, c = np.concatenate(r), np.concatenate(c)
    v = rng.integers(-8, 9, r.size).astype(np.float64) if integers else rng.uniform(-1, 1, r.size)
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int64)
    return gen.CSR(n, rp, c.astype(np.int32), v, "small"), (np.arange(n) // part).astype(np.int32)


def _products(eh, A, pv, x, part, **kw):
    out = {}
    xd = torch.from_numpy(x).cuda()
    for low in (1, 2):
        for group in (1, 4):
            P = eh.Plan(A, part_vec=pv, slice_rows=part, lowp=low, lowp_group=group, **kw)
            y = torch.full_like(xd.float(), np.nan)
            P.spmv_lowp(xd.float(), y)
            out[f"low{low}/{group}"] = y.cpu().numpy().astype(np.float64)
    y, xp, yp = (torch.full_like(xd, np.nan) for _ in range(3))
    P.spmv(xd, y)
    out["spmv"] = y.cpu().numpy()
    P.permute(True, xd, xp)
    P.spmv_permuted(xp, yp)
    P.permute(False, yp, y)
    out["permuted"] = y.cpu().numpy()
    buf = torch.full((A.n + 1,), np.nan, dtype=torch.float64, device="cuda")    # x and y at an odd 8-byte offset
    buf2 = torch.empty(A.n + 1, dtype=torch.float64, device="cuda")
    buf2[1:] = xd
    P.spmv(buf2[1:], buf[1:])
    out["offset"] = buf[1:].cpu().numpy()
    assert P.check() == 0
    return out


@pytest.mark.parametrize("n,part,tpr", [(1, 1, 1), (31, 31, 1), (255, 255, 1), (257, 256, 1), (2000, 257, 1),
                                        (3000, 500, 1), (3000, 512, 1), (4000, 513, 1), (5000, 1023, 1),
                                        (5000, 1024, 1), (5000, 1025, 1), (1500, 100, 4), (900, 31, 32), (700, 7, 2)])
def test_sizes(n, part, tpr):
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(n, part, n + part, True)
    x = gen.int_vector(A.n, 5)
    ref = oracle.spmv(A, x)
    for name, y in _products(eh, A, pv, x, part, ell_tpr=tpr).items():
        assert np.array_equal(y, ref), name


@pytest.mark.parametrize("part", [200, 400, 900])     # 7, 13 and 29 slices: 32, 16 and 8 slots held
@pytest.mark.parametrize("width,extra", [(1, 1), (4, 3), (7, 4), (8, 5), (9, 8), (15, 9), (16, 20), (17, 21), (31, 36),
                                         (32, 37), (33, 68), (70, 96)])
def test_widths_bit_for_bit(part, width, extra):
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(3 * part - 5, part, width, False, width, extra)
    x = gen.uniform(A.n, 7)
    small = _products(eh, A, pv, x, part)
    general = _products(eh, A, pv, x, part, block_threads=32)
    for name in small:
        assert np.array_equal(small[name], general[name]), name
    assert np.array_equal(small["spmv"], small["permuted"]) and np.array_equal(small["spmv"], small["offset"])


def test_chain_of_products_in_stream_order():
    # each product reads what the one before wrote, with the next kernel already resident: 40 in a row
    import paper_2204_06666_gb300 as eh
    A = gen.fem2d_p1(N=150)
    P, Q = eh.Plan(A), eh.Plan(A, block_threads=32)
    v = torch.from_numpy(gen.uniform(A.n, 3)).cuda()
    outs = []
    for plan in (P, Q):
        a, b = v.clone(), torch.empty_like(v)
        for _ in range(20):
            plan.spmv(a, b)
            plan.spmv(b, a)
        outs.append(a.cpu().numpy())
    assert np.array_equal(outs[0], outs[1])


def test_products_run_on_the_current_stream():
    # the binding asks torch for the current stream at every call, also after the first one
    import threading

    import paper_2204_06666_gb300 as eh
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    assert eh._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert eh._stream(None) == side.cuda_stream
        seen = []

        def look():
            with torch.cuda.stream(other):
                seen.append(eh._stream(None))
            seen.append(eh._stream(None))
        t = threading.Thread(target=look)
        t.start()
        t.join()
        assert seen == [other.cuda_stream, torch.cuda.default_stream().cuda_stream]
        assert eh._stream(None) == side.cuda_stream
    assert eh._stream(side) == side.cuda_stream and eh._stream(7) == 7
    with pytest.raises(TypeError):
        eh._dev(torch.zeros(3, dtype=torch.float32, device="cuda"), "float64")
    with pytest.raises(TypeError):
        eh._dev(torch.zeros(4, 4, dtype=torch.float64, device="cuda")[:, 1], "float64")
    with pytest.raises(TypeError):
        eh._dev(torch.zeros(3, dtype=torch.float64), "float64")
