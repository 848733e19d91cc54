"""GPU: long rows that are all alike are summed as one chain, on every path; chunks begin where the longest row has four
times the mean row's entries.  In one partition er_layout 1 has no extra rows and always sums a slab row as one chain."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import gen
import oracle
from test_gpu_wide_rows import _run

pytestmark = pytest.mark.gpu


def _matrix(lens, part, seed=5):
    """Rows of the given lengths; `part` rows a partition, half of each row's columns in its own where there are others."""
    rng = np.random.default_rng(seed)
    n = len(lens)
    cols = []
    for i, k in enumerate(lens):
        p0 = i // part * part
        own = k if part >= n else k - k // 2
        cols.append(np.concatenate([p0 + rng.integers(0, min(part, n - p0), own), rng.integers(0, n, k - own)]))
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    A = gen.CSR(n, rp, np.concatenate(cols).astype(np.int32), rng.uniform(-1, 1, int(rp[-1])), "even")
    return A, (np.arange(n) // part).astype(np.int32)


def _lens(kind, n=300):
    rng = np.random.default_rng(2)
    if kind == "same":
        return np.full(n, 97)
    if kind == "even":                       # 60 to 243, as at the faces and inside of a grid
        return rng.integers(60, 244, n)
    lens = np.full(n, 50)                    # one row of 4 times the mean, or one entry less
    k = 4 * 50 * (n - 1) / (n - 4)
    lens[n // 2] = int(np.ceil(k)) if kind == "uneven" else int(np.ceil(k)) - 1
    return lens


@pytest.mark.parametrize("kind", ("same", "even", "just even"))
def test_one_chain(kind):
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(_lens(kind), 300)
    x = gen.uniform(A.n, 6)
    xd = torch.from_numpy(x).cuda()
    ys = []
    for lay in (0, 1, 2):
        P = eh.Plan(A, part_vec=pv, slice_rows=300, er_layout=lay)
        y = torch.empty_like(xd)
        P.spmv(xd, y)
        ys.append(y.cpu().numpy())
    assert np.array_equal(ys[0], ys[1]) and np.array_equal(ys[2], ys[1])
    k = np.diff(A.row_ptr)
    assert np.all(np.abs(ys[0] - oracle.spmv(A, x)) <= 2 * oracle.gamma(k + 6) * oracle.abs_spmv(A, x))


@pytest.mark.parametrize("kind", ("same", "even", "just even", "uneven"))
def test_one_order_on_every_path(kind):
    import paper_2204_06666_gb300 as eh
    A, pv = _matrix(2 * _lens(kind), 100)    # twice the entries: both parts of the long rows are above 96
    x = gen.uniform(A.n, 6)
    base = _run(eh, A, pv, x)
    for kw in ({"group": 1}, {"lay": 2, "group": 4}, {"threads": 1024}):
        for name, y in _run(eh, A, pv, x, **kw).items():
            assert np.array_equal(y, base[name] if name.startswith("low") else base["spmv"]), (kw, name)
    for name, y in base.items():
        if not name.startswith("low"):
            assert np.array_equal(y, base["spmv"]), name
