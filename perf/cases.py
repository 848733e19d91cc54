"""Performance cases of the EHYB sparse matrix-vector library: what its users have it do, through its Python binding.

A case is a dict of plain values.  "op" is the call, "kind" and "N" (or "n", "alpha") the matrix:
  tri    2D P1 triangles, N x N nodes, 7 entries a row        tet    3D P1 tetrahedra, N^3 nodes, 15 entries a row
  hexs   3D Q1 hexahedra, scalar, 27 entries a row            hexe   3D Q1 elasticity, 3 unknowns a node, 81 a row
  power  symmetric power-law rows (n rows, exponent alpha): short rows and a few of hundreds to thousands of entries
Every matrix has its rows relabelled at random, as assembled matrices arrive; the seed gives the mesh, the
relabelling and the vectors.
"""
import math
import threading

import numpy as np
import torch

import gen
import paper_2204_06666_gb300 as eh


def listed():
    return [
        # a small 2D problem, all of it in cache: one product is launch and latency
        {"name": "spmv_tri_40k", "op": "spmv", "kind": "tri", "N": 200},
        # the two 3D workloads of the benchmark: narrow rows (diffusion) and wide rows (elasticity)
        {"name": "spmv_tet_2m", "op": "spmv", "kind": "tet", "N": 126},
        {"name": "spmv_hex_1m", "op": "spmv", "kind": "hexe", "N": 70},
        # a graph or circuit matrix: ragged rows, hubs, many entries outside their partition
        {"name": "spmv_power_200k", "op": "spmv", "kind": "power", "n": 200003, "alpha": 2.5},
        # the products of the mixed-precision solvers: FP32 values on narrow rows, BF16 values on wide ones
        {"name": "lowp_f32_tet_1m", "op": "lowp", "kind": "tet", "N": 101, "lowp": 1},
        {"name": "lowp_bf16_hex_270k", "op": "lowp", "kind": "hexe", "N": 45, "lowp": 2},
        # several right-hand sides (load cases) against one stiffness matrix
        {"name": "spmm_k8_hex_190k", "op": "spmm", "kind": "hexe", "N": 40, "k": 8},
        # many matrices of uneven size in one launch (subdomains, parameter studies)
        {"name": "batch_24", "op": "batch", "count": 24, "n_min": 5000, "n_max": 100000},
        # a whole FP64 solve of a diffusion problem to 1e-10
        {"name": "cg_tet_512k", "op": "cg", "kind": "tet", "N": 80},
        # one implicit time step of an elastic body: mixed-precision FSAI-preconditioned CG from the last state
        {"name": "pcg_step_hex_190k", "op": "pcg", "kind": "hexe", "N": 40},
        # vectors that live in host memory, streamed through one plan
        {"name": "host_stream_hex_270k", "op": "host", "kind": "hexe", "N": 45, "count": 4},
        # one training step of the knob tuner's network on the features of 2,000 matrices
        {"name": "tuner_step_2000", "op": "mlp", "rows": 2000},
    ]


# rows of the drawn matrices: from where one launch is all latency to about half of the largest listed ones
_RANGE = {"tri": (70, 1000), "tet": (18, 100), "hexs": (18, 80), "hexe": (12, 48)}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, kinds):
    kind = rng.choice(kinds)
    if kind == "power":
        return {"kind": kind, "n": _log_int(rng, 5000, 250000), "alpha": round(rng.uniform(2.0, 3.0), 2)}
    lo, hi = _RANGE[kind]
    return {"kind": kind, "N": _log_int(rng, lo, hi)}


def draw(rng):
    op = rng.choice(["spmv", "spmv", "spmv", "permuted", "lowp", "lowp", "spmm", "batch", "cg", "pcg", "host", "mlp"])
    fem, every = ["tri", "tet", "hexs", "hexe"], ["tri", "tet", "hexs", "hexe", "power"]
    if op in ("spmv", "permuted"):
        return {"op": op, **_draw_matrix(rng, every)}
    if op == "lowp":
        return {"op": op, **_draw_matrix(rng, every), "lowp": rng.choice([1, 2])}
    if op == "spmm":
        c = {"op": op, **_draw_matrix(rng, every), "k": rng.choice([2, 3, 4, 5, 8, 16, 24, 32])}
        if "N" in c:  # X and Y hold k columns each
            c["N"] = max(12, c["N"] * 2 // 3)
        return c
    if op == "batch":
        lo = _log_int(rng, 2000, 20000)
        return {"op": op, "count": rng.randint(5, 32), "n_min": lo, "n_max": lo * rng.randint(2, 6)}
    if op == "cg":
        return {"op": op, "kind": "tet", "N": _log_int(rng, 16, 72)}
    if op == "pcg":
        c = {"op": op, **_draw_matrix(rng, fem)}
        c["N"] = max(12, c["N"] * 3 // 4)
        return c
    if op == "host":
        return {"op": op, **_draw_matrix(rng, fem), "count": rng.randint(1, 6)}
    return {"op": "mlp", "rows": _log_int(rng, 150, 4000)}


# ---------------------------------------------------------------- matrices

_TAU_SHIFT = 0.1  # implicit Euler: K + c I with c = 0.1 x the mean diagonal of K


def _matrix(case, seed):
    sm, sp = 2 * seed + 1, 2 * seed + 2
    kind = case["kind"]
    if kind == "tri":
        return gen.fem2d_p1(N=case["N"], seed_mesh=sm, seed_perm=sp)
    if kind == "tet":  # zero values on the boundary for the solve, natural ones otherwise
        return gen.tet_lap3d(N=case["N"], seed_mesh=sm, seed_perm=sp, dirichlet=case["op"] == "cg")
    if kind == "hexs":
        return gen.hex_lap3d(case["N"], seed_mesh=sm, seed_perm=sp)
    if kind == "hexe":
        return gen.hex_elast3d(N=case["N"], seed_mesh=sm, seed_perm=sp)
    return gen.powerlaw_csr(case["n"], seed, case["alpha"])


def _shape(case):
    """(rows, entries) of a case's matrix; the power-law entries by their expected number."""
    kind, N = case["kind"], case.get("N", 0)
    if kind == "tri":
        return N * N, N * N + 2 * (2 * N * (N - 1) + (N - 1) ** 2)
    if kind == "tet":
        return N ** 3, N ** 3 + 2 * (3 * N * N * (N - 1) + 3 * N * (N - 1) ** 2 + (N - 1) ** 3)
    if kind in ("hexs", "hexe"):
        d = 1 if kind == "hexs" else 3
        return d * N ** 3, d * d * (3 * N - 2) ** 3
    k = np.arange(2, 5001, dtype=np.float64)
    w = k ** -case["alpha"]
    return case["n"], int(case["n"] * (1 + 2 * float((k * w).sum() / w.sum())))


def _batch_cases(case):
    """The matrices of a batch: sizes spread evenly over the logarithm, kinds in turn."""
    out = []
    for i in range(case["count"]):
        n = case["n_min"] * (case["n_max"] / case["n_min"]) ** (i / max(1, case["count"] - 1))
        kind = ("tri", "tet", "hexs", "hexe")[i % 4]
        N = n ** 0.5 if kind == "tri" else (n / 3) ** (1 / 3) if kind == "hexe" else n ** (1 / 3)
        out.append({"op": "batch", "kind": kind, "N": max(4, round(N))})
    return out


def _batch_matrices(case, seed):
    sub = _batch_cases(case)
    out = [None] * len(sub)

    def make(t, step):
        for i in range(t, len(sub), step):
            out[i] = _matrix(sub[i], 100 * seed + i)
    threads = [threading.Thread(target=make, args=(t, 8)) for t in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return out


def _vector(n, seed, lo=-1.0, hi=1.0):
    return torch.from_numpy(gen.uniform(n, seed, lo, hi))


def _mean_diagonal(A):
    rows = np.repeat(np.arange(A.n, dtype=np.int32), np.diff(A.row_ptr))
    return float(A.val[A.col == rows].mean())


def _solve_problem(case, seed):
    """(matrix, right-hand side, starting vector) of a solve, on the host."""
    A = _matrix(case, seed)
    u = _vector(A.n, 7 * seed + 5)
    if case["op"] == "cg":
        return A, _csr64(A) @ u.cuda(), torch.zeros_like(u)
    c = _TAU_SHIFT * _mean_diagonal(A)
    return gen.shifted(A, c), c * u, u


# ---------------------------------------------------------------- the calls

def _mlp_problem(case, seed):
    g = torch.Generator().manual_seed(seed)
    parts = []
    for fan_out, fan_in in ((64, 16), (64, 64), (4, 64)):  # He-uniform weights, zero biases, as tune.py starts
        b = math.sqrt(6.0 / fan_in)
        parts += [(torch.rand(fan_out * fan_in, generator=g) * 2 - 1) * b, torch.zeros(fan_out)]
    return torch.cat(parts), torch.randn(case["rows"], 16, generator=g), torch.randn(case["rows"], 4, generator=g)


def prepare(case, seed):
    op = case["op"]
    if op == "mlp":
        params, X, T = _mlp_problem(case, seed)
        return {"op": op, "net": eh.Mlp(params), "X": X.cuda(), "T": T.cuda()}
    if op == "batch":
        mats = _batch_matrices(case, seed)
        # partitions by work and at most half a block's shared memory, as plans for a batch are built
        plans = [eh.Plan(A, part_nnz=640000, smem_budget=50 * 1024) for A in mats]
        xs = [_vector(A.n, 7 * seed + i).cuda() for i, A in enumerate(mats)]
        return {"op": op, "batch": eh.Batch(plans), "xs": xs, "ys": [torch.empty_like(x) for x in xs]}
    if op == "cg":
        A, b, x0 = _solve_problem(case, seed)
        return {"op": op, "plan": eh.Plan(A), "b": b.cuda(), "x0": x0.cuda()}
    if op == "pcg":
        A, b, x0 = _solve_problem(case, seed)
        P = eh.Plan(A, lowp=1)
        return {"op": op, "plan": P, "M": eh.Fsai(P, A, lowp=2), "b": b.cuda(), "x0": x0.cuda()}
    A = _matrix(case, seed)
    if op == "spmm":
        X = _vector(A.n * case["k"], 7 * seed + 3).reshape(A.n, case["k"]).cuda()
        return {"op": op, "plan": eh.Plan(A, spmm_rhs=case["k"]), "x": X, "y": torch.empty_like(X)}
    x = _vector(A.n, 7 * seed + 3)
    if op == "host":
        xs = [_vector(A.n, 7 * seed + 3 + i).pin_memory() for i in range(case["count"])]
        return {"op": op, "plan": eh.Plan(A), "xs": xs, "ys": [torch.empty_like(x).pin_memory() for x in xs]}
    if op == "lowp":
        x = x.float().cuda()
        return {"op": op, "plan": eh.Plan(A, lowp=case["lowp"]), "x": x, "y": torch.empty_like(x)}
    x = x.cuda()
    P = eh.Plan(A)
    if op == "permuted":  # the solvers' form: the vector is carried in the plan's numbering
        xp = torch.empty_like(x)
        P.permute(True, x, xp)
        x = xp
    return {"op": op, "plan": P, "x": x, "y": torch.empty_like(x)}


def run(state):
    op = state["op"]
    if op == "spmv":
        state["plan"].spmv(state["x"], state["y"])
        return state["y"]
    if op == "permuted":
        state["plan"].spmv_permuted(state["x"], state["y"])
        return state["y"]
    if op == "lowp":
        state["plan"].spmv_lowp(state["x"], state["y"])
        return state["y"]
    if op == "spmm":
        state["plan"].spmm(state["x"], state["y"])
        return state["y"]
    if op == "batch":
        state["batch"].spmv(state["xs"], state["ys"])
        return state["ys"]
    if op == "cg":
        x = state["x0"].clone()
        state["plan"].cg(state["b"], x, rtol=1e-10)
        return x
    if op == "pcg":
        x = state["x0"].clone()
        state["plan"].pcg_refined(state["M"], state["b"], x, rtol=1e-10)
        return x
    if op == "host":
        state["plan"].spmv_host_many(state["xs"], state["ys"])
        return state["ys"]
    net = state["net"]
    loss, grad = net.loss_grad(state["X"], state["T"])
    net.adam(lr=3e-3)
    return {"loss": loss, "grad": grad, "params": net.params}


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    op = case["op"]
    if op == "mlp":
        B, p = case["rows"], 5508
        macs = 16 * 64 + 64 * 64 + 64 * 4
        # forward, weight gradients, and the input gradients of the two upper layers
        return {"bytes": 4 * (20 * B + 6 * p), "flops": 2 * B * (2 * macs + 64 * 64 + 64 * 4)}
    if op == "batch":
        shapes = [_shape(c) for c in _batch_cases(case)]
        return {"bytes": sum(10 * z + 16 * n for n, z in shapes), "flops": 2 * sum(z for _, z in shapes)}
    n, z = _shape(case)
    if op == "lowp":
        return {"bytes": (8 - 2 * case["lowp"]) * z + 8 * n, "flops": 2 * z}  # values of 4 or 2 bytes, 2-byte columns
    if op == "spmm":
        return {"bytes": 10 * z + 16 * n * case["k"], "flops": 2 * z * case["k"]}
    if op == "host":
        return {"bytes": 10 * z + 16 * n * case["count"], "flops": 2 * z * case["count"]}
    if op == "cg":  # a step reads the matrix and its two products' worth of vectors; about 3.9 N steps
        steps = int(3.9 * case["N"])
        return {"bytes": steps * (10 * z + 16 * n), "flops": steps * (2 * z + 10 * n)}
    if op == "pcg":  # A in FP32, the two triangles of G in BF16; about 20 steps
        steps = 20
        return {"bytes": steps * (6 * z + 4 * (z + n) + 8 * n), "flops": steps * (4 * z + 14 * n)}
    return {"bytes": 10 * z + 16 * n, "flops": 2 * z}


# ---------------------------------------------------------------- the same in 64 bits

def _csr64(A, val=None):
    v = torch.from_numpy(A.val if val is None else val).cuda()
    return torch.sparse_csr_tensor(torch.from_numpy(A.row_ptr).cuda(), torch.from_numpy(A.col.astype(np.int64)).cuda(),
                                   v, size=(A.n, A.n))


def _solve64(A, b):
    """Conjugate gradients, restarted on the recomputed residual until it no longer falls."""
    M = _csr64(A)
    b = b.cuda()
    x, best = torch.zeros_like(b), math.inf
    for _ in range(6):
        r = b - M @ x
        rr = float(r @ r)
        if not rr < 0.25 * best:
            break
        best, p = rr, r.clone()
        for _ in range(3000):
            q = M @ p
            a = rr / float(p @ q)
            x += a * p
            r -= a * q
            rr, old = float(r @ r), rr
            if rr <= 1e-26 * best or rr == 0.0:
                break
            p = r + (rr / old) * p
    return x


def _mlp64(case, seed):
    params, X, T = _mlp_problem(case, seed)
    p = params.double().requires_grad_()
    W1, b1, W2, b2, W3, b3 = torch.split(p, [1024, 64, 4096, 64, 256, 4])
    h = torch.relu(X.double() @ W1.reshape(64, 16).T + b1)
    h = torch.relu(h @ W2.reshape(64, 64).T + b2)
    loss = ((h @ W3.reshape(4, 64).T + b3 - T.double()) ** 2).mean()
    (g,) = torch.autograd.grad(loss, p)
    m, v = 0.1 * g, 0.001 * g * g  # the first Adam step
    new = p.detach() - 3e-3 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return {"loss": loss.detach().reshape(1), "grad": g, "params": new}


def exact(case, seed):
    op = case["op"]
    if op == "mlp":
        return _mlp64(case, seed)
    if op == "batch":
        mats = _batch_matrices(case, seed)
        return [_csr64(A) @ _vector(A.n, 7 * seed + i).cuda() for i, A in enumerate(mats)]
    if op in ("cg", "pcg"):
        A, b, _ = _solve_problem(case, seed)
        return _solve64(A, b)
    if op == "permuted":
        return None  # the numbering is the plan's own
    A = _matrix(case, seed)
    if op == "spmm":
        return _csr64(A) @ _vector(A.n * case["k"], 7 * seed + 3).reshape(A.n, case["k"]).cuda()
    if op == "host":
        M = _csr64(A)
        return [(M @ _vector(A.n, 7 * seed + 3 + i).cuda()).cpu() for i in range(case["count"])]
    x = _vector(A.n, 7 * seed + 3)
    if op == "lowp":  # the product of the values as they are stored
        val = torch.from_numpy(A.val).float()
        val = val.bfloat16() if case["lowp"] == 2 else val
        return _csr64(A, val.double().numpy()) @ x.float().double().cuda()
    return _csr64(A) @ x.cuda()
