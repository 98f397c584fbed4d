"""The workloads this library's speed is measured on.

Each case is one call a program makes through the public entry points: a
sparse product (whole, by row blocks, stacked in a graph, with gradients), a
graph contraction, a Markov-clustering expansion or step, a pruned GNN layer
with its backward, or bulk neighbourhood sampling. Inputs are synthetic
graphs built on the GPU from a seed: Erdos-Renyi and R-MAT graphs with the
degrees, skew and values of the library's own generators (gen.py).

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the inputs, plan and workspace a program keeps
    run(state)          one pass
    work(case)          bytes and flops of one pass that no method avoids
    exact(case, seed)   what run returns, in 64 bits, by plain torch
"""
import math
import zlib

import torch

from paper_2512_12036_gb300 import autograd, gnn, mcl, sampling
from paper_2512_12036_gb300.api import DeviceCSR, Plan
from paper_2512_12036_gb300.batched import BatchedSpGEMM

RMAT = (0.57, 0.19, 0.19)      # a, b, c of every R-MAT graph
CHUNK = 1 << 26                # products per step of exact()


def listed():
    return [
        # one small product: a 4096-vertex graph squared, where latency and
        # launches are what a caller sees
        dict(name="er4096_square", kind="product", graph="er", n=4096, degree=8.0, square=True),
        # requests as a service gets them: A*B with unrelated operands, an even
        # graph of ragged size and a skewed one
        dict(name="request_er", kind="product", graph="er", n=100003, degree=16.0, square=False),
        dict(name="request_rmat", kind="product", graph="rmat", n=300007, degree=20.0, square=False),
        # a skewed graph squared with the default plan: hub rows of every tier
        dict(name="rmat15_square", kind="product", graph="rmat", n=32768, degree=28.0, square=True),
        # a share of the rows of a 2^20-vertex graph squared, in the row-block
        # form with the row bitmap cache that products of this size use
        dict(name="rmat20_rows", kind="rows", n=1 << 20, degree=32.0, stride=32, cache_mb=1536),
        # graph contraction S^T * A * S
        dict(name="contract_rmat18", kind="contraction", n=1 << 18, degree=30.0, clusters=16384),
        # Markov clustering: an expansion of a pruned matrix, and the step
        # (prune, top-k, inflate, normalise) after an expansion
        dict(name="mcl_expand", kind="expansion", n=1 << 17, per_row=32),
        dict(name="mcl_step", kind="mcl_step", n=50021, mean_len=600.0, k=32, order=0),
        # GNN aggregation A*X over a batch of subgraphs: replayed as a graph in
        # inference, with both gradients in training
        dict(name="gnn_batch_replay", kind="batch", graphs=256, features=256, k=32),
        dict(name="gnn_batch_grad", kind="batch_grad", graphs=1024, features=256, k=32),
        # one pruned GCN layer, forward and backward (features 256 -> 256)
        dict(name="gcn_layer", kind="layer", graphs=512, d_in=256, d_out=256, k=32),
        # bulk neighbourhood sampling for mini-batches, two layers
        dict(name="sample_rmat19", kind="sample", n=1 << 19, degree=30.0, batch=65536, fanout1=25,
             fanout2=10, mode=sampling.UNIFORM),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["product", "product", "product", "rows", "contraction", "expansion",
                       "mcl_step", "batch", "batch_grad", "layer", "sample"])
    if kind == "product":
        if rng.random() < 0.5:
            return dict(kind=kind, graph="er", n=int(_log(rng, 1000, 300000)),
                        degree=round(rng.uniform(4, 32), 2), square=rng.random() < 0.5)
        if rng.random() < 0.5:
            return dict(kind=kind, graph="rmat", n=int(_log(rng, 1000, 40000)),
                        degree=round(rng.uniform(4, 28), 2), square=True)
        return dict(kind=kind, graph="rmat", n=int(_log(rng, 1000, 300000)),
                    degree=round(rng.uniform(4, 20), 2), square=False)
    if kind == "rows":
        n = int(_log(rng, 1 << 18, 1 << 20))
        return dict(kind=kind, n=n, degree=round(rng.uniform(16, 32), 2),
                    stride=rng.randint(33, 160), cache_mb=1536)
    if kind == "contraction":
        n = int(_log(rng, 1 << 14, 1 << 18))
        return dict(kind=kind, n=n, degree=round(rng.uniform(8, 30), 2), clusters=max(64, n // rng.randint(8, 32)))
    if kind == "expansion":
        return dict(kind=kind, n=int(_log(rng, 1 << 13, 1 << 17)), per_row=rng.randint(8, 32))
    if kind == "mcl_step":
        return dict(kind=kind, n=int(_log(rng, 2000, 50000)), mean_len=round(_log(rng, 60, 600), 1),
                    k=rng.randint(8, 64), order=rng.randint(0, 1))
    if kind == "batch":
        return dict(kind=kind, graphs=int(_log(rng, 16, 256)), features=rng.choice([64, 100, 128, 256, 300]),
                    k=rng.randint(8, 32))
    if kind == "batch_grad":
        return dict(kind=kind, graphs=int(_log(rng, 32, 1024)), features=rng.choice([64, 100, 128, 256]),
                    k=rng.randint(8, 32))
    if kind == "layer":
        return dict(kind=kind, graphs=int(_log(rng, 16, 512)), d_in=rng.choice([64, 100, 128, 256]),
                    d_out=rng.choice([16, 47, 64, 128, 256]), k=rng.randint(8, 32))
    return dict(kind=kind, n=int(_log(rng, 1 << 15, 1 << 19)), degree=round(rng.uniform(8, 30), 2),
                batch=int(_log(rng, 1024, 65536)), fanout1=rng.randint(5, 25), fanout2=rng.randint(5, 10),
                mode=rng.randint(0, 2))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _base(case):
    """The generator of a case's structure: the same for every seed, so that results of a case have
    one shape. A seed then draws the labels of the vertices (and so every index and the order of
    every row) and the values."""
    text = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    return _gen(zlib.crc32(text.encode()))


def _uniform(g, n):
    """fp32 values in (0, 1]."""
    return 1.0 - torch.rand(n, generator=g, device="cuda")


def _perm(g, n):
    return torch.randperm(n, generator=g, device="cuda")


def _rows_of(A):
    rp = A.row_ptr.long()
    return torch.repeat_interleave(torch.arange(A.rows, device="cuda"), rp[1:] - rp[:-1])


def _from_keys(rows, cols, key, val):
    """CSR from sorted distinct keys row * cols + col."""
    row = torch.div(key, cols, rounding_mode="floor")
    rp = torch.searchsorted(row, torch.arange(rows + 1, device="cuda")).to(torch.int32)
    return DeviceCSR(rows, cols, rp, (key - row * cols).to(torch.int32), val)


def _relabel(M, to_row, to_col, val, rows=None, cols=None):
    """M with row r as row to_row[r] and column c as column to_col[c]; val[q] goes with entry q."""
    rows, cols = rows or M.rows, cols or M.cols
    key, order = torch.sort(to_row[_rows_of(M)] * cols + to_col[M.col.long()])
    return _from_keys(rows, cols, key, val[order])


def _normalised(M):
    """M with every row divided by its sum (by magnitude)."""
    row = _rows_of(M)
    M.val = M.val / torch.zeros(M.rows, dtype=torch.float64, device="cuda").index_add_(0, row, M.val.double()).float()[row]
    return M


def _symmetric(n, u, v):
    """The undirected edges u-v, loops and repeats dropped, both ways."""
    key = (torch.minimum(u, v) * n + torch.maximum(u, v))[u != v]
    key = torch.unique(key)
    lo = torch.div(key, n, rounding_mode="floor")
    key, _ = torch.sort(torch.cat([key, (key - lo * n) * n + lo]))
    return _from_keys(n, n, key, None)


def _er(n, degree, g):
    m = int(n * degree / 2)
    u = torch.randint(n, (m,), generator=g, device="cuda")
    v = torch.randint(n, (m,), generator=g, device="cuda")
    return _symmetric(n, u, v)


def _rmat_edges(n, m, g):
    """About m directed R-MAT edges on n vertices (those of 2^k >= n vertices that lie below n)."""
    a, b, c = RMAT
    scale = max(1, math.ceil(math.log2(n)))
    draw_n = m if n == 1 << scale else int(m * 1.15)
    u = torch.zeros(draw_n, dtype=torch.int64, device="cuda")
    v = torch.zeros(draw_n, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = torch.rand(draw_n, generator=g, device="cuda")
        u = 2 * u + (r >= a + b)
        v = 2 * v + (((r >= a) & (r < a + b)) | (r >= a + b + c))
    keep = (u < n) & (v < n)
    return u[keep][:m], v[keep][:m]


def _rmat(n, degree, g):
    return _symmetric(n, *_rmat_edges(n, int(n * degree / 2), g))


def _some_rows(A, count, base):
    """The structure of `count` rows of A, drawn at random."""
    rp = A.row_ptr.long()
    pick = _perm(base, A.rows)[:count]
    lens = rp[pick + 1] - rp[pick]
    out = torch.zeros(pick.numel() + 1, dtype=torch.int64, device="cuda")
    out[1:] = torch.cumsum(lens, 0)
    at = torch.repeat_interleave(rp[pick] - out[:-1], lens) + torch.arange(int(out[-1]), device="cuda")
    return DeviceCSR(pick.numel(), A.cols, out.to(torch.int32), A.col[at].clone(), None)


def _stochastic(n, per_row, g):
    """The structure of a pruned Markov matrix: up to per_row entries a row, popular columns drawn
    more often, and the diagonal."""
    _, v = _rmat_edges(n, n * per_row, g)
    row = _perm(g, n * per_row)[: v.numel()] % n
    diag = torch.arange(n, device="cuda")
    return _from_keys(n, n, torch.unique(torch.cat([row * n + v, diag * n + diag])), None)


def _expanded(n, mean_len, g):
    """A Markov matrix after an expansion: log-normal row lengths, a few large values a row."""
    sigma = 1.2
    lens = torch.exp(torch.randn(n, generator=g, device="cuda") * sigma + math.log(mean_len) - sigma ** 2 / 2)
    lens = lens.clamp(1, n // 2).long()
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)
    key = torch.unique(row * n + torch.randint(n, (row.numel(),), generator=g, device="cuda"))
    return _normalised(_from_keys(n, n, key, _uniform(g, key.numel()) ** 4))


def _subgraphs(graphs, g):
    """The structure of `graphs` Erdos-Renyi subgraphs with self-loops as one block-diagonal matrix,
    n log-uniform in [64, 2048], average degree in [4, 32]; and the subgraph of every vertex."""
    r = torch.rand(2, graphs, generator=g, device="cuda", dtype=torch.float64)
    sizes = torch.exp(math.log(64) + r[0] * math.log(32)).long()
    want = (sizes * (4 + 28 * r[1]) / 2).long()
    off = torch.cumsum(sizes, 0) - sizes
    n = int(sizes.sum())
    of = torch.repeat_interleave(torch.arange(graphs, device="cuda"), want)
    r = torch.rand(2, of.numel(), generator=g, device="cuda", dtype=torch.float64)
    u, v = ((r * sizes[of]).long() + off[of]).unbind(0)
    diag = torch.arange(n, device="cuda")
    lo, hi = torch.minimum(u, v), torch.maximum(u, v)
    key = torch.unique(torch.cat([lo * n + hi, hi * n + lo, diag * n + diag]))
    return _from_keys(n, n, key, None), torch.repeat_interleave(torch.arange(graphs, device="cuda"), sizes)


def _normalised_batch(case, g):
    """A_hat = D^-1/2 (A + I) D^-1/2 of the case's subgraphs, the vertices of each relabelled."""
    base = _base(case)
    A, of = _subgraphs(case["graphs"], base)
    _, order = torch.sort(of.double() + torch.rand(A.rows, generator=g, device="cuda", dtype=torch.float64) * 0.99)
    to = torch.empty_like(order)
    to[order] = torch.arange(A.rows, device="cuda")
    deg = (A.row_ptr[1:] - A.row_ptr[:-1]).double()
    return _relabel(A, to, to, (deg[_rows_of(A)] * deg[A.col.long()]).rsqrt().float()), to, base


def _topk_features(n, features, k, base):
    """The k largest of `features` normal values in every row, as CSR."""
    k = min(k, features)
    cols, vals = [], []
    for r0 in range(0, n, 1 << 18):
        X = torch.randn(min(n - r0, 1 << 18), features, generator=base, device="cuda")
        c, _ = torch.sort(torch.topk(X, k, dim=1).indices, dim=1)
        cols.append(c.to(torch.int32))
        vals.append(torch.gather(X, 1, c))
    rp = torch.arange(0, n * k + 1, k, dtype=torch.int32, device="cuda")
    return DeviceCSR(n, features, rp, torch.cat(cols).reshape(-1), torch.cat(vals).reshape(-1))


def _operands(case, seed):
    """The sparse operands of a case, and what else it needs."""
    g, kind, n = _gen(seed), case["kind"], case.get("n")
    if kind == "product":
        make, base = _rmat if case["graph"] == "rmat" else _er, _base(case)
        A, p, q = make(n, case["degree"], base), _perm(g, n), _perm(g, n)
        if case["square"]:
            A = _relabel(A, p, p, _uniform(g, A.nnz))
            return A, A
        B = make(n, case["degree"], base)
        # the popular vertices of the two graphs have nothing to do with each other
        A = _relabel(A, p, q, _uniform(g, A.nnz))
        return A, _relabel(B, q[_perm(base, n)], _perm(g, n), _uniform(g, B.nnz))
    if kind == "rows":
        base = _base(case)
        B = _rmat(n, case["degree"], base)
        A, p = _some_rows(B, n // case["stride"], base), _perm(g, n)
        return (_relabel(A, _perm(g, A.rows), p, _uniform(g, A.nnz)), _relabel(B, p, p, _uniform(g, B.nnz)))
    if kind == "contraction":
        base, m = _base(case), case["clusters"]
        A = _rmat(n, case["degree"], base)
        lab, p = torch.randint(m, (n,), generator=base, device="cuda"), _perm(g, n)
        A = _relabel(A, p, p, _uniform(g, A.nnz))
        lab = _perm(g, m)[lab][torch.argsort(p)]
        one = torch.ones(n, device="cuda")
        S = DeviceCSR(n, m, torch.arange(n + 1, dtype=torch.int32, device="cuda"), lab.to(torch.int32), one)
        key, _ = torch.sort(lab * n + torch.arange(n, device="cuda"))
        return A, S, _from_keys(m, n, key, one.clone()), lab
    if kind == "expansion":
        M, p = _stochastic(n, case["per_row"], _base(case)), _perm(g, n)
        M = _normalised(_relabel(M, p, p, _uniform(g, M.nnz) ** 2 + 1e-3))
        return M, M
    if kind == "mcl_step":
        E = _expanded(n, case["mean_len"], _base(case))
        return (_relabel(E, _perm(g, n), _perm(g, n), E.val),)
    if kind in ("batch", "batch_grad"):
        A, to, base = _normalised_batch(case, g)
        X = _topk_features(A.rows, case["features"], case["k"], base)
        X = _relabel(X, to, _perm(g, X.cols), X.val * (0.9 + 0.2 * torch.rand(X.nnz, generator=g, device="cuda")))
        if kind == "batch":
            return A, X
        # the gradient that comes from the layers above, long enough for any C
        return A, X, torch.randn(A.rows * X.cols, generator=g, device="cuda")
    if kind == "layer":
        A, _, _ = _normalised_batch(case, g)
        return (A, torch.randn(A.rows, case["d_in"], generator=g, device="cuda"),
                torch.randn(case["d_in"], case["d_out"], generator=g, device="cuda") / case["d_in"] ** 0.5,
                torch.randn(A.rows, case["d_out"], generator=g, device="cuda"))
    if kind == "sample":
        # vertices without an edge lie between the others, at places that the seed draws: the order
        # inside every row stays, and so does how many columns the draws of a row hit
        base, m = _base(case), int(n * 0.9)
        A = _rmat(m, case["degree"], base)
        val, verts = _uniform(base, A.nnz), _perm(base, m)[: case["batch"]]
        A = _relabel(A, *[p := _perm(base, m)] * 2, val)
        at, _ = torch.sort(_perm(g, n)[:m])
        return _relabel(A, at, at, A.val, n, n), at[p[verts]].cpu().numpy()
    raise ValueError(kind)


def prepare(case, seed):
    ops, kind = _operands(case, seed), case["kind"]
    state = {"kind": kind, "case": case, "ops": ops}
    if kind == "rows":
        state["plan"] = Plan(row_cache_mb=case["cache_mb"])
        state["ws"] = state["plan"].workspace(*ops)
    elif kind == "batch":
        state["batch"] = BatchedSpGEMM(*ops)
        state["batch"].capture()
    else:
        state["plan"] = Plan()
    if kind == "batch_grad":
        state["a"] = ops[0].val.clone().requires_grad_(True)
        state["x"] = ops[1].val.clone().requires_grad_(True)
    if kind == "layer":
        state["X"] = ops[1].clone().requires_grad_(True)
        state["W"] = ops[2].clone().requires_grad_(True)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _out(C):
    return {"row_ptr": C.row_ptr, "col": C.col, "val": C.val}


def run(state):
    kind, ops, case = state["kind"], state["ops"], state["case"]
    if kind in ("product", "expansion"):
        return _out(state["plan"].spgemm(*ops))
    if kind == "rows":
        blocks, _, _ = state["plan"].spgemm_blocks(*ops, ws=state["ws"])
        return [_out(C) for _, _, C in blocks]
    if kind == "contraction":
        A, S, St, _ = ops
        return _out(state["plan"].spgemm(state["plan"].spgemm(St, A), S))
    if kind == "mcl_step":
        return _out(mcl.mcl_step(state["plan"], ops[0], 1e-4, case["k"], 2.0, case["order"]))
    if kind == "batch":
        state["batch"].run()
        return _out(state["batch"].result())
    if kind == "batch_grad":
        A, X, dC = ops
        C = autograd.spgemm(state["a"], state["x"], A, X, state["plan"])
        dA, dX = torch.autograd.grad(C.val, (state["a"], state["x"]), grad_outputs=dC[: C.nnz])
        return dict(_out(C), dA=dA, dX=dX)
    if kind == "layer":
        Y = gnn.pruned_aggregation(ops[0], state["X"], state["W"], case["k"], state["plan"])
        dX, dW = torch.autograd.grad(Y, (state["X"], state["W"]), grad_outputs=ops[3])
        return {"Y": Y, "dX": dX, "dW": dW}
    if kind == "sample":
        adj, qs, _ = sampling.sample_layers(ops[0], ops[1], [case["fanout1"], case["fanout2"]],
                                            state["plan"], mode=case["mode"], seed=0)
        return {"adj": [_out(a) for a in adj], "frontier": [q.col for q in qs]}
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# the least work of a pass
# ---------------------------------------------------------------------------

def _lens(M):
    rp = M.row_ptr.long()
    return rp[1:] - rp[:-1]


def _products(A, B):
    """Products per row of A*B."""
    ip = torch.zeros(A.rows + 1, dtype=torch.int64, device="cuda")
    ip[1:] = torch.cumsum(torch.bincount(_rows_of(A), _lens(B)[A.col.long()].double(), A.rows).long(), 0)
    return ip[1:] - ip[:-1]


def _expected_nnz(A, B):
    """Distinct columns of A*B if each row's products fell on B's columns by their counts."""
    ip = _products(A, B).double()
    pop, mult = torch.unique(torch.bincount(B.col.long(), minlength=B.cols), return_counts=True)
    pop = pop.double() / max(1, B.nnz)
    at = torch.logspace(0, math.log10(float(ip.max().clamp(min=2))), 64, dtype=torch.float64, device="cuda")
    f = (mult * (1 - torch.exp(-at[:, None] * pop))).sum(1)
    q = torch.searchsorted(at, ip.clamp(min=1)).clamp(1, 63)
    t = (ip - at[q - 1]) / (at[q] - at[q - 1])
    return float(((f[q - 1] + t * (f[q] - f[q - 1])) * (ip > 0)).sum())


def _csr_bytes(M):
    return 8 * M.nnz + 4 * (M.rows + 1)


def work(case):
    ops, kind = _operands(case, 1), case["kind"]
    if kind in ("product", "expansion", "rows", "batch", "batch_grad"):
        A, B = ops[:2]
        ip, nnz = float(_products(A, B).sum()), _expected_nnz(A, B)
        read = _csr_bytes(A) + (0 if A is B else _csr_bytes(B))
        w = {"bytes": read + 8 * nnz + 4 * (A.rows + 1), "flops": 2 * ip}
        if kind == "batch_grad":          # also dC in, dA and dX out, two products per product
            w = {"bytes": w["bytes"] + 4 * (nnz + A.nnz + B.nnz), "flops": 3 * w["flops"]}
        return w
    if kind == "contraction":
        A, S, St, lab = ops
        return {"bytes": _csr_bytes(A) + 2 * _csr_bytes(S) + 8 * A.nnz, "flops": 4.0 * A.nnz}
    if kind == "mcl_step":
        kept = float(_lens(ops[0]).clamp(max=case["k"]).sum())
        return {"bytes": _csr_bytes(ops[0]) + 8 * kept + 4 * case["n"], "flops": ops[0].nnz + 3 * kept}
    if kind == "layer":
        A, X, W, dY = ops
        spm = 2.0 * A.nnz * min(case["k"], case["d_in"])
        return {"bytes": 2 * _csr_bytes(A) + 4.0 * (2 * X.numel() + 2 * dY.numel() + 3 * W.numel()),
                "flops": 2 * spm + 3 * 2.0 * A.rows * W.numel()}
    A, verts = ops
    deg = _lens(A)[torch.from_numpy(verts).cuda()].double()
    drawn = float(deg.clamp(max=case["fanout1"]).sum())
    # the rows of A around the batch and around the first layer's vertices
    near = float(deg.sum()) + min(drawn, case["n"]) * A.nnz / case["n"]
    return {"bytes": 8 * near + 16.0 * drawn, "flops": near}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------

def _expand(A, B, j0, j1):
    """All products of A's entries [j0, j1): (A entry, B entry) index pairs."""
    rp = B.row_ptr.long()
    k = A.col[j0:j1].long()
    lens = rp[k + 1] - rp[k]
    off = torch.cumsum(lens, 0) - lens
    ja = torch.repeat_interleave(torch.arange(j0, j1, device="cuda"), lens)
    return ja, torch.arange(ja.numel(), device="cuda") + torch.repeat_interleave(rp[k] - off, lens)


def _row_chunks(A, B):
    csum = torch.cumsum(_products(A, B), 0).cpu()
    r0, base = 0, 0
    while r0 < A.rows:
        r1 = max(r0 + 1, int(torch.searchsorted(csum, base + CHUNK, right=True)))
        yield r0, min(r1, A.rows)
        r0, base = r1, int(csum[min(r1, A.rows) - 1])


def _product64(A, B):
    """Sorted structure and fp64 values of A*B."""
    rp, rows, cols, vals = A.row_ptr.long().cpu(), _rows_of(A), [], []
    counts = torch.zeros(A.rows, dtype=torch.int64, device="cuda")
    for r0, r1 in _row_chunks(A, B):
        ja, tb = _expand(A, B, int(rp[r0]), int(rp[r1]))
        a, b = A.val[ja].double(), B.val[tb].double()
        key, order = torch.sort(rows[ja] * B.cols + B.col[tb])
        key, inv = torch.unique_consecutive(key, return_inverse=True)
        vals.append(torch.zeros(key.numel(), dtype=torch.float64, device="cuda").index_add_(0, inv, (a * b)[order]))
        row = torch.div(key, B.cols, rounding_mode="floor")
        cols.append((key - row * B.cols).to(torch.int32))
        counts += torch.bincount(row, minlength=A.rows)
    out = torch.zeros(A.rows + 1, dtype=torch.int64, device="cuda")
    out[1:] = torch.cumsum(counts, 0)
    return {"row_ptr": out.to(torch.int32), "col": torch.cat(cols), "val": torch.cat(vals)}


def _csr64(M, val=None):
    v = (M.val if val is None else val).double()
    return torch.sparse_csr_tensor(M.row_ptr.long(), M.col.long(), v, (M.rows, M.cols))


def _transposed(A):
    key, order = torch.sort(A.col.long() * A.rows + _rows_of(A))
    return _from_keys(A.cols, A.rows, key, A.val[order])


def _dense64(X, val=None):
    D = torch.zeros(X.rows, X.cols, dtype=torch.float64, device="cuda")
    D[_rows_of(X), X.col.long()] = X.val.double() if val is None else val
    return D


def _row_dots(A, L, R):
    """sum_c L[i, c] * R[k, c] for every entry (i, k) of A."""
    rows, out = _rows_of(A), []
    for j in range(0, A.nnz, 1 << 19):
        out.append((L[rows[j: j + (1 << 19)]] * R[A.col[j: j + (1 << 19)].long()]).sum(1))
    return torch.cat(out)


def exact(case, seed):
    ops, kind = _operands(case, seed), case["kind"]
    if kind in ("product", "expansion"):
        return _product64(*ops)
    if kind == "rows":
        return [_product64(*ops)]
    if kind == "contraction":
        A, _, _, lab = ops
        m = case["clusters"]
        key, inv = torch.unique(lab[_rows_of(A)] * m + lab[A.col.long()], return_inverse=True)
        val = torch.zeros(key.numel(), dtype=torch.float64, device="cuda").index_add_(0, inv, A.val.double())
        return _out(_from_keys(m, m, key, val))
    if kind == "mcl_step":
        E = ops[0]
        row, v = _rows_of(E), E.val
        weight = v.double() * v.double()
        decide = v if case["order"] == 0 else weight.float()
        order = torch.sort(decide, descending=True, stable=True).indices
        order = order[torch.sort(row[order], stable=True).indices]
        rank = torch.empty_like(order)
        rank[order] = torch.arange(E.nnz, device="cuda") - E.row_ptr.long()[row]
        keep = (decide >= 1e-4) & (rank < case["k"])
        w = weight * keep
        w = w / torch.zeros(E.rows, dtype=torch.float64, device="cuda").index_add_(0, row, w)[row]
        return _out(_from_keys(E.rows, E.cols, (row * E.cols + E.col)[keep], w[keep]))
    if kind in ("batch", "batch_grad"):
        A, X = ops[:2]
        D = _dense64(X)
        there = _csr64(A, torch.ones_like(A.val)) @ _dense64(X, torch.ones((), dtype=torch.float64, device="cuda")) > 0
        C = _csr64(A) @ D
        rows, cols = torch.nonzero(there, as_tuple=True)
        res = _out(_from_keys(A.rows, X.cols, rows * X.cols + cols, C[rows, cols]))
        if kind == "batch":
            return res
        G = torch.zeros_like(C)
        G[rows, cols] = ops[2][: rows.numel()].double()
        dX = (_csr64(_transposed(A)) @ G)[_rows_of(X), X.col.long()]
        return dict(res, dA=_row_dots(A, G, D), dX=dX)
    if kind == "layer":
        A, X, W, dY = ops
        best = torch.sort(X, dim=1, descending=True, stable=True).indices[:, : case["k"]]
        mask = torch.zeros_like(X, dtype=torch.bool).scatter_(1, best, True)
        C = _csr64(A) @ (X.double() * mask)
        dX = (_csr64(_transposed(A)) @ (dY.double() @ W.double().T)) * mask
        return {"Y": C @ W.double(), "dX": dX, "dW": C.T @ dY.double()}
    return None                     # sampling copies values: there is nothing to round
