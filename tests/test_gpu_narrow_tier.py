"""Narrow tiers (B of at most 1,024 columns): bitmap words and lane groups at
their edges, B rows shorter and longer than a warp, repeated and unsorted
columns, B's bitmaps built or not (A of many or few entries), fp32 and fp64
rows, row blocks, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_12036_gb300 import DeviceCSR, Plan, gen
from paper_2512_12036_gb300.batched import BatchedSpGEMM
from parity import compare

pytestmark = pytest.mark.gpu


def narrow_b(rows, cols, repeats, rng):
    lens = rng.choice([0, 1, 2, 7, 31, 32, 33, 64, 65, 200], size=rows)
    lens = np.minimum(lens, cols)
    r = np.repeat(np.arange(rows), lens)
    c = np.concatenate([rng.choice(cols, size=n, replace=False) for n in lens])
    if repeats:
        r, c = np.concatenate([r, r[::5]]), np.concatenate([c, c[::5]])
        p = np.lexsort((rng.random(r.size), r))
        r, c = r[p], c[p]
    return gen.csr_from_coo(rows, cols, r, c, gen.uniform_open_closed(rng, r.size), sort=not repeats)


@pytest.mark.parametrize("cols", [1, 31, 32, 33, 64, 100, 256, 257, 513, 1000, 1024])
@pytest.mark.parametrize("repeats", [False, True])
@pytest.mark.parametrize("few", [False, True])
def test_narrow_rows(cols, repeats, few):
    rng = np.random.default_rng(cols * 4 + 2 * repeats + few)
    B = narrow_b(4000 if few else 700, cols, repeats, rng)
    lens = rng.choice([0, 1, 3, 31, 32, 33, 40], size=40 if few else 300)
    lens[:4] = 166, 168, 200, 300
    r = np.repeat(np.arange(lens.size), lens)
    c = rng.integers(0, B.rows, size=r.size)
    A = gen.csr_from_coo(lens.size, B.rows, r, c, gen.uniform_open_closed(rng, r.size), sort=False)
    assert (A.nnz >= B.rows // 2) == (not few)
    ref = oracle.spgemm(A, B)
    dA, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    for opts in ({}, {"narrow_warps": 16, "narrow_max_ip": 600}):
        plan = Plan(**opts)
        compare(plan.spgemm(dA, dB).to_host(), ref)
        blocks, ip, nnz = plan.spgemm_blocks(dA, dB, max_block_nnz=max(1, int(ref.row_ptr[-1]) // 3 + 1024))
        torch.cuda.synchronize()
        assert nnz == int(ref.row_ptr[-1])
        cols_out = np.concatenate([C.to_host().col for _, _, C in blocks])
        assert np.array_equal(cols_out, ref.col)


@pytest.mark.parametrize("cols", [33, 256, 1024])
@pytest.mark.parametrize("repeats", [False, True])
def test_narrow_rows_without_room_for_bitmaps(cols, repeats):
    # more rows of C than the tables of a small B leave room for: both phases
    # mark the products
    rng = np.random.default_rng(7 * cols + repeats)
    B = narrow_b(40, cols, repeats, rng)
    lens = rng.choice([1, 8, 20, 33, 40, 170], size=60_000, p=[.2, .2, .2, .2, .19, .01])
    r = np.repeat(np.arange(lens.size), lens)
    A = gen.csr_from_coo(lens.size, B.rows, r, rng.integers(0, B.rows, size=r.size),
                         gen.uniform_open_closed(rng, r.size), sort=False)
    words = (cols + 31) // 32
    assert 4 * words * lens.size > 20 * B.nnz + 8 * B.rows + 12 * (cols + 1) + 8 * 256
    C = Plan().spgemm(DeviceCSR.from_host(A), DeviceCSR.from_host(B))
    torch.cuda.synchronize()
    compare(C.to_host(), oracle.spgemm(A, B))


@pytest.mark.parametrize("cols", [1, 10, 32, 33, 1024])
@pytest.mark.parametrize("esc_max", [1, 32])
def test_long_rows_of_no_or_one_product(cols, esc_max):
    # rows of A beyond esc_max entries whose rows of B are all empty, or all but
    # one with one entry (sparse labels), between ordinary fp32 and fp64 rows; in
    # one call, in row blocks and in a replayed batch, each with a workspace that
    # holds another structure's bitmaps
    rng = np.random.default_rng(cols + esc_max)
    empty, single, rows = 1000, 400, 2400
    lens = np.concatenate([np.zeros(empty, int), np.ones(single, int),
                           np.minimum(rng.integers(30, 60, size=rows - empty - single), cols)])
    rb = np.repeat(np.arange(rows), lens)
    cb = np.concatenate([rng.choice(cols, size=n, replace=False) for n in lens])
    B = gen.csr_from_coo(rows, cols, rb, cb, gen.uniform_open_closed(rng, rb.size))
    na = np.array([2, 3, 33, 40, 64, 166, 168, 200] * 20)
    rng.shuffle(na)
    ra = np.repeat(np.arange(na.size), na)
    kind = rng.integers(0, 3, size=na.size)                  # no product, one product, an ordinary row
    old, new = [], []
    for n, q in zip(na, kind):
        old.append(empty + single + rng.choice(rows - empty - single, size=n, replace=False))
        k = old[-1] if q == 2 else rng.choice(empty, size=n, replace=False)
        if q == 1:
            k[rng.integers(n)] = empty + rng.integers(single)
        new.append(k)
    val = gen.uniform_open_closed(rng, ra.size)
    first, A = (gen.csr_from_coo(na.size, rows, ra, np.concatenate(c), val, sort=False) for c in (old, new))
    assert np.array_equal(first.row_ptr, A.row_ptr)
    words = (cols + 31) // 32                                # (C's bitmaps are kept)
    assert 4 * words * (na.size + rows) + 256 < 20 * B.nnz + 8 * rows + 12 * cols
    ip, _ = oracle.ip_count(A, B)
    assert ((ip == 1) & (na > 32)).any() and (ip[kind == 0] == 0).all()
    ref, ref_first = oracle.spgemm(A, B), oracle.spgemm(first, B)
    plan = Plan(esc_max=esc_max)
    dA, d1, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(first), DeviceCSR.from_host(B)
    compare(plan.spgemm(dA, dB).to_host(), ref)
    ws = plan.workspace(dA, dB)
    compare(plan.spgemm(d1, dB, ws=ws).to_host(), ref_first)
    compare(plan.spgemm(dA, dB, ws=ws).to_host(), ref)
    compare(plan.spgemm(d1, dB, ws=ws).to_host(), ref_first)
    blocks, _, _ = plan.spgemm_blocks(dA, dB, max_block_nnz=int(ref.row_ptr[-1]) // 3 + 1024, ws=ws)
    torch.cuda.synchronize()
    plan.check_status(ws, "row blocks")
    for r0, r1, C in blocks:
        compare(C.to_host(), oracle.spgemm(A, B, rows=np.arange(r0, r1)))
    batch = BatchedSpGEMM(d1, dB, plan, capacity=int(ref_first.row_ptr[-1]))
    batch.capture()
    batch.run()
    compare(batch.result().to_host(), ref_first)
    d1.col.copy_(dA.col)
    batch.run()
    compare(batch.result().to_host(), ref)
