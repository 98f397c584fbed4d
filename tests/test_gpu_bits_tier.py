"""Bitmap tiers at the edges of their tiles, row classes and column limits,
against the oracle: A rows around the tile sizes, few and many products an
entry, rows of a handful to nearly all columns, fp32 and fp64 rows, repeated
and unsorted columns in B."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_12036_gb300 import DeviceCSR, Plan, gen
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [1025, 4097, 40_000, 131_071, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("messy", [False, True])
def test_rows_at_tile_and_class_edges(cols, messy):
    rng = np.random.default_rng(cols + messy)
    lens = np.concatenate([np.full(1500, 24), np.full(300, 0), np.full(40, min(cols, 900))])
    r = np.repeat(np.arange(lens.size), lens)
    c = np.concatenate([rng.choice(cols, size=n, replace=False) for n in lens])
    c[0], c[-1] = cols - 1, 0
    if messy:                                     # repeated columns, rows out of order
        r, c = np.concatenate([r, r[::7]]), np.concatenate([c, c[::7]])
        p = np.lexsort((rng.random(r.size), r))
        r, c = r[p], c[p]
    B = gen.csr_from_coo(lens.size, cols, r, c, gen.uniform_open_closed(rng, r.size), sort=not messy)
    ra, ca = [], []
    for na in [30, 60, 127, 128, 129, 167, 168, 255, 256, 257, 511, 512, 513, 1100]:
        for long_rows in (0, 1, 12, 40):          # 24 to 60,000 products a row
            k = rng.choice(1800, size=na, replace=False)
            k[:min(long_rows, na)] = 1800 + rng.choice(40, size=min(long_rows, na), replace=False)
            ra.append(np.full(na, len(ra)))
            ca.append(rng.permutation(k))
    A = gen.csr_from_coo(len(ra), lens.size, np.concatenate(ra), np.concatenate(ca),
                         gen.uniform_open_closed(rng, sum(x.size for x in ra)), sort=False)
    ref = oracle.spgemm(A, B)
    dA, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    for opts in ({}, {"warp_max_nnz": 100, "block_max_nnz": 2000}):
        C = Plan(**opts).spgemm(dA, dB)
        torch.cuda.synchronize()
        compare(C.to_host(), ref)


@pytest.mark.parametrize("cols,panel", [(300_000, 16384), (300_000, 4096), (40_000, 1024), (1_200_000, 16384)])
@pytest.mark.parametrize("repeats", [False, True])
def test_few_heavy_rows_cut_into_column_ranges(cols, panel, repeats):
    # a handful of fp64-bound rows of 2^15 to 2^20 products: the lightest in
    # one range, the heaviest in as many as the columns allow
    rng = np.random.default_rng(cols + panel + repeats)
    lens = rng.integers(100, 500, size=3000)
    r = np.repeat(np.arange(lens.size), lens)
    c = np.concatenate([np.sort(rng.choice(cols, size=n, replace=False)) for n in lens])
    c[::97] = rng.integers(0, 50, size=c[::97].size)                # hot columns
    key = np.unique(r * np.int64(cols) + c)
    r, c = key // cols, key % cols
    if repeats:
        r, c = np.concatenate([r, r[::50]]), np.concatenate([c, c[::50]])
    B = gen.csr_from_coo(lens.size, cols, r, c, gen.uniform_open_closed(rng, r.size))
    na = [170, 400, 900, 1100, 2000, 3000]
    ra = np.repeat(np.arange(len(na)), na)
    ca = np.concatenate([rng.choice(lens.size, size=n, replace=False) for n in na])
    A = gen.csr_from_coo(len(na), lens.size, ra, ca, gen.uniform_open_closed(rng, ra.size))
    ip, _ = oracle.ip_count(A, B)
    assert ip.min() < 1 << 17 and ip.max() > 1 << 19
    C = Plan(panel_cols=panel).spgemm(DeviceCSR.from_host(A), DeviceCSR.from_host(B))
    torch.cuda.synchronize()
    compare(C.to_host(), oracle.spgemm(A, B))


def test_part_counts_of_another_call_are_reported():
    # rows cut into column ranges read their parts' counts from the workspace
    # (its last array): counts that cannot be theirs set the status word, and
    # nothing is written outside the rows
    from paper_2512_12036_gb300 import SpgemmError
    rng = np.random.default_rng(3)
    cols, k = 300_000, 3000
    rb = np.repeat(np.arange(k), 300)
    B = gen.csr_from_coo(k, cols, rb, rng.integers(0, cols, size=rb.size), gen.uniform_open_closed(rng, rb.size))
    na = [1100, 2000, 2900]
    ra = np.repeat(np.arange(len(na)), na)
    ca = np.concatenate([rng.choice(k, size=n, replace=False) for n in na])
    A = gen.csr_from_coo(len(na), k, ra, ca, gen.uniform_open_closed(rng, ra.size))
    plan, dA, dB = Plan(), DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    for fill in (-5, 0x7fffffff):
        ws = plan.workspace(dA, dB)
        ip_row, _ = plan.count(dA, dB, ws)
        row_nnz, nnz = plan.symbolic(dA, dB, ip_row, ws)
        rp, _ = plan.row_ptr(row_nnz, ws)
        ws[-256:].view(torch.int32).fill_(fill)
        buf = torch.full((2, nnz + 2048), -7, dtype=torch.int32, device="cuda")
        col, val = buf[0, 1024:1024 + nnz], buf[1, 1024:1024 + nnz].view(torch.float32)
        plan.numeric(dA, dB, ip_row, rp, ws, col, val)
        torch.cuda.synchronize()
        assert (buf[:, :1024] == -7).all() and (buf[:, 1024 + nnz:] == -7).all()
        with pytest.raises(SpgemmError):
            plan.check_status(ws, "stale part counts")


def test_part_counts_of_the_wrong_ranges_stay_in_their_slices():
    # counts that could be the row's but are not: a sum that is not the row's
    # writes none of it, and a shift between two ranges leaves every entry in
    # the slice of its own range (the blocks of a row write side by side)
    from paper_2512_12036_gb300 import SpgemmError
    rng = np.random.default_rng(4)
    cols, k, parts = 300_000, 3000, 8
    rb = np.repeat(np.arange(k), 300)
    B = gen.csr_from_coo(k, cols, rb, rng.integers(0, cols, size=rb.size), gen.uniform_open_closed(rng, rb.size))
    na = [1100, 2000, 2900]
    ra = np.repeat(np.arange(len(na)), na)
    ca = np.concatenate([rng.choice(k, size=n, replace=False) for n in na])
    A = gen.csr_from_coo(len(na), k, ra, ca, gen.uniform_open_closed(rng, ra.size))
    plan, dA, dB = Plan(), DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    panels = -(-cols // plan.opts["panel_cols"])
    edge = [panels * q // parts * plan.opts["panel_cols"] for q in range(parts)] + [cols]
    for change in ("less", "more", "down", "up"):
        ws = plan.workspace(dA, dB)
        ip_row, _ = plan.count(dA, dB, ws)
        row_nnz, nnz = plan.symbolic(dA, dB, ip_row, ws)
        rp, _ = plan.row_ptr(row_nnz, ws)
        counts = ws[-256:].view(torch.int32)[:parts * len(na)].view(len(na), parts)
        assert torch.equal(counts.sum(1, dtype=torch.int32), row_nnz)
        delta = torch.zeros(parts, dtype=torch.int32, device="cuda")
        delta[3] = -40 if change in ("less", "down") else 40
        if change in ("down", "up"):
            delta[4] = -delta[3]
        counts += delta
        buf = torch.full((2, nnz + 2048), -7, dtype=torch.int32, device="cuda")
        col, val = buf[0, 1024:1024 + nnz], buf[1, 1024:1024 + nnz].view(torch.float32)
        plan.numeric(dA, dB, ip_row, rp, ws, col, val)
        torch.cuda.synchronize()
        assert (buf[:, :1024] == -7).all() and (buf[:, 1024 + nnz:] == -7).all()
        got, slices = col.cpu().numpy(), np.cumsum(counts.cpu().numpy(), axis=1)
        for r, s in enumerate(rp.cpu().numpy()[:-1]):
            if change in ("less", "more"):
                assert (got[s:s + int(row_nnz[r])] == -7).all()
                continue
            for q in range(parts):
                here = got[s + (slices[r, q - 1] if q else 0):s + slices[r, q]]
                here = here[here != -7]
                assert ((here >= edge[q]) & (here < edge[q + 1])).all() and here.size
        with pytest.raises(SpgemmError):
            plan.check_status(ws, "wrong part counts")


@pytest.mark.parametrize("cols,panel", [(300_000, 16384), (40_000, 1024)])
@pytest.mark.parametrize("kind", ["one_row", "every_row", "repeats"])
def test_column_ranges_with_unsorted_b(cols, panel, kind):
    # B rows out of order have no usable panel table: every range of a row then
    # walks all its products and keeps those of its columns
    rng = np.random.default_rng(cols + len(kind))
    lens = rng.integers(100, 500, size=3000)
    r = np.repeat(np.arange(lens.size), lens)
    c = np.concatenate([np.sort(rng.choice(cols, size=n, replace=False)) for n in lens])
    c[::97] = rng.integers(0, 50, size=c[::97].size)                # hot columns
    key = np.unique(r * np.int64(cols) + c)
    r, c = key // cols, key % cols
    if kind == "repeats":
        r, c = np.concatenate([r, r[::50]]), np.concatenate([c, c[::50]])
    if kind == "one_row":
        at = np.nonzero(r == 1700)[0]
        c[at] = rng.permutation(c[at])
    else:
        p = np.lexsort((rng.random(r.size), r))
        r, c = r[p], c[p]
    B = gen.csr_from_coo(lens.size, cols, r, c, gen.uniform_open_closed(rng, r.size), sort=False)
    na = [170, 900, 1100, 3000]
    ra = np.repeat(np.arange(len(na)), na)
    ca = np.concatenate([rng.choice(lens.size, size=n, replace=False) for n in na])
    A = gen.csr_from_coo(len(na), lens.size, ra, ca, gen.uniform_open_closed(rng, ra.size))
    ip, _ = oracle.ip_count(A, B)
    assert ip.min() < 1 << 17 and ip.max() > 1 << 19
    C = Plan(panel_cols=panel).spgemm(DeviceCSR.from_host(A), DeviceCSR.from_host(B))
    torch.cuda.synchronize()
    compare(C.to_host(), oracle.spgemm(A, B))
