"""Sort tier (rows of up to 512 products) and accumulation warp tier at the
edges of their row classes and sort sizes, fp32 and fp64, with columns that
share a 32-bit word with a position or table slot and with columns too wide
for that, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_12036_gb300 import DeviceCSR, Plan, gen
from parity import compare

pytestmark = pytest.mark.gpu

EDGES = [33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025]


@pytest.mark.parametrize("cols", [100_000, 1 << 21, (1 << 21) + 1, (1 << 23) - 1, 1 << 23])
@pytest.mark.parametrize("load", [0, 25, 90])
def test_rows_at_class_edges(cols, load):
    rng = np.random.default_rng(cols % 1000 + load)
    # B: 128 rows of 16 columns, 1,100 rows of 1 column, every column once;
    # then 50 empty rows
    picked = rng.choice(cols, size=128 * 16 + 1100, replace=False)
    picked[:2] = 0, cols - 1
    picked = np.unique(picked)
    picked = rng.permutation(picked)
    rows_b = np.concatenate([np.repeat(np.arange(128), 16), 128 + np.arange(picked.size - 128 * 16)])
    B = gen.csr_from_coo(128 + 1100 + 50, cols, rows_b, picked,
                         gen.uniform_open_closed(rng, picked.size))
    ones = picked.size - 128 * 16
    r, c = [], []
    for i, n in enumerate(EDGES * 4):
        if i < len(EDGES):                       # few long B rows: fp32
            full, single = n // 16, n % 16
        elif i < 2 * len(EDGES):                 # many one-entry B rows: fp64 from 168 up
            full, single = max(0, (n - 700) // 16), n - 16 * max(0, (n - 700) // 16)
        else:                                    # as the first, with products that meet (below)
            full, single = n // 16, n % 16
        k = np.concatenate([rng.choice(128, size=full, replace=False),
                            128 + rng.choice(ones, size=single, replace=False)])
        if i >= 3 * len(EDGES):
            k = np.tile(k, 3)
        elif i >= 2 * len(EDGES):
            k = np.concatenate([k, k[: k.size // 2]])
        empty = 1228 + rng.integers(0, 50, size=5)
        k = rng.permutation(np.concatenate([k, empty]))
        r.append(np.full(k.size, i))
        c.append(k)
    r, c = np.concatenate(r), np.concatenate(c)
    A = gen.csr_from_coo(4 * len(EDGES), B.rows, r, c, gen.uniform_open_closed(rng, r.size), sort=False)
    nnz = np.diff(oracle.spgemm(A, B).row_ptr)
    assert set(EDGES) <= set(nnz.tolist())
    plan = Plan(hash_load_pct=load)
    C = plan.spgemm(DeviceCSR.from_host(A), DeviceCSR.from_host(B))
    torch.cuda.synchronize()
    compare(C.to_host(), oracle.spgemm(A, B))
