"""Rows of very uneven length: where even the coarse list of row pieces cuts a row,
a launch below four waves takes the fine list (pieces of 64 records), whose
longest piece does not set the time.  A dequantised INT8 row shows its pieces:
one piece is rounded once, several are rounded and added.  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built

pytestmark = pytest.mark.gpu


def _row(long_row):
    """Row 7 (150 records) of 400 rows of 70, one of them `long_row` long, and
    what one rounding of its integer sums gives."""
    rosko = built()
    rng = np.random.default_rng(9)
    K, N = 4096, 256
    q = np.zeros((400, K), np.int8)
    for i in range(400):
        n = {7: 150, 11: long_row}.get(i, 70)
        q[i, rng.choice(K, n, replace=False)] = rng.integers(1, 127, n)
    b = rng.integers(-127, 128, (K, N)).astype(np.int8)
    rs = torch.from_numpy(rng.uniform(0.01, 0.03, 400).astype(np.float32)).cuda()
    cs = torch.from_numpy(rng.uniform(0.01, 0.03, N).astype(np.float32)).cuda()
    h = rosko.rosko_pack(torch.from_numpy(q).cuda(), rosko.I8, row_scale=rs)
    C = torch.empty((400, N), device="cuda")
    rosko.rosko_spmm(h, torch.from_numpy(b).cuda(), C, col_scale=cs,
                     tile=rosko.make_tile(dense_split_pm=1001))
    sums = torch.from_numpy(q[7].astype(np.int64) @ b.astype(np.int64)).cuda()
    once = (sums.float() * rs[7]) * cs
    exact = sums.double() * rs[7].double() * cs.double()
    err = (C[7].double() - exact).abs() / (exact.abs() + 1.0)
    assert float(err.max()) < 1e-5
    return C[7], once


def test_fine_pieces_where_a_row_is_cut_anyway():
    got, once = _row(3000)
    assert not torch.equal(got, once)


def test_whole_rows_where_none_is_cut():
    got, once = _row(140)
    assert torch.equal(got, once)
