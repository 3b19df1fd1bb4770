"""Dense copies written eight columns at a time: K that is no multiple of 8,
rows of A that are and are not 16-byte aligned (an odd leading dimension, a
view that starts off the boundary), every source type, against the unpacked
matrix through the tensor cores (identity B: C is the dense copy itself).
Exact: BF16 and INT8 values times one.  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from oracle.quant import bf16_round, quantize_rows_int8
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("src", ["f32", "bf16", "f32->i8"])
@pytest.mark.parametrize("M,K,pad,off", [(130, 61, 0, 0), (260, 64, 8, 0), (128, 72, 5, 0),
                                         (200, 129, 7, 3), (129, 8, 8, 4), (300, 130, 6, 0)])
def test_dense_copy_is_the_matrix(src, M, K, pad, off):
    rosko = built()
    A = gen.sparse_weight(M, K, 0.6, gen.rng_for(95, M, K), "uniform")
    dt = torch.bfloat16 if src == "bf16" else torch.float32
    buf = torch.zeros((M, K + pad + off), dtype=dt, device="cuda")
    view = buf[:, off:off + K]
    view.copy_(torch.from_numpy(A).to(dt))
    i8 = src.endswith("i8")
    h = rosko.rosko_pack(view, rosko.I8 if i8 else rosko.BF16)
    n = -(-K // 16) * 16
    B = torch.eye(K, n, device="cuda").to(torch.int8 if i8 else torch.bfloat16)[:, :K]
    C = torch.empty((M, K), dtype=torch.int32 if i8 else torch.float32, device="cuda")
    t = rosko.make_tile(dense_split_pm=1)
    assert rosko.rosko_spmm_plan(h, B, C, tile=t)["dense_tiles"] == -(-M // 128)
    rosko.rosko_spmm(h, B, C, tile=t)
    want = quantize_rows_int8(A)[0] if i8 else bf16_round(A)
    assert np.array_equal(C.cpu().numpy().astype(np.float64), want.astype(np.float64))


@pytest.mark.parametrize("src", ["f32", "bf16", "f32->i8"])
@pytest.mark.parametrize("M,K", [(3, 256), (3, 257), (40, 2047), (20, 2049), (17, 4500),
                                 (2432, 300), (2433, 300)])
def test_row_stream_is_the_matrix(src, M, K):
    """Rows written by one warp or by a whole block in turns of 2048 columns,
    long rows in several pieces, through both traversals that read the row
    stream (identity B, exact)."""
    rosko = built()
    A = gen.sparse_weight(M, K, 0.7, gen.rng_for(96, M, K), "uniform")
    A[M // 2] = 0.0
    A[M - 1] = np.arange(1, K + 1) % 7 + 1.0
    dt = torch.bfloat16 if src == "bf16" else torch.float32
    i8 = src.endswith("i8")
    h = rosko.rosko_pack(torch.from_numpy(A).to("cuda", dt), rosko.I8 if i8 else rosko.BF16)
    n = -(-K // 16) * 16
    B = torch.eye(K, n, device="cuda").to(torch.int8 if i8 else torch.bfloat16)[:, :K]
    want = (quantize_rows_int8(A)[0] if i8 else bf16_round(A)).astype(np.float64)
    for order in (3, 4):
        C = torch.empty((M, K), dtype=torch.int32 if i8 else torch.float32, device="cuda")
        rosko.rosko_spmm(h, B, C, tile=rosko.make_tile(order=order, dense_split_pm=1001))
        assert np.array_equal(C.cpu().numpy().astype(np.float64), want), order
