"""INT8 x INT8 on the tensor cores with a dequantised FP32 result, and the
INT32 sums kept in registers across K chunks: chunk edges, cut and whole
tiles, ragged and unaligned C, accumulation, mixed dense and sparse tiles.
INT32 is bit-exact; FP32 is within 1e-5 of the normalised error (the parity
bar).  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_int8_tc import _case
from tests.test_gpu_spmm import _ldpad
from oracle.quant import quantize_cols_int8, quantize_rows_int8
from oracle.spmm import normalized_error, spmm_int
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,TN,ctas", [
    (300, 1023, 260, 256, 2),      # one chunk short of a slab, whole tiles
    (257, 2049, 131, 128, 2),      # a third chunk of one row of B, odd C rows
    (130, 3000, 96, 128, 0),       # K cut between pairs
    (100, 2100, 300, 256, 0),      # a single row tile (no pair), cut
    (384, 1088, 1100, 128, 4),     # several tiles per pair, whole and cut
])
@pytest.mark.parametrize("accumulate", [False, True])
def test_int8_results(M, K, N, TN, ctas, accumulate):
    rosko = built()
    A, qa, qb = _case(M, K, N, 0.5, 51)
    _, sa = quantize_rows_int8(A)
    sb = quantize_cols_int8(gen.normal((K, N), gen.rng_for(51, K, N)))[1]
    h = rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.I8)
    Bd = _ldpad(torch.from_numpy(qb), 1)
    t = rosko.make_tile(dense_split_pm=1, dense_n_r=TN, dense_split_k=ctas)
    rng = np.random.default_rng(8)
    Ci0 = rng.integers(-1000, 1000, (M, N)).astype(np.int32)
    Ci = torch.from_numpy(Ci0.copy()).cuda() if accumulate else \
        torch.full((M, N), -7, dtype=torch.int32, device="cuda")
    rosko.rosko_spmm(h, Bd, Ci, tile=t, accumulate=accumulate)
    Cf0 = rng.standard_normal((M, N)).astype(np.float32)
    Cf = torch.from_numpy(Cf0.copy()).cuda() if accumulate else \
        torch.full((M, N), float("nan"), device="cuda")
    cs = torch.from_numpy(sb).cuda()
    assert rosko.rosko_spmm_plan(h, Bd, Cf, col_scale=cs, tile=t)["dense_tiles"] == -(-M // 128)
    rosko.rosko_spmm(h, Bd, Cf, col_scale=cs, tile=t, accumulate=accumulate)
    torch.cuda.synchronize()
    assert rosko.rosko_device_status(clear=True) == 0
    want = spmm_int(qa, qb)
    assert np.array_equal(Ci.cpu().numpy().astype(np.int64),
                          want + (Ci0.astype(np.int64) if accumulate else 0))
    scale = sa[:, None].astype(np.float64) * sb[None, :].astype(np.float64)
    ref = want * scale
    D = (np.abs(qa).astype(np.float64) @ np.abs(qb).astype(np.float64)) * scale
    if accumulate:
        ref, D = ref + Cf0, D + np.abs(Cf0)
    assert normalized_error(Cf.cpu().numpy(), ref, D) <= 1e-5


def test_dequant_mixed_tiles():
    # some 128-row tiles on the tensor cores, the others row-direct
    rosko = built()
    A, qa, qb = _case(700, 1500, 300, 0.95, 52, "powerlaw")
    _, sa = quantize_rows_int8(A)
    sb = np.linspace(0.5, 2.0, 300, dtype=np.float32)
    h = rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.I8)
    Bd = _ldpad(torch.from_numpy(qb), 1)
    dens = sorted((qa[r:r + 128] != 0).mean() * 1000.0 for r in range(0, 700, 128))
    t = rosko.make_tile(dense_split_pm=int(dens[len(dens) // 2]) + 1)
    C = torch.full((700, 300), float("nan"), device="cuda")
    cs = torch.from_numpy(sb).cuda()
    pl = rosko.rosko_spmm_plan(h, Bd, C, col_scale=cs, tile=t)
    assert pl["dense_tiles"] > 0 and pl["sparse_panels"] > 0
    rosko.rosko_spmm(h, Bd, C, col_scale=cs, tile=t)
    scale = sa[:, None].astype(np.float64) * sb[None, :].astype(np.float64)
    D = (np.abs(qa).astype(np.float64) @ np.abs(qb).astype(np.float64)) * scale
    assert normalized_error(C.cpu().numpy(), spmm_int(qa, qb) * scale, D) <= 1e-5
