"""Every variant of the few-column kernel (1, 2, 4 and 8 16-byte chunks per strip,
FP32 and BF16, short and long pieces), checked to be what runs: one row that is
cut and added, one empty row, a ragged last strip, several strips, accumulation,
and the panels that the tensor cores leave.  Within 1e-5 of the normalised error
(the parity bar).  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad
from oracle.quant import bf16_round
from oracle.spmm import normalized_error, spmm
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu

# columns per strip, M, K, N, density
BF16 = [(8, 1500, 12800, 5, 0.05), (8, 1200, 12800, 3, 0.1), (8, 2000, 2000, 1, 0.1),
        (16, 2000, 3000, 13, 0.1), (16, 1000, 6400, 16, 0.1), (32, 2500, 3200, 30, 0.05),
        (32, 2500, 3000, 20, 0.1), (64, 3000, 1600, 33, 0.1), (64, 2600, 1000, 100, 0.3)]
F32 = [(4, 1500, 12800, 5, 0.05), (4, 1200, 12800, 3, 0.1), (8, 2000, 6000, 7, 0.05),
       (8, 1000, 6400, 16, 0.1), (16, 2500, 3200, 30, 0.05), (16, 2500, 3000, 20, 0.1),
       (32, 3000, 1600, 33, 0.05), (32, 2600, 1000, 100, 0.3)]


def _check(rosko, A, B, bf16, strip, accumulate, tile, dense_tiles):
    M, N = A.shape[0], B.shape[1]
    dt, size = (torch.bfloat16, 2) if bf16 else (torch.float32, 4)
    h = rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.BF16 if bf16 else rosko.F32)
    Bd = _ldpad(torch.from_numpy(B).to(dt), size)
    C0 = np.random.default_rng(3).standard_normal((M, N)).astype(np.float32) if accumulate else None
    C = torch.from_numpy(C0).cuda() if accumulate else torch.full((M, N), float("nan"), device="cuda")
    plan = rosko.rosko_spmm_plan(h, Bd, C, tile=tile, accumulate=accumulate)
    assert plan["few_n_r"] == strip and plan["dense_tiles"] == dense_tiles
    # the cut row is added into C
    assert plan["zero_fill"] == (0 if accumulate else 1)
    rosko.rosko_spmm(h, Bd, C, tile=tile, accumulate=accumulate)
    a, b = (bf16_round(A), bf16_round(B)) if bf16 else (A, B)
    ref, D = spmm(a, b, C0=C0)
    if accumulate:
        D = D + np.abs(C0)
    assert normalized_error(C.cpu().numpy(), ref, D) <= 1e-5


@pytest.mark.parametrize("bf16,case,accumulate",
                         [(True, c, i % 2 == 1) for i, c in enumerate(BF16)] +
                         [(False, c, i % 2 == 0) for i, c in enumerate(F32)])
def test_variant(bf16, case, accumulate):
    strip, M, K, N, d = case
    A = gen.sparse_weight(M, K, 1.0 - d, gen.rng_for(41, strip), "uniform")
    A[5] = gen.normal((1, K), gen.rng_for(42))
    A[M // 2] = 0
    B = gen.normal((K, N), gen.rng_for(43))
    rosko = built()
    _check(rosko, A, B, bf16, strip, accumulate, rosko.make_tile(dense_split_pm=1001), 0)


@pytest.mark.parametrize("case,accumulate", [((16, 2000, 3000, 13, 0.1), False),
                                             ((64, 2600, 1000, 100, 0.3), True)])
def test_beside_the_tensor_cores(case, accumulate):
    strip, M, K, N, d = case
    A = gen.sparse_weight(M, K, 1.0 - d, gen.rng_for(44, strip), "uniform")
    A[256:384] = gen.sparse_weight(128, K, 0.2, gen.rng_for(45, strip), "uniform")
    A[1500] = gen.normal((1, K), gen.rng_for(46))
    A[7] = 0
    B = gen.normal((K, N), gen.rng_for(47))
    rosko = built()
    _check(rosko, A, B, True, strip, accumulate, rosko.make_tile(dense_split_pm=600), 1)
