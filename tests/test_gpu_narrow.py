"""Row-direct with few columns of C: the kernel that keeps a strip of B in
shared memory.  Chunk counts (1, 2, 4, 8 per strip), several strips, a ragged
last chunk, K up to the largest strip, rows without and with many nonzeros,
cut rows, accumulation, and rows of B that no nonzero meets holding non-finite
values (never read into C).  FP32 and BF16 within 1e-5 of the normalised error
(the parity bar).  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad, _problem, check, run
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["f32", "bf16"])
@pytest.mark.parametrize("M,K,N,s", [
    (70, 300, 1, 0.9), (33, 17, 3, 0.5), (500, 1500, 8, 0.9), (200, 3200, 17, 0.95),
    (300, 6400, 40, 0.97), (100, 12800, 9, 0.99), (90, 12801, 9, 0.99), (96, 640, 200, 0.9),
    (1, 1, 1, 0.0), (1000, 100, 100, 0.8),
])
@pytest.mark.parametrize("accumulate", [False, True])
def test_few_columns(mode, M, K, N, s, accumulate):
    rosko = built()
    A, B = _problem(M, K, N, s, seed=81)
    A[M // 2] = 0
    C0 = np.random.default_rng(2).standard_normal((M, N)).astype(np.float32) if accumulate else None
    t = rosko.make_tile(dense_split_pm=1001)
    check(mode, *run(rosko, A, B, mode, m_r=16, tile=t, accumulate=accumulate, C0=C0))


@pytest.mark.parametrize("mode", ["f32", "bf16"])
def test_cut_rows_and_mixed_tiles(mode):
    rosko = built()
    A = gen.sparse_weight(400, 2000, 0.97, gen.rng_for(82), "powerlaw")
    A[5] = 1.0
    B = gen.normal((2000, 24), gen.rng_for(83))
    for pm in (1001, 40):
        check(mode, *run(rosko, A, B, mode, m_r=16, tile=rosko.make_tile(dense_split_pm=pm)))


@pytest.mark.parametrize("dtype,code", [(torch.float32, 0), (torch.bfloat16, 1)])
def test_untouched_rows_of_b_are_skipped(dtype, code):
    rosko = built()
    rng = np.random.default_rng(4)
    A = np.zeros((50, 400), np.float32)
    for i in range(50):
        A[i, 2 * rng.choice(200, 37, replace=False)] = 1.0   # even columns only
    B = rng.standard_normal((400, 12)).astype(np.float32)
    B[1::2] = np.inf
    h = rosko.rosko_pack(torch.from_numpy(A).cuda(), code)
    Bd = _ldpad(torch.from_numpy(B).to(dtype), torch.empty((), dtype=dtype).element_size())
    C = torch.full((50, 12), float("nan"), device="cuda")
    rosko.rosko_spmm(h, Bd, C, tile=rosko.make_tile(dense_split_pm=1001))
    assert torch.isfinite(C).all()
