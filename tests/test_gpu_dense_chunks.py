"""Tensor-core sums of short K ranges.  The tensor core truncates every addition
toward zero, so that a chain's relative error grows with its length (twice the
chain, about twice the error); the kernel closes the sums of a short range
every 8 slabs of 64 and adds them rounding to nearest, so that the error of a
tile of 16 or 24 slabs is that of one of 8, plus roundings far below it.
GPU only."""
import pytest
import torch

from tests._lib import built

pytestmark = pytest.mark.gpu


def _error(rosko, K, TN, batch=False):
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn((512, K), device="cuda", generator=g)
    B = torch.randn((K, 512), device="cuda", generator=g).to(torch.bfloat16)
    h = rosko.rosko_pack(A, rosko.BF16)
    C = torch.empty((512, 512), device="cuda")
    t = rosko.make_tile(dense_split_pm=1, dense_n_r=TN)
    plan = rosko.rosko_spmm_plan(h, B, C, tile=t)
    assert plan["dense_tiles"] == 4 and plan["zero_fill"] == 0   # whole tiles
    if batch:
        rosko.rosko_spmm_batched([h], [B], [C], tiles=[t])
    else:
        rosko.rosko_spmm(h, B, C, tile=t)
    exact = A.to(torch.bfloat16).double() @ B.double()
    return float((C.double() - exact).norm() / exact.norm())


@pytest.mark.parametrize("TN,K", [(256, 1024), (128, 1024), (128, 1344)])
def test_error_does_not_grow_with_a_short_range(TN, K):
    rosko = built()
    assert _error(rosko, K, TN) <= 1.3 * _error(rosko, 512, TN)


@pytest.mark.parametrize("TN,K", [(128, 832), (256, 896), (128, 960)])
def test_the_only_dense_problem_of_a_batch(TN, K):
    # fewer than 16 slabs: a batch, which shares its workers by (tile, slab),
    # used to cut such tiles
    rosko = built()
    assert _error(rosko, K, TN, batch=True) <= 1.3 * _error(rosko, 512, TN)
