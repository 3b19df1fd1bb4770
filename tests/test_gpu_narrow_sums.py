"""Rounding error of the few-column kernel on long rows: a lane closes its sums
every 32 records, so that the result is no further from the 64-bit one than the
general row-direct kernel's (which closes its sums every 64).  GPU only."""
import pytest
import torch

from tests._lib import built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,d", [(2048, 1600, 32, 0.5), (4096, 4096, 8, 0.5),
                                     (11008, 1500, 64, 0.3)])
def test_long_rows_are_as_exact_as_in_the_general_kernel(M, K, N, d):
    rosko = built()
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn((M, K), device="cuda", generator=g)
    A *= torch.rand((M, K), device="cuda", generator=g) < d
    B = torch.randn((K, N), device="cuda", generator=g)
    h = rosko.rosko_pack(A, rosko.F32)
    exact = A.double() @ B.double()
    C = torch.empty((M, N), device="cuda")

    def error(tile):
        rosko.rosko_spmm(h, B, C, tile=tile)
        return float((C.double() - exact).norm() / exact.norm())

    # (a width of 128 columns is the general kernel's)
    assert error(None) <= 1.1 * error(rosko.make_tile(n_r=128))
