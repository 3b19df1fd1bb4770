"""512-column strips have no second set of sums: rows that would be one long
chain there are cut (a given width) or run in 256-column strips (the rule), so
that the error against 64 bits is that of the narrower strips, whose sums close
every 64 records.  GPU only."""
import pytest
import torch

from tests._lib import built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,d", [(2048, 32768, 1024, 0.012), (600, 11008, 2048, 0.012),
                                     (800, 8000, 1504, 0.014)])
def test_long_rows_in_wide_strips(M, K, N, d):
    rosko = built()
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn((M, K), device="cuda", generator=g)
    A *= torch.rand((M, K), device="cuda", generator=g) < d
    B = torch.randn((K, N), device="cuda", generator=g).to(torch.bfloat16)
    h = rosko.rosko_pack(A, rosko.BF16)
    exact = A.to(torch.bfloat16).double() @ B.double()
    C = torch.empty((M, N), device="cuda")

    def error(**kw):
        rosko.rosko_spmm(h, B, C, tile=rosko.make_tile(dense_split_pm=1001, **kw))
        return float((C.double() - exact).norm() / exact.norm())

    narrower = error(n_r=256)
    assert error(n_r=512) <= 1.1 * narrower
    assert error() <= 1.1 * narrower
