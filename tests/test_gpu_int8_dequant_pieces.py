"""Dequantised INT8 products: every piece of a cut tile or row is rounded when it
is added to C, so the default schedule does not cut tiles into so many pieces
that the result is further from 64 bits than the CUDA cores' is.  GPU only."""
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,d", [(881, 8331, 58, 0.0283), (2543, 5414, 14, 0.0395)])
def test_default_is_as_exact_as_the_cuda_cores(M, K, N, d):
    rosko = built()
    g = torch.Generator(device="cuda").manual_seed(6)
    A = torch.randn((M, K), device="cuda", generator=g)
    A *= torch.rand((M, K), device="cuda", generator=g) < d
    B = torch.randn((K, N), device="cuda", generator=g)
    t = B.abs().amax(0) / 127.0
    q = (B / t).round()
    h = rosko.rosko_pack(A, rosko.I8)
    scale = A.abs().amax(1, keepdim=True) / torch.tensor(127.0, device="cuda")
    codes = (A / scale).round().clamp(-127, 127)
    exact = (codes.double() * scale.double()) @ (q.double() * t.double())
    Bd = _ldpad(q.to(torch.int8).cpu(), 1)
    C = torch.empty((M, N), device="cuda")

    def error(tile):
        rosko.rosko_spmm(h, Bd, C, col_scale=t, tile=tile)
        return float((C.double() - exact).norm() / exact.norm())

    assert error(None) <= 1.1 * error(rosko.make_tile(dense_split_pm=1001, n_r=256))
