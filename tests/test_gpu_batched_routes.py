"""BF16 layers of little work are computed with FMAs (round to nearest), not on
the tensor cores (truncating sums), alone and in a batch whose other layers run
there.  In the batch their rows are not cut, so that the results equal those of
the single call bit for bit; alone, the error against 64 bits is that of the
FMAs.  GPU only."""
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def test_a_batch_keeps_layers_of_little_work():
    rosko = built()
    shapes = [(512, 4608, 3136, 0.9), (1385, 144, 254, 0.87), (80, 74, 6608, 0.87),
              (91, 171, 5489, 0.87), (2772, 1163, 804, 0.7)]
    hs, Bs, alone, routes = [], [], [], []
    for j, (M, K, N, s) in enumerate(shapes):
        h = rosko.rosko_pack(torch.from_numpy(gen.sparse_weight(M, K, s, gen.rng_for(61, j),
                                                                "uniform")).cuda(), rosko.BF16)
        B = _ldpad(torch.from_numpy(gen.relu_normal((K, N), gen.rng_for(62, j))).to(torch.bfloat16), 2)
        C = torch.empty((M, N), device="cuda")
        routes.append(rosko.rosko_spmm_plan(h, B, C)["dense_tiles"])
        hs.append(h)
        Bs.append(B)
        alone.append(rosko.rosko_spmm(h, B, C))
    # both routes are in the batch
    assert routes[0] > 0 and routes[4] > 0 and routes[1:4] == [0, 0, 0]
    Cs = [torch.empty_like(C) for C in alone]
    rosko.rosko_spmm_batched(hs, Bs, Cs)
    for j in (1, 2, 3):
        assert torch.equal(Cs[j], alone[j]), shapes[j]


@pytest.mark.parametrize("M,K,N,s", [(176, 1465, 29, 0.58), (406, 3101, 99, 0.836),
                                     (1929, 665, 6153, 0.9861)])
def test_single_layers_of_little_work(M, K, N, s):
    rosko = built()
    A = torch.from_numpy(gen.sparse_weight(M, K, s, gen.rng_for(63), "uniform")).cuda()
    B = _ldpad(torch.from_numpy(gen.normal((K, N), gen.rng_for(64))).to(torch.bfloat16), 2)
    h = rosko.rosko_pack(A, rosko.BF16)
    C = torch.empty((M, N), device="cuda")
    assert rosko.rosko_spmm_plan(h, B, C)["dense_tiles"] == 0
    exact = A.to(torch.bfloat16).double() @ B.double()

    def error(tile):
        rosko.rosko_spmm(h, B, C, tile=tile)
        return float((C.double() - exact).norm() / exact.norm())

    # the same sums, or (cut rows) the same pieces in another order
    assert error(None) <= 1.1 * error(rosko.make_tile(dense_split_pm=1001))
