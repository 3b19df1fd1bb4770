"""The few-column kernel behind a tile: a plan passed back runs what the call ran,
and a call that cannot run the kernel (a width of its own, another traversal,
FORCED) is not kept off the tensor cores for its sake.  GPU only."""
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def _problem(rosko, M, K, N, s, code, seed=71):
    A = torch.from_numpy(gen.sparse_weight(M, K, s, gen.rng_for(seed), "uniform")).cuda()
    dt, size = (torch.bfloat16, 2) if code == rosko.BF16 else (torch.float32, 4)
    B = _ldpad(torch.from_numpy(gen.normal((K, N), gen.rng_for(seed, 1))).to(dt), size)
    return rosko.rosko_pack(A, code), B, torch.empty((M, N), device="cuda")


@pytest.mark.parametrize("M,K,N,s,bf16", [(11008, 4096, 16, 0.9, True), (4096, 4096, 8, 0.7, True),
                                          (4096, 1500, 32, 0.9, False)])
def test_a_plan_passed_back_runs_the_same(M, K, N, s, bf16):
    rosko = built()
    h, B, C = _problem(rosko, M, K, N, s, rosko.BF16 if bf16 else rosko.F32)
    plan = rosko.rosko_spmm_plan(h, B, C)
    assert plan["few_n_r"] > 0 and plan["dense_tiles"] == 0
    tile = rosko.make_tile(**plan["tile"])
    again = rosko.rosko_spmm_plan(h, B, C, tile=tile)
    assert again == plan
    first = rosko.rosko_spmm(h, B, C).clone()
    assert torch.equal(rosko.rosko_spmm(h, B, C, tile=tile), first)


@pytest.mark.parametrize("kw", [dict(n_r=128), dict(order=2), dict(order=1),
                                dict(mode=3, order=4, n_r=256, k_c=8, m_c=16, split_k=1)])
def test_other_kernels_are_weighed_against_the_tensor_cores(kw):
    rosko = built()
    h, B, C = _problem(rosko, 11008, 4096, 16, 0.9, rosko.BF16)
    plan = rosko.rosko_spmm_plan(h, B, C, tile=rosko.make_tile(**kw))
    assert plan["dense_tiles"] == 86 and plan["few_n_r"] == 0
    assert rosko.rosko_spmm_plan(h, B, C)["few_n_r"] > 0
