"""Batches of layers with few columns of C (a decoding step): within 1e-5 of the
normalised error (the parity bar), and not slower than the same calls one after
another by more than half, by default and with the tiles that the single calls'
plans report (before: six times and ten times slower).  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad
from oracle.quant import bf16_round
from oracle.spmm import normalized_error, spmm
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def _layers(rosko, shapes, bf16):
    dt, size = (torch.bfloat16, 2) if bf16 else (torch.float32, 4)
    out = []
    for j, (M, K, N, s, pat) in enumerate(shapes):
        A = gen.sparse_weight(M, K, s, gen.rng_for(81, j), pat)
        B = gen.normal((K, N), gen.rng_for(82, j))
        h = rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.BF16 if bf16 else rosko.F32)
        out.append((A, B, h, _ldpad(torch.from_numpy(B).to(dt), size),
                    torch.full((M, N), float("nan"), device="cuda")))
    return out


def _us(fn):
    for _ in range(3):
        fn()
    torch.cuda.synchronize()
    best = float("inf")
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(10):
            fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 100.0)
    return best


@pytest.mark.parametrize("planned", [False, True])
def test_decode_batch_is_not_slower_than_its_calls(planned):
    rosko = built()
    ls = _layers(rosko, [(11008, 4096, 16, 0.9, "uniform"), (4096, 11008, 16, 0.9, "uniform")] * 2, True)
    hs, Bs, Cs = ([x[k] for x in ls] for k in (2, 3, 4))
    tiles = [rosko.make_tile(**rosko.rosko_spmm_plan(h, B, C)["tile"])
             for h, B, C in zip(hs, Bs, Cs)] if planned else None

    def alone():
        for h, B, C in zip(hs, Bs, Cs):
            rosko.rosko_spmm(h, B, C)

    # (the least of three: the host's own pauses)
    assert min(_us(lambda: rosko.rosko_spmm_batched(hs, Bs, Cs, tiles=tiles)) / _us(alone)
               for _ in range(3)) <= 1.5


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("accumulate", [False, True])
def test_few_column_problems_beside_others(bf16, accumulate):
    # few columns with cut rows and empty ones, a problem of the shared launch,
    # and (BF16) one whose densest tiles run on the tensor cores
    rosko = built()
    ls = _layers(rosko, [(4000, 2000, 24, 0.8, "powerlaw"), (300, 500, 257, 0.95, "uniform"),
                         (3000, 3000, 9, 0.7, "uniform"), (700, 1000, 130, 0.9, "powerlaw")], bf16)
    tiles = [rosko.make_tile(dense_split_pm=pm) for pm in (1001, 1001, 1001, 100)]
    C0 = [np.random.default_rng(j).standard_normal(x[4].shape).astype(np.float32)
          for j, x in enumerate(ls)]
    for x, c in zip(ls, C0):
        if accumulate:
            x[4].copy_(torch.from_numpy(c))
    hs, Bs, Cs = ([x[k] for x in ls] for k in (2, 3, 4))
    l0 = rosko.rosko_kernel_launches()
    rosko.rosko_spmm_batched(hs, Bs, Cs, accumulate=accumulate, tiles=tiles)
    # two of their own, one shared, with BF16 the tensor cores'
    assert rosko.rosko_kernel_launches() - l0 == 3 + bf16
    for j, (A, B, h, Bd, C) in enumerate(ls):
        a, b = (bf16_round(A), bf16_round(B)) if bf16 else (A, B)
        ref, D = spmm(a, b, C0=C0[j] if accumulate else None)
        if accumulate:
            D = D + np.abs(C0[j])
        assert normalized_error(C.cpu().numpy(), ref, D) <= 1e-5, j
