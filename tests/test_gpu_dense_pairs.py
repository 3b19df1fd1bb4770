"""The tensor-core path's work split on CTA pairs, against the FP64 oracle on
the BF16-rounded inputs (normalised error <= 1e-5, the parity bar of the dense
panel): whole tiles in several rounds with a cut remainder, more than one
column group, odd row-tile counts (a pair whose second half is empty) and
batches that mix single-tile and many-tile problems.  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_dense_panel import _run
from tests.test_gpu_spmm import _ldpad
from oracle.spmm import spmm, normalized_error
from oracle.quant import bf16_round
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,TN,ctas", [
    (384, 1100, 1300, 128, 4),     # 2 x 11 tiles on 2 pairs: rounds, two column groups
    (640, 2100, 1290, 256, 8),     # 3 x 6 tiles on 4 pairs: rounds, then 2 tiles cut
    (257, 4200, 70, 128, 0),       # 2 tiles cut over every pair
    (129, 1024, 2305, 128, 6),     # 19 tiles, K of exactly two minimum pieces
    (300, 960, 2000, 256, 10),     # K below two minimum pieces: never cut
    (256, 5100, 700, 128, 2),      # one pair, 6 tiles of 80 slabs (5 chunks) each
    (200, 9000, 900, 128, 4),      # 8 tiles of 9 chunks on two pairs, taken in turn
])
@pytest.mark.parametrize("accumulate", [False, True])
def test_pair_split(M, K, N, TN, ctas, accumulate):
    rosko = built()
    A = gen.sparse_weight(M, K, 0.6, gen.rng_for(91, M, K), "uniform")
    B = gen.normal((K, N), gen.rng_for(92, K, N))
    C0 = np.random.default_rng(6).standard_normal((M, N)).astype(np.float32) if accumulate else None
    t = rosko.make_tile(dense_split_pm=1, dense_n_r=TN, dense_split_k=ctas)
    err, launches = _run(rosko, A, B, t, accumulate=accumulate, C0=C0)
    assert err <= 1e-5, err
    assert launches == 1


def test_batch_of_single_and_many_tile_problems():
    # a few tiles of long K (cut between pairs) beside single-tile problems
    rosko = built()
    shapes = [(100, 3000, 200), (300, 2500, 300), (128, 1100, 130), (520, 1300, 257)]
    probs = [(gen.sparse_weight(M, K, 0.7, gen.rng_for(93, j), "uniform"),
              gen.normal((K, N), gen.rng_for(94, j))) for j, (M, K, N) in enumerate(shapes)]
    hs = [rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.BF16) for A, _ in probs]
    Bs = [_ldpad(torch.from_numpy(B).to(torch.bfloat16), 2) for _, B in probs]
    Cs = [torch.full((A.shape[0], B.shape[1]), float("nan"), device="cuda") for A, B in probs]
    tiles = [rosko.make_tile(dense_split_pm=1) for _ in probs]
    rosko.rosko_spmm_batched(hs, Bs, Cs, tiles=tiles)
    torch.cuda.synchronize()
    assert rosko.rosko_device_status(clear=True) == 0
    for (A, B), C in zip(probs, Cs):
        ref, D = spmm(bf16_round(A), bf16_round(B))
        assert normalized_error(C.cpu().numpy(), ref, D) <= 1e-5
