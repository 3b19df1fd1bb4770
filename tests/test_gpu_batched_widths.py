"""Batches whose row-direct remainders have different strip widths (n_r): the
zero fill ahead of the launches and the launches agree on width and row pieces,
so that no problem's finished tensor-core tiles are zeroed again.  Within 1e-5
of the normalised error (the parity bar).  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad
from oracle.quant import bf16_round
from oracle.spmm import normalized_error, spmm
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def _problems():
    """An even layer; one of 1100 rows of ~150 nonzeros (three pieces in the
    fine list, whole in the coarse one) whose second 128-row tile is the only
    one above 12 per mille; a ragged one; and one with enough tensor-core tiles
    that the launch it shares with that tile deals whole tiles (no zero fill)."""
    out = [(gen.sparse_weight(300, 1000, 0.99, gen.rng_for(91), "uniform"), 512)]
    A = gen.sparse_weight(1100, 16384, 0.9905, gen.rng_for(92), "uniform")
    A[128:256] = gen.sparse_weight(128, 16384, 0.985, gen.rng_for(93), "uniform")
    out.append((A, 1024))
    out.append((gen.sparse_weight(200, 700, 0.95, gen.rng_for(94), "powerlaw"), 300))
    out.append((gen.sparse_weight(2048, 1088, 0.9, gen.rng_for(97), "uniform"), 5120))
    return [(A, gen.relu_normal((A.shape[1], N), gen.rng_for(95, j))) for j, (A, N) in enumerate(out)]


@pytest.mark.parametrize("widths", [(128, 0, 128), (128, 512, 256), (256, 128, 512), (0, 512, 0)])
@pytest.mark.parametrize("accumulate", [False, True])
def test_mixed_widths_keep_every_tile(widths, accumulate):
    rosko = built()
    probs = _problems()
    tiles = [rosko.make_tile(n_r=w, dense_split_pm=pm) for w, pm in zip(widths + (0,), (1001, 12, 1001, 12))]
    hs = [rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.BF16) for A, _ in probs]
    Bs = [_ldpad(torch.from_numpy(B).to(torch.bfloat16), 2) for _, B in probs]
    C0s = [np.random.default_rng(j).standard_normal((A.shape[0], B.shape[1])).astype(np.float32)
           for j, (A, B) in enumerate(probs)]
    Cs = [torch.from_numpy(C0).cuda() for C0 in C0s]
    l0 = rosko.rosko_kernel_launches()
    rosko.rosko_spmm_batched(hs, Bs, Cs, accumulate=accumulate, tiles=tiles)
    # one tensor-core launch and one row-direct launch per width
    assert rosko.rosko_kernel_launches() - l0 <= 1 + len({w or 256 for w in widths})
    for j, ((A, B), C) in enumerate(zip(probs, Cs)):
        rows = np.unique(np.r_[0:A.shape[0]:11, 128:min(256, A.shape[0]):9])
        ref, D = spmm(bf16_round(A[rows]), bf16_round(B), C0=C0s[j][rows] if accumulate else None)
        if accumulate:
            D = D + np.abs(C0s[j][rows])
        assert normalized_error(C.cpu().numpy()[rows], ref, D) <= 1e-5, j


def test_width_below_a_warp_is_refused():
    """A strip narrower than 32 columns is an invalid tile, in a batch as in a
    single call."""
    rosko = built()
    A = gen.sparse_weight(512, 4096, 0.5, gen.rng_for(96), "uniform")
    h = rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.BF16)
    B = torch.zeros((4096, 64), dtype=torch.bfloat16, device="cuda")
    C = torch.zeros((512, 64), device="cuda")
    t = rosko.make_tile(n_r=16, dense_split_pm=1001)
    with pytest.raises(RuntimeError, match="INVALID_ARG"):
        rosko.rosko_spmm(h, B, C, tile=t)
    with pytest.raises(RuntimeError, match="INVALID_ARG"):
        rosko.rosko_spmm_batched([h], [B], [C], tiles=[t])
