"""Work segments of the row-direct traversal, planned on the device: every row
covered once whatever its length (empty, one piece, many pieces), the panel
height, the block boundaries of the planning kernels (256 rows) and the list a
launch takes (all panels, or those below the dense split).  An image of an
earlier library, which also held the segments in row order, still loads.
FP32 / BF16 within 1e-5 of the normalised error, INT8 exact.  GPU only."""
import struct

import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad, check, run
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def _rows(M, K, lengths, seed):
    """M x K with row i holding lengths[i] nonzeros."""
    rng = np.random.default_rng(seed)
    A = np.zeros((M, K), np.float32)
    for i, n in enumerate(lengths):
        if n:
            A[i, rng.choice(K, n, replace=False)] = rng.standard_normal(n).astype(np.float32) + 3.0
    return A


@pytest.mark.parametrize("mode", ["f32", "bf16", "i8"])
@pytest.mark.parametrize("m_r", [8, 16, 32])
def test_lengths_and_blocks(mode, m_r):
    rosko = built()
    M, K, N = 517, 1300, 70
    rng = np.random.default_rng(3)
    lengths = rng.integers(0, 40, M)
    lengths[[0, 255, 256, 511, 516]] = [64, 65, 0, 1300, 129]   # block edges, exact pieces
    lengths[300:310] = 700                                       # several cut rows together
    A = _rows(M, K, lengths, 4)
    B = gen.normal((K, N), gen.rng_for(5))
    for pm in (1001, 60):   # every panel row-direct; the densest tile elsewhere
        t = rosko.make_tile(order=4, dense_split_pm=pm)
        check(mode, *run(rosko, A, B, mode, m_r=m_r, tile=t))


def test_even_long_rows_use_one_piece_each():
    # mean 300: the coarse list keeps rows whole up to 608 records
    rosko = built()
    A = _rows(300, 900, np.full(300, 300), 6)
    A[7] = 1.0
    B = gen.normal((900, 130), gen.rng_for(7))
    for n_r in (128, 256):
        t = rosko.make_tile(order=4, n_r=n_r, dense_split_pm=1001)
        check("bf16", *run(rosko, A, B, "bf16", m_r=16, tile=t))


def test_all_empty_rows_but_one():
    rosko = built()
    lengths = np.zeros(600, int)
    lengths[599] = 200
    A = _rows(600, 250, lengths, 8)
    B = gen.normal((250, 33), gen.rng_for(9))
    check("f32", *run(rosko, A, B, "f32", m_r=16, tile=rosko.make_tile(order=4)))


def _fnv1a(data):
    h = 1469598103934665603
    for b in data:
        h = ((h ^ b) * 1099511628211) & 0xFFFFFFFFFFFFFFFF
    return h


def test_image_with_row_order_segments_loads():
    rosko = built()
    A = _rows(40, 200, np.full(40, 9), 10)
    h = rosko.rosko_pack(torch.from_numpy(A).cuda(), rosko.BF16)
    img = bytearray(rosko.rosko_pack_save(h))
    at = 112 + 14 * 8                     # the header's pointer slot 14 (of 20)
    assert struct.unpack_from("<q", img, at)[0] == -1
    struct.pack_into("<q", img, at, 256)
    struct.pack_into("<q", img, at + 16, 256)
    struct.pack_into("<Q", img, len(img) - 8, _fnv1a(img[:-8]))
    h2 = rosko.rosko_pack_load(bytes(img))
    B = _ldpad(torch.from_numpy(gen.normal((200, 40), gen.rng_for(11))).to(torch.bfloat16), 2)
    C, C2 = torch.empty((40, 40), device="cuda"), torch.empty((40, 40), device="cuda")
    rosko.rosko_spmm(h, B, C)
    rosko.rosko_spmm(h2, B, C2)
    assert torch.equal(C, C2)
