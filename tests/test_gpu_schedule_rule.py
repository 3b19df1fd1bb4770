"""Searched and learned schedules where the analytic rule runs a kernel that no
candidate names (few columns of C, INT8 on the tensor cores): the autotuner
returns the rule when it wins, and the learned mode keeps it.  GPU only."""
import numpy as np
import pytest
import torch

from tests._lib import built
from tests.test_gpu_spmm import _ldpad
from paper_2307_03930_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def _problem(rosko, kind):
    M, K, N, s = (11008, 4096, 16, 0.9) if kind == "few" else (512, 4608, 3136, 0.9)
    A = torch.from_numpy(gen.sparse_weight(M, K, s, gen.rng_for(51), "uniform")).cuda()
    B = gen.normal((K, N), gen.rng_for(52))
    if kind == "few":
        return (rosko.rosko_pack(A, rosko.BF16), _ldpad(torch.from_numpy(B).to(torch.bfloat16), 2),
                torch.empty((M, N), device="cuda"), None)
    t = np.abs(B).max(0) / 127.0
    q = torch.from_numpy(np.rint(B / t).clip(-127, 127).astype(np.int8))
    return (rosko.rosko_pack(A, rosko.I8), _ldpad(q, 1), torch.empty((M, N), device="cuda"),
            torch.from_numpy(t.astype(np.float32)).cuda())


def _own(plan):
    """What the rule runs that no candidate names."""
    return plan["few_n_r"], plan["dense_tiles"]


@pytest.mark.parametrize("kind", ["few", "dequant"])
def test_autotune_keeps_the_rule_where_it_wins(kind):
    rosko = built()
    h, B, C, t = _problem(rosko, kind)
    rule = _own(rosko.rosko_spmm_plan(h, B, C, col_scale=t))
    assert any(rule)
    best, times = rosko.rosko_autotune(h, B, C, col_scale=t)
    assert len(times) == rosko.rosko_num_candidates()
    assert _own(rosko.rosko_spmm_plan(h, B, C, col_scale=t, tile=best)) == rule
    mode = rosko.make_tile(mode=rosko.SCHED_AUTOTUNE)
    assert _own(rosko.rosko_spmm_plan(h, B, C, col_scale=t, tile=mode)) == rule


@pytest.mark.parametrize("kind", ["few", "dequant"])
def test_learned_mode_keeps_the_rule(kind):
    rosko = built()
    h, B, C, t = _problem(rosko, kind)
    N, n_out = C.shape[1], rosko.rosko_num_candidates()
    f = rosko.rosko_features(h, N)
    target = next(i for i in range(n_out) if rosko.rosko_candidate(h, N, i) is not None)
    params = np.zeros(rosko.rosko_mlp_param_count(16, n_out), np.float32)
    params[-n_out + target] = 5.0
    rosko.rosko_selector_set(params, np.zeros(16), np.ones(16), f - 1, f + 1)
    rule = rosko.rosko_spmm_plan(h, B, C, col_scale=t)
    mode = rosko.make_tile(mode=rosko.SCHED_LEARNED)
    assert rosko.rosko_spmm_plan(h, B, C, col_scale=t, tile=mode) == rule
