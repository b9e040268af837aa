"""Tensor-core score kernel at the edges of its tiles, chunks and value pieces, for both head
dimensions, and its fallback to a running maximum."""
import numpy as np
import pytest
import torch

import paper_2509_09754_b200 as lava
from lava_workloads import get_config, to_numpy64
from oracle import lava_oracle as O
from tests.parity_harness import SCORE_ATOL, SCORE_RTOL, compare_eviction, make_plan, upload_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,kw", [
    (64, dict(seq_lens=(33,))),                                # one candidate
    (64, dict(seq_lens=(128,))), (64, dict(seq_lens=(129,))),  # a tile and one more
    (64, dict(seq_lens=(513,), window=16, n_kv_heads=2)),      # a chunk and one more, group 16
    (64, dict(seq_lens=(1000,), window=128, n_q_heads=8)),     # one query head fills the tile
    (64, dict(seq_lens=(700, 64, 1301), window=64, pool_kind=2, pool_kernel=5)),   # split, ragged, avg
    (64, dict(seq_lens=(2600,), n_q_heads=28, n_kv_heads=4, pool_kind=0)),         # split 4 + 3 heads
    (128, dict(seq_lens=(32, 545, 33))),                       # a sequence without candidates
    (128, dict(seq_lens=(609,), window=16, n_q_heads=16)),
    (128, dict(seq_lens=(4097,), n_layers=3, pool_kernel=63)),  # widest halo
])
def test_tile_edges_match_the_oracle(d, kw):
    kw = dict(dict(n_layers=2, head_dim=d), **kw)
    cfg = get_config("llama8b_8k").scaled(**kw)
    w = cfg.window
    budget = max(w, (min(cfg.seq_lens) + w) // 2)
    compare_eviction(cfg.scaled(budget_per_head=budget))


@pytest.mark.parametrize("d", [64, 128])
def test_logits_far_above_the_first_block(d):
    """The first 40 keys are small, the rest large: exponentials relative to the first block's maximum
    would overflow, so the tile is done again with a running maximum."""
    cfg = get_config("llama8b_8k").scaled(seq_lens=(900,), n_layers=1, head_dim=d, budget_per_head=200)
    q, k, v, cu = upload_model(cfg)
    k[:, :, :40] *= 0.01
    k[:, :, 40:] *= 25.0
    plan = make_plan(cfg, q, k, v, cu)
    lava.evict_model(plan, q, k, v)
    assert lava.lava_poll_status(plan.workspace) == 0
    want = O.lava_scores(to_numpy64(q[0, 0]), to_numpy64(k[0]), to_numpy64(v[0]), cfg.window, cfg.pool_kind,
                         cfg.pool_kernel)
    got = plan.scores[0].cpu().numpy().reshape(want.shape).astype(np.float64)
    assert np.isfinite(got).all()
    # logits of magnitude 300 carry 300 * 2^-24 * (a few roundings of the 128-term sums) into the
    # exponent: well inside the relative tolerance of the scores
    assert np.all(np.abs(got - want) <= SCORE_RTOL * np.abs(want) + SCORE_ATOL)
