"""Layer entropy taken from the final score array (split query groups): one block per (layer,
sequence) up to 32768 scores, slices and a second launch beyond; checked on both sides of the line."""
import numpy as np
import pytest
import torch

import paper_2509_09754_b200 as lava
from lava_workloads import get_config
from tests.parity_harness import ENTROPY_RTOL, upload_model

pytestmark = pytest.mark.gpu

W = 64      # G 4 x w 64: the query group is scored as two halves


@pytest.mark.parametrize("lens", [
    (W,), (W + 1,), (W + 511,),                   # no candidates, one per head, a block's worth
    (W + 4096,), (W + 4097,), (W + 8193,),        # 32768 scores: one block; two and three slices
    (W + 9000, W + 1, W, W + 700),                # a batch: the longest sequence sets the slices
])
def test_entropy_of_split_groups_matches_the_scores(lens):
    cfg = get_config("mistral7b_ragged").scaled(seq_lens=lens, n_layers=1, needle=False)
    q, k, v, cu = upload_model(cfg)
    desc = lava.LayerDesc.for_tensors(q[0], k[0], v[0], W, cfg.pool_kind, cfg.pool_kernel,
                                      cu_seqlens=cu if cfg.batch > 1 else None, max_seqlen=max(lens))
    assert lava.lava_score_path(desc) == 2
    ws = torch.zeros(lava.lava_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
    sc = torch.empty(max(1, desc.total_scores), device="cuda")
    vbar = torch.empty((cfg.batch, cfg.n_kv_heads), device="cuda")
    ent = torch.full((cfg.batch,), -1.0, dtype=torch.float64, device="cuda")
    lava.lava_score_layer(desc, q[0], k[0], v[0], None, sc, vbar, ent, ws)
    assert lava.lava_poll_status(ws) == 0
    got, scores, at = ent.cpu().numpy(), sc.cpu().numpy().astype(np.float64), 0
    for b, n in enumerate(lens):
        s = scores[at: at + cfg.n_kv_heads * (n - W)]
        at += s.size
        s = s[s > 0]
        want = 0.0
        if s.size:
            p = s / s.sum()
            want = -(p * np.log(p)).sum() / (cfg.n_kv_heads * n)
        assert abs(got[b] - want) <= ENTROPY_RTOL * abs(want) + 1e-15
