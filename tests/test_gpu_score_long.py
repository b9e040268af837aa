"""Scores of sequences long enough for the chunks to be lengthened (see test_score_lead_long.py)."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,group,chunk_tiles", [
    (1_200_000, 7, 0),      # split query group
    (1_800_000, 4, 0),      # one unit per KV head
    (300_000, 4, 1),        # a chunk length that is asked for and too short
])
def test_scores_of_long_sequences(n, group, chunk_tiles):
    d, w = 64, 32
    g = torch.Generator(device="cuda").manual_seed(1)
    k, v = (torch.randn((1, n, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((1, group, w, d), generator=g, device="cuda").bfloat16()
    desc = lava.LayerDesc.for_tensors(q, k, v, w, max_seqlen=n)
    scores = torch.full((n - w,), -1.0, device="cuda")
    vbar, entropy = torch.empty(1, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
    before = lava.lava_get_option("score_chunk_tiles")
    lava.lava_set_option("score_chunk_tiles", chunk_tiles)
    try:
        ws = torch.zeros(lava.lava_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
        lava.lava_score_layer(desc, q, k, v, None, scores, vbar, entropy, ws)
        assert lava.lava_poll_status(ws) == 0
    finally:
        lava.lava_set_option("score_chunk_tiles", before)
    # scores of every head from the softmax over all keys that a window query sees
    best = torch.zeros(n - w, dtype=torch.float64, device="cuda")
    for h in range(group):
        z = q[0, h].double() @ k[0].double().T / d ** 0.5
        z.masked_fill_(torch.arange(n, device="cuda")[None] > (n - w + torch.arange(w, device="cuda"))[:, None],
                       float("-inf"))
        a = torch.softmax(z, dim=1).mean(dim=0)[:n - w]
        best = torch.maximum(best, torch.nn.functional.max_pool1d(a[None, None], 7, 1, 3)[0, 0])
    want = best * v.double().abs().sum(-1).max()
    assert bool(((scores.double() - want).abs() <= 1e-3 * want + 1e-6 * want.max()).all())
    assert float((scores.double() - want).norm() / want.norm()) < 1e-5
