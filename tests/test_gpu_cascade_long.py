"""Cascades long enough for what short ones do not reach: both selections of a step run side by side for most
of their time, the lists need several CTAs each, and steps move enough rows for two of them per thread.  The
state after some steps is compared with the oracle's cascade on the same stored scores, bytes exactly."""
import numpy as np
import pytest
import torch

import paper_2509_09754_b200 as lava
from oracle import lava_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,hq,hkv,n,per_head,looks", [
    (20, 16, 8, 8192, 1024, (7, 19, 20)),
    (12, 8, 4, 30011, 4000, (2, 12)),
    (20, 16, 8, 8192, 64, (20,)),
])
def test_long_cascade_matches_the_oracle(layers, hq, hkv, n, per_head, looks):
    w, d = 32, 128
    g = torch.Generator(device="cuda").manual_seed(layers + n)

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    # layers of different sharpness, so that budgets differ
    q = (randn(layers, 1, hq, w, d) * torch.linspace(0.5, 2.0, layers, device="cuda").view(-1, 1, 1, 1, 1)).bfloat16()
    k, v = randn(layers, hkv, n, d).bfloat16(), randn(layers, hkv, n, d).bfloat16()
    desc = lava.LayerDesc.for_tensors(q[0], k[0], v[0], w, max_seqlen=n)
    ws = torch.zeros(lava.lava_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
    scores = torch.empty((layers, desc.total_scores), device="cuda")
    entropy = torch.empty((layers, 1), dtype=torch.float64, device="cuda")
    vbar = torch.empty((1, hkv), device="cuda")
    for l in range(layers):
        lava.lava_score_layer(desc, q[l], k[l], v[l], None, scores[l], vbar, entropy[l], ws)
    stored = [s.reshape(hkv, n - w).astype(np.float64) for s in scores.cpu().numpy()]
    ent = entropy.cpu().numpy()[:, 0]

    total = layers * hkv * per_head
    cas = lava.Cascade(desc, layers, total, kv_dtype=k.dtype)
    cas.begin(torch.tensor([total], dtype=torch.int64, device="cuda"))
    for l in range(layers):
        cas.step(q[l], k[l], v[l])
        if l + 1 not in looks:
            continue
        assert lava.lava_poll_status(cas.workspace) == 0
        view = cas.view()
        np.testing.assert_array_equal(view["entropy"].cpu().numpy()[:l + 1, 0], ent[:l + 1])
        keep, budgets, _ = O.cascade_evict(stored[:l + 1], n, w, total, entropy=ent[:l + 1])
        assert view["layer_budget"].cpu().numpy()[:l + 1, 0].tolist() == budgets
        hoff, roff = view["head_offsets"].cpu().numpy(), view["layer_row_offset"].cpu().numpy()
        pos = view["kept_pos"].cpu().numpy()
        for t in range(l + 1):
            r0 = int(roff[t])
            for h in range(hkv):
                a, e = int(hoff[t, 0, h]), int(hoff[t, 0, h + 1])
                at = r0 + a - h * w
                np.testing.assert_array_equal(pos[at:at + e - a - w], keep[t][h])
                rows = torch.from_numpy(np.concatenate([keep[t][h], np.arange(n - w, n)])).cuda()
                assert e - a == len(rows)
                assert torch.equal(view["k_out"][r0 + a:r0 + e], k[t, h, rows])
                assert torch.equal(view["v_out"][r0 + a:r0 + e], v[t, h, rows])
    cas.close()
