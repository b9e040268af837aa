"""Layer-wide selection where its split over CTAs, vectors and rows can go wrong: sequences that start
off a 16-byte boundary, parts of a few keys, sizes around what one CTA takes (8192), keeps in shared
memory (14336) and keeps masks for (131072), heads shorter than a vector or a row, clusters larger than
the keys ask for.  Whole numbers: compared exactly with the oracle."""
import numpy as np
import pytest
import torch

import paper_2509_09754_b200 as lava
from oracle import lava_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv,w,prefixes,cluster,budget_parts", [
    (1, 16, (1, 2, 3, 4, 5, 6, 7), 0, (0.0, 0.5, 1.0)),
    (3, 16, (1, 127, 129, 42, 43), 0, (0.01, 0.4, 0.99)),
    (1, 32, (8191, 8192, 8193, 14335, 14337), 0, (0.001, 0.03, 0.7)),
    (5, 32, (3277, 1, 1639, 2867), 0, (0.02, 0.5)),
    (2, 32, (40, 5000, 9000), 8, (0.05, 0.9)),
    (7, 16, (2, 3, 30001, 1), 16, (0.05, 0.9)),
    (3, 32, (700001, 100001), 0, (0.004,)),
])
def test_selection_at_the_edges_of_its_split(hkv, w, prefixes, cluster, budget_parts):
    lens = [p + w for p in prefixes]
    total, batch = sum(lens), len(lens)
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32, device="cuda")
    desc = lava.LayerDesc(n_q_heads=hkv, n_kv_heads=hkv, head_dim=128, window=w, batch=batch,
                          max_seqlen=max(lens), cu_seqlens=cu, total_tokens=total,
                          k_stride_head=total * 128, k_stride_tok=128, v_stride_head=total * 128,
                          v_stride_tok=128)
    rng = np.random.RandomState(hkv * 31 + len(prefixes))
    runs = np.repeat(rng.rand(hkv * (total - batch * w) // 7 + 1), 7)  # what max pooling leaves: ties
    for s in (runs, np.round(runs, 2), np.full_like(runs, 0.5)):
        s = s[:desc.total_scores].astype(np.float32)
        for part in budget_parts:
            budgets = [hkv * w + int(part * hkv * p) for p in prefixes]
            lava.lava_set_option("select_cluster", cluster)
            try:
                keep = torch.full((desc.total_scores,), -1, dtype=torch.int32, device="cuda")
                hoff = torch.zeros(batch, hkv + 1, dtype=torch.int32, device="cuda")
                lava.lava_select_topk(desc, torch.from_numpy(s).cuda(),
                                      torch.tensor(budgets, dtype=torch.int64, device="cuda"), keep, hoff)
            finally:
                lava.lava_set_option("select_cluster", 0)
            got, off, at = keep.cpu().numpy(), hoff.cpu().numpy(), 0
            for b, p in enumerate(prefixes):
                want, want_off = O.select_topk(s[at:at + hkv * p].reshape(hkv, p).astype(np.float64),
                                               budgets[b], w)
                np.testing.assert_array_equal(off[b], want_off, err_msg=str((b, part)))
                kept = off[b][-1] - hkv * w
                np.testing.assert_array_equal(got[at:at + kept], np.concatenate(want), err_msg=str((b, part)))
                assert np.all(got[at + kept:at + hkv * p] == -1), "written beyond the selected count"
                at += hkv * p
