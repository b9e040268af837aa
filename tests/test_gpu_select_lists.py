"""Layer-wide selection where the threshold is found among listed candidates: how many keys share its
first digit, on both sides of what a CTA lists (2048) and of what all CTAs together do (4096), in one place
or spread over the CTAs, all distinct or tied.  Whole numbers: compared exactly with the oracle."""
import numpy as np
import pytest
import torch

import paper_2509_09754_b200 as lava
from oracle import lava_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prefix,cluster", [(4099, 0), (20011, 0), (20011, 16), (300007, 8)])
@pytest.mark.parametrize("shared", [1, 2047, 2048, 2049, 4096, 4097])
def test_thresholds_among_listed_candidates(prefix, cluster, shared):
    hkv, w, n = 2, 32, prefix + 32
    total = hkv * prefix
    desc = lava.LayerDesc(n_q_heads=hkv, n_kv_heads=hkv, head_dim=128, window=w, total_tokens=n,
                          k_stride_head=n * 128, k_stride_tok=128, v_stride_head=n * 128, v_stride_tok=128)
    rng = np.random.RandomState(shared + prefix)
    for spread in (False, True):
        for tied in (False, True):
            s = np.where(rng.rand(total) < 0.1, 4.0 + rng.rand(total), 0.5 * rng.rand(total)).astype(np.float32)
            at = rng.permutation(total)[:shared] if spread else np.arange(total - shared, total)
            # [1, 1.25): one value of the first eleven bits
            s[at] = 1.0 + (rng.randint(3, size=shared) / 16 if tied else rng.permutation(shared) / 2.0 ** 15)
            above = int((s >= 4).sum())
            for kept in {above + 1, above + (shared + 1) // 2, above + shared}:
                keep = torch.full((total,), -1, dtype=torch.int32, device="cuda")
                hoff = torch.zeros(hkv + 1, dtype=torch.int32, device="cuda")
                lava.lava_set_option("select_cluster", cluster)
                try:
                    lava.lava_select_topk(desc, torch.from_numpy(s).cuda(),
                                          torch.tensor([hkv * w + kept], dtype=torch.int64, device="cuda"), keep, hoff)
                finally:
                    lava.lava_set_option("select_cluster", 0)
                want, want_off = O.select_topk(s.reshape(hkv, prefix).astype(np.float64), hkv * w + kept, w)
                np.testing.assert_array_equal(hoff.cpu().numpy(), want_off)
                np.testing.assert_array_equal(keep.cpu().numpy()[:kept], np.concatenate(want))
