"""Layer-wide selection around the number of keys up to which it lists candidates (one key in 32, 256 to 2048)
and the part of a CTA up to which it does (65533 keys), in parts that fit shared memory and in larger ones, with
idle CTAs in the cluster and without.  Whole numbers: compared exactly with a stable sort."""
import numpy as np
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("total,cluster", [
    (998, 0), (8190, 0), (8198, 0), (28682, 16), (65534, 8), (65538, 16), (8 * 14336 - 8, 8), (8 * 14336, 8), (8 * 14336 + 2, 8),
    (400006, 8), (8 * 65533, 8), (8 * 65533 + 2, 8), (8 * 65536 + 2, 8)])
def test_lists_up_to_their_limit(total, cluster):
    hkv, w = 2, 32
    prefix, limit = total // hkv, min(2048, max(256, total // 32))
    n = prefix + w
    desc = lava.LayerDesc(n_q_heads=hkv, n_kv_heads=hkv, head_dim=128, window=w, total_tokens=n,
                          k_stride_head=n * 128, k_stride_tok=128, v_stride_head=n * 128, v_stride_tok=128)
    rng = np.random.RandomState(total)
    before = lava.lava_get_option("select_cluster")
    lava.lava_set_option("select_cluster", cluster)
    try:
        for shared in (limit - 1, limit, limit + 1):
            for tied in (False, True):
                s = np.where(rng.rand(total) < 0.3, 4.0 + rng.rand(total), 0.5 * rng.rand(total)).astype(np.float32)
                at = rng.permutation(total)[:shared] if tied else np.arange(total - shared, total)
                # [1, 1.25): one value of the first eleven bits
                s[at] = 1.0 + (rng.randint(3, size=shared) / 16 if tied else rng.permutation(shared) / 2.0 ** 15)
                order = np.argsort(-s, kind="stable")
                above = int((s >= 4).sum())
                # one short of 16 bytes at both ends: the array may start and end anywhere
                scores = torch.zeros(total + 2, device="cuda")[1:total + 1]
                scores.copy_(torch.from_numpy(s))
                for kept in (above + 1, above + shared // 2, above + shared):
                    keep = torch.full((total,), -1, dtype=torch.int32, device="cuda")
                    hoff = torch.zeros(hkv + 1, dtype=torch.int32, device="cuda")
                    lava.lava_select_topk(desc, scores, torch.tensor([hkv * w + kept], dtype=torch.int64, device="cuda"),
                                          keep, hoff)
                    flat = np.sort(order[:kept])
                    np.testing.assert_array_equal(keep.cpu().numpy()[:kept], flat % prefix)
                    first = [int((flat < h * prefix).sum()) + h * w for h in range(hkv + 1)]
                    np.testing.assert_array_equal(hoff.cpu().numpy(), first)
    finally:
        lava.lava_set_option("select_cluster", before)
