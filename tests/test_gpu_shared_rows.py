"""Queries, K and V whose heads or layers share their rows (stride 0, as expand() makes them) give the same
scores, bit for bit, as copies of them; the compacted rows too."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,hq", [(128, 8), (128, 12), (64, 8)])    # 12: a split query group (6 x 32 rows)
@pytest.mark.parametrize("kernel", [0, 2])      # 2: the single-pass kernel is asked for
@pytest.mark.parametrize("shared", ["k heads", "v heads", "q layers", "k layers", "v layers", "all"])
def test_shared_rows_score_like_copies(d, hq, shared, kernel):
    layers, hkv, n, w = 3, 2, 700, 32
    g = torch.Generator(device="cuda").manual_seed(8)

    def rows(shape, one_layer, one_head=False):
        t = torch.randn((1 if one_layer else shape[0], 1 if one_head else shape[1]) + shape[2:], generator=g,
                        device="cuda").bfloat16()
        return t.expand(shape)

    q = rows((layers, 1, hq, w, d), shared in ("q layers", "all"))
    k = rows((layers, hkv, n, d), shared in ("k layers", "all"), shared in ("k heads", "all"))
    v = rows((layers, hkv, n, d), shared in ("v layers", "all"), shared in ("v heads", "all"))
    got = []
    lava.lava_set_option("score_kernel", kernel)
    try:
        for tensors in ((q, k, v), [t.contiguous() for t in (q, k, v)]):
            desc = lava.LayerDesc.for_tensors(tensors[0][0], tensors[1][0], tensors[2][0], w, max_seqlen=n)
            plan = lava.EvictionPlan.create(desc, layers, [layers * hkv * 200], [n])
            lava.evict_model(plan, *tensors)
            assert lava.lava_poll_status(plan.workspace) == 0
            got.append((plan.scores, plan.vbar, plan.entropy, plan.head_offsets, plan.k_out, plan.v_out))
    finally:
        lava.lava_set_option("score_kernel", 0)
    for a, b in zip(*got):
        if kernel == 0 or d == 64 or shared in ("v heads", "v layers"):
            assert torch.equal(a, b)
        elif a.dtype.is_floating_point and a.shape == got[0][0].shape:
            # shared Q or K take the two-pass kernel, the copies the single-pass one (fp16 exponentials)
            torch.testing.assert_close(a, b, rtol=1e-3, atol=1e-6)
