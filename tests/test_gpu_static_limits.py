"""lava_score_layer_static close to the end of its built-in scratch: batches whose layer fits it with the
generic path's long blocks only, and at head dimension 64 without the tensor-core path's share."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,n,batch", [(torch.float32, 2000, 40), (torch.bfloat16, 8000, 40)])
def test_batches_that_fit_the_scratch_with_the_smallest_layout(dtype, n, batch):
    hq, hkv, d, w = 32, 8, 64, 32
    g = torch.Generator(device="cuda").manual_seed(4)
    total = n * batch
    q = torch.randn((batch, hq, w, d), generator=g, device="cuda").to(dtype)
    k, v = (torch.randn((hkv, total, d), generator=g, device="cuda").to(dtype) for _ in range(2))
    cu = torch.arange(0, total + 1, n, dtype=torch.int32, device="cuda")
    desc = lava.LayerDesc.for_tensors(q, k, v, w, cu_seqlens=cu, max_seqlen=n)
    need = lava.lava_workspace_bytes(desc, 1)
    assert need > 8 << 20                    # with the layout that lava_score_layer uses
    got, want = ([torch.full((desc.total_scores,), -1.0, device="cuda"), torch.empty((batch, hkv), device="cuda"),
                  torch.empty(batch, dtype=torch.float64, device="cuda")] for _ in range(2))
    lava.lava_score_layer(desc, q, k, v, None, *want, torch.zeros(need, dtype=torch.uint8, device="cuda"))
    status = torch.full((1,), 77, dtype=torch.int32, device="cuda")
    lava.lava_score_layer_static(desc, q, k, v, None, *got, status)
    assert int(status[0]) == 0
    for a, b in zip(got, want):
        # two kernels, or two orders of the same fp32 sums, over logits of up to 16
        torch.testing.assert_close(a, b, rtol=1e-4, atol=0)
