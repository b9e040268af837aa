"""Chunk length of split query groups on both sides of the lengths where it changes, against the
CUDA-core path.  Both sum in fp32 over keys in another order, in partial sums of at most 2048 keys: a few
times 2^-24 * sqrt(2048), below 1e-5, in the 2-norm."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens", [(8192,), (8193,), (9001, 33, 4099), (32768,), (32771,)])
def test_chunks_of_split_groups(lens):
    layers, hq, hkv, w, d, n = 5, 28, 4, 32, 128, sum(lens)   # more than sixteen tiles for each of 148 CTAs
    g = torch.Generator(device="cuda").manual_seed(3)

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda").bfloat16()

    q, k, v = randn(layers, len(lens), hq, w, d), randn(layers, hkv, n, d), randn(layers, hkv, n, d)
    cu = torch.tensor([0] + list(lens)).cumsum(0).int().cuda() if len(lens) > 1 else None
    desc = lava.LayerDesc.for_tensors(q[0], k[0], v[0], w, cu_seqlens=cu, max_seqlen=max(lens))
    assert lava.lava_score_path(desc) == 2
    out = []
    before = lava.lava_get_option("force_generic")
    try:
        for generic in (0, 1):
            lava.lava_set_option("force_generic", generic)
            ws = torch.zeros(lava.lava_workspace_bytes(desc, layers), dtype=torch.uint8, device="cuda")
            scores = torch.full((layers, desc.total_scores), -1.0, device="cuda")
            vbar = torch.empty((layers, len(lens), hkv), device="cuda")
            entropy = torch.empty((layers, len(lens)), dtype=torch.float64, device="cuda")
            lava.lava_score_layers(desc, layers, q, k, v, q.stride(0), k.stride(0), v.stride(0), None, scores,
                                   vbar, entropy, ws)
            assert lava.lava_poll_status(ws) == 0
            out.append((scores.double(), vbar.double(), entropy))
    finally:
        lava.lava_set_option("force_generic", before)
    for got, want in zip(*out):
        assert float((got - want).norm() / want.norm()) < 1e-5
