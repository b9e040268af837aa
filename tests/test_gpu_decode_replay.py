"""A captured decode call that is replayed after the row counts have changed in place: heads of one chunk
become heads of many whose partial results lie in the same slots, and back."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [128, 64])
def test_a_replay_sees_the_row_counts_of_its_own_time(d):
    layers, kv, group, longest = 8, 8, 4, 32768
    heads, total = layers * kv, 32768
    short, long = [90] * heads, [0] * heads
    for h in range(0, heads, kv):
        long[h] = 4096
    # a last chunk of one row: its block is the first to look for the others
    pairs = [[n, 0] * (heads // 2) for n in (129, 513)]
    layouts = [short, pairs[0], short, pairs[1], short, long, [500] * heads, [32768] + [0] * (heads - 1), short]
    g = torch.Generator(device="cuda").manual_seed(5)
    k, v = (torch.randn((total, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.empty((heads * group, d), dtype=torch.bfloat16, device="cuda")
    hoff = torch.zeros((layers, 1, kv + 1), dtype=torch.int32, device="cuda")
    roff = torch.zeros(layers + 1, dtype=torch.int64, device="cuda")
    out = torch.empty((heads * group, d), device="cuda")
    desc = lava.LayerDesc(n_q_heads=kv * group, n_kv_heads=kv, head_dim=d, window=16, max_seqlen=longest,
                          total_tokens=longest, k_stride_head=longest * d, k_stride_tok=d,
                          v_stride_head=longest * d, v_stride_tok=d)
    # every partial result that is read before it is written shows as a NaN
    ws = torch.full((lava.lava_decode_workspace_bytes(desc, layers),), 255, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lava.lava_decode_attention_layers(desc, layers, q, k, v, hoff, roff, out, ws)
    for rows in layouts + layouts[::-1]:
        n = torch.tensor(rows).view(layers, kv)
        q.copy_(2.0 * torch.randn((heads * group, d), generator=g, device="cuda"))
        hoff[:, 0, 1:] = n.cumsum(1).int().cuda()
        roff[1:] = n.sum(1).cumsum(0).cuda()
        out.fill_(float("nan"))
        graph.replay()
        at = 0
        for h, count in enumerate(rows):
            if count == 0:
                assert bool((out[h * group:(h + 1) * group] == 0).all())
                continue
            qh = q[h * group:(h + 1) * group].double()
            kh, vh = k[at:at + count].double(), v[at:at + count].double()
            p = torch.softmax(qh @ kh.T / d ** 0.5, dim=1)
            # bf16 probabilities: 2^-8 of the weighted magnitudes, and room for the fp32 sums
            tol = 2.0 ** -8 * (p @ vh.abs()) + 1e-6
            got = out[h * group:(h + 1) * group].double()
            assert bool(((got - p @ vh).abs() <= tol).all()), (rows, h)
            at += count
