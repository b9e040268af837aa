"""A layer's decode attention is the same, bit for bit, alone and in a call of many layers that takes the
listed path, and on both sides of the lines between the paths; rows on both sides of a block, of a part
(128 rows) and of a chunk (512)."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


def _cache(rows, d, group):
    """rows [layers, kv]: queries, packed K and V and their offsets."""
    layers, kv = rows.shape
    hoff = torch.zeros((layers, 1, kv + 1), dtype=torch.int64)
    hoff[:, 0, 1:] = rows.cumsum(dim=1)
    roff = torch.zeros(layers + 1, dtype=torch.int64)
    roff[1:] = rows.sum(dim=1).cumsum(dim=0)
    g = torch.Generator(device="cuda").manual_seed(3)
    k, v = (torch.randn((int(roff[-1]), d), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = (2.0 * torch.randn((layers, 1, kv * group, d), generator=g, device="cuda")).bfloat16()
    return q, k, v, hoff.int().cuda(), roff.cuda()


def _desc(kv, group, d, longest):
    return lava.LayerDesc(n_q_heads=kv * group, n_kv_heads=kv, head_dim=d, window=16, max_seqlen=longest,
                          total_tokens=longest, k_stride_head=longest * d, k_stride_tok=d,
                          v_stride_head=longest * d, v_stride_tok=d)


def _decode(desc, layers, q, k, v, hoff, roff):
    ws = torch.empty(lava.lava_decode_workspace_bytes(desc, layers), dtype=torch.uint8, device="cuda")
    out = torch.empty(q.shape, device="cuda")
    lava.lava_decode_attention_layers(desc, layers, q, k, v, hoff, roff, out, ws)
    return out


@pytest.mark.parametrize("d,group", [(128, 4), (64, 7)])
def test_a_layer_gives_the_same_bits_alone_and_among_others(d, group):
    kv, layers, longest = 4, 64, 16384          # 4.2 M rows at most together, 65 536 alone
    sizes = [1, 15, 17, 100, 127, 128, 129, 255, 300, 385, 511, 512, 513, 640, 1025, 2000, 5000, 0]
    rows = torch.tensor([sizes[(5 * i) % len(sizes)] for i in range(layers * kv)]).view(layers, kv)
    q, k, v, hoff, roff = _cache(rows, d, group)
    desc = _desc(kv, group, d, longest)
    out = _decode(desc, layers, q, k, v, hoff, roff)
    for l in range(layers):
        assert torch.equal(_decode(desc, 1, q[l:l + 1], k, v, hoff[l], roff[l:]), out[l:l + 1])


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("layers,kv,rows,here,there", [
    (1, 4, [131072, 700, 0, 4], 131072, 131073),   # as many chunks as the one kernel's fold looks at
    (8, 4, [1500, 3, 129, 640], 90000, 100000),    # rows at most: 2.9 and 3.2 M
    (75, 4, [600, 3, 129, 1030], 8700, 8800),      # more heads than blocks at once: 2.61 and 2.64 M
])
def test_both_paths_give_the_same_bits(d, layers, kv, rows, here, there):
    group = 4
    args = _cache(torch.tensor(rows * layers).view(layers, kv), d, group)
    assert torch.equal(_decode(_desc(kv, group, d, here), layers, *args),
                       _decode(_desc(kv, group, d, there), layers, *args))
