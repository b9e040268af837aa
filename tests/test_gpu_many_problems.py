"""Calls of more (layer, sequence) problems than a grid's second and third dimensions can hold."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


def test_cascade_of_65536_layers_and_sequences():
    layers, batch, n, d, w = 64, 1024, 4, 64, 1
    g = torch.Generator(device="cuda").manual_seed(6)
    q = torch.randn((layers, batch, 1, w, d), generator=g, device="cuda")
    k, v = (torch.randn((layers, 1, batch * n, d), generator=g, device="cuda") for _ in range(2))
    total = torch.full((batch,), 2 * layers, dtype=torch.int64, device="cuda")   # two rows a layer on average

    def run(b0, b1):
        cu = torch.arange(0, (b1 - b0) * n + 1, n, dtype=torch.int32, device="cuda")
        qs, ks, vs = q[:, b0:b1].contiguous(), k[:, :, b0 * n:b1 * n].contiguous(), v[:, :, b0 * n:b1 * n].contiguous()
        desc = lava.LayerDesc.for_tensors(qs[0], ks[0], vs[0], w, cu_seqlens=cu, max_seqlen=n)
        cas = lava.Cascade(desc, layers, 2 * layers * (b1 - b0), kv_dtype=k.dtype)
        cas.begin(total[b0:b1].contiguous())
        for l in range(layers):
            cas.step(qs[l], ks[l], vs[l])
        view = {name: t.clone() for name, t in cas.view().items() if torch.is_tensor(t)}
        cas.close()
        return view

    whole, halves = run(0, batch), [run(0, batch // 2), run(batch // 2, batch)]
    for name in ("layer_budget", "head_offsets"):
        parts = [h[name].view(layers, batch // 2, -1) for h in halves]
        assert torch.equal(whole[name].view(layers, batch, -1), torch.cat(parts, dim=1))
    rows = whole["layer_row_offset"].view(-1)[:layers * batch + 1]
    for i, half in enumerate(halves):
        part = half["layer_row_offset"].view(-1)[:layers * batch // 2 + 1]
        for l in range(layers):   # a layer's sequences of one half lie together in both
            a, b = int(rows[l * batch + i * batch // 2]), int(rows[l * batch + (i + 1) * batch // 2])
            c, e = int(part[l * batch // 2]), int(part[(l + 1) * batch // 2])
            for name in ("k_out", "v_out"):
                assert torch.equal(whole[name][a:b], half[name][c:e])


def test_entropies_of_66048_layers_and_sequences():
    # a split query group (16 x 16 rows), whose entropies are taken from the final scores; one layer's
    # inputs stand for all
    layers, batch, n, d, w, group = 129, 512, 40, 64, 16, 16
    g = torch.Generator(device="cuda").manual_seed(7)
    q = torch.randn((1, batch, group, w, d), generator=g, device="cuda").bfloat16().expand(layers, -1, -1, -1, -1)
    k, v = (torch.randn((1, 1, batch * n, d), generator=g, device="cuda").bfloat16().expand(layers, -1, -1, -1)
            for _ in range(2))
    cu = torch.arange(0, batch * n + 1, n, dtype=torch.int32, device="cuda")
    desc = lava.LayerDesc.for_tensors(q[0], k[0], v[0], w, cu_seqlens=cu, max_seqlen=n)

    def score(count):
        out = (torch.empty((count, desc.total_scores), device="cuda"), torch.empty((count, batch, 1), device="cuda"),
               torch.empty((count, batch), dtype=torch.float64, device="cuda"))
        ws = torch.zeros(lava.lava_workspace_bytes(desc, count), dtype=torch.uint8, device="cuda")
        lava.lava_score_layers(desc, count, q, k, v, q.stride(0), k.stride(0), v.stride(0), None, *out, ws)
        assert lava.lava_poll_status(ws) == 0
        return out

    one, many = score(1), score(layers)
    for a, b in zip(one, many):
        assert bool((b == a).all())
