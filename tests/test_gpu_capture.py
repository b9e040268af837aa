"""The whole path under stream capture: a graph of one eviction and one decode step, or of a cascade, is
replayed over other inputs in the same buffers and gives the bits of the same calls made directly."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,dtype,hq,n", [
    (128, torch.bfloat16, 8, 3000), (64, torch.bfloat16, 8, 700), (128, torch.bfloat16, 14, 2500),   # 14: split groups
    (64, torch.float32, 8, 1500),
])
@pytest.mark.parametrize("cascade", [False, True])
def test_a_captured_pass_is_replayed_over_other_inputs(d, dtype, hq, n, cascade):
    layers, hkv, w, budget = 3, 2, 32, 150
    q, k, v, new = (torch.empty((layers,) + s, dtype=dtype, device="cuda")
                    for s in ((1, hq, w, d), (hkv, n, d), (hkv, n, d), (1, hq, d)))
    desc = lava.LayerDesc.for_tensors(q[0], k[0], v[0], w, max_seqlen=n)
    total = layers * hkv * budget
    out = torch.empty((layers, 1, hq, d), device="cuda")
    ws = torch.zeros(max(256, lava.lava_decode_workspace_bytes(desc, layers)), dtype=torch.uint8, device="cuda")
    if cascade:
        state = lava.Cascade(desc, layers, total, kv_dtype=dtype)
        budgets = torch.tensor([total], dtype=torch.int64, device="cuda")
    else:
        plan = lava.EvictionPlan.create(desc, layers, [total], [n], kv_dtype=dtype)

    def run():
        if cascade:
            state.begin(budgets)
            for l in range(layers):
                state.step(q[l], k[l], v[l])
            view = state.view()
            cache = [view[name] for name in ("k_out", "v_out", "head_offsets", "layer_row_offset")]
        else:
            lava.evict_model(plan, q, k, v)
            cache = [plan.k_out, plan.v_out, plan.head_offsets, plan.layer_row_offset]
        lava.lava_decode_attention_layers(desc, layers, new, *cache, out, ws)
        return cache + [out]

    def draw(seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        for t in (q, k, v, new):
            t.copy_(torch.randn(t.shape, generator=g, device="cuda"))

    draw(1)
    run()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        results = run()
    for seed in (2, 3, 1):
        draw(seed)
        want = [t.clone() for t in run()]
        for t in results:
            t.zero_()
        graph.replay()
        for a, b in zip(results, want):
            assert torch.equal(a, b)
