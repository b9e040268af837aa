"""The CUDA-core score and decode kernels where their split can go wrong: prompts at the edges of a tile
of 64 keys and of a slice (48 and 64 keys, longer ones in longer sequences), pooling wider than the halo
that a slice leaves room for, windows that do not fill their rows, groups that need several batches of
query heads, both types and head dimensions.  Against plain fp32 tensor code of the same definition; the
inputs are rounded to the type first, so what differs is the order of fp32 sums of at most n terms:
2e-6 relative per logit-sized sum, and 1e-4 leaves room for the exponentials of logits up to 16."""
import pytest
import torch
import torch.nn.functional as F

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


def _reference(q, k, v, w, kind, kernel):
    hq, hkv, n, d = q.shape[0], k.shape[0], k.shape[1], k.shape[2]
    kk = k.repeat_interleave(hq // hkv, 0)
    z = q @ kk.transpose(1, 2) / d ** 0.5
    hide = torch.arange(n, device="cuda")[None] > torch.arange(n - w, n, device="cuda")[:, None]
    a = z.masked_fill(hide, float("-inf")).softmax(-1).mean(1)[:, :n - w]
    if kind == lava.LAVA_POOL_MAX:
        a = F.max_pool1d(a[None], kernel, 1, kernel // 2)[0]
    elif kind == lava.LAVA_POOL_AVG:
        a = F.avg_pool1d(a[None], kernel, 1, kernel // 2)[0]
    vbar = v.abs().sum(-1).amax(-1)
    return a.view(hkv, hq // hkv, -1).amax(1) * vbar[:, None], vbar


@pytest.mark.parametrize("dtype,d,hq,hkv,w,n,kind,kernel", [
    ("f32", 64, 8, 2, 32, 33, "MAX", 7), ("f32", 64, 8, 2, 32, 80, "MAX", 7), ("f32", 64, 8, 2, 32, 81, "AVG", 5),
    ("f32", 128, 4, 4, 16, 128 + 16, "MAX", 17), ("f32", 128, 4, 1, 7, 129 + 7, "MAX", 19),
    ("f32", 64, 16, 1, 20, 500, "MAX", 63), ("f32", 64, 40, 2, 64, 700, "NONE", 1),
    ("f32", 128, 6, 3, 128, 4096, "MAX", 7), ("f32", 64, 4, 2, 48, 4097, "AVG", 3),
    ("f32", 64, 4, 1, 16, 20000, "MAX", 7), ("f32", 64, 66, 1, 16, 20000, "MAX", 7),
    ("bf16", 64, 8, 2, 5, 1000, "MAX", 5), ("bf16", 128, 18, 2, 24, 9001, "MAX", 7),
])
def test_generic_scores_at_the_edges_of_the_split(dtype, d, hq, hkv, w, n, kind, kernel):
    gen = torch.Generator("cuda").manual_seed(n + w)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    q, k, v = (torch.randn(h, m, d, device="cuda", generator=gen).to(dt) for h, m in ((hq, w), (hkv, n), (hkv, n)))
    kind = getattr(lava, "LAVA_POOL_" + kind)
    desc = lava.LayerDesc(n_q_heads=hq, n_kv_heads=hkv, head_dim=d, window=w, total_tokens=n,
                          k_stride_head=n * d, k_stride_tok=d, v_stride_head=n * d, v_stride_tok=d,
                          dtype=lava.LAVA_F32 if dtype == "f32" else lava.LAVA_BF16,
                          pool_kind=kind, pool_kernel=kernel)
    scores = torch.full((desc.total_scores,), -1.0, device="cuda")
    vbar = torch.empty(hkv, device="cuda")
    ent = torch.empty(1, dtype=torch.float64, device="cuda")
    work = torch.full((lava.lava_workspace_bytes(desc, 1),), 255, dtype=torch.uint8, device="cuda")
    lava.lava_set_option("force_generic", 1)
    try:
        lava.lava_score_layer(desc, q, k, v, None, scores, vbar, ent, work)
    finally:
        lava.lava_set_option("force_generic", 0)
    want, want_vbar = _reference(q.double(), k.double(), v.double(), w, kind, kernel)
    torch.testing.assert_close(vbar.double(), want_vbar, rtol=1e-5, atol=0)
    torch.testing.assert_close(scores.double().view(hkv, -1), want, rtol=1e-4, atol=0)
    p = want / want.sum()
    torch.testing.assert_close(ent, (-(p * p.log()).sum() / (hkv * n)).view(1), rtol=1e-4, atol=0)


@pytest.mark.parametrize("dtype,d,group", [("f32", 64, 1), ("f32", 128, 4), ("bf16", 64, 9), ("bf16", 128, 16)])
def test_generic_decode_at_the_edges_of_the_split(dtype, d, group):
    hkv, lens = 7, (0, 1, 31, 32, 1023, 1025, 2500)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator("cuda").manual_seed(d + group)
    rows = sum(lens)
    q = torch.randn(1, hkv * group, d, device="cuda", generator=gen).to(dt)
    k, v = (torch.randn(rows, d, device="cuda", generator=gen).to(dt) for _ in range(2))
    off = torch.tensor([[sum(lens[:i]) for i in range(hkv + 1)]], dtype=torch.int32, device="cuda")
    desc = lava.LayerDesc(n_q_heads=hkv * group, n_kv_heads=hkv, head_dim=d, window=1, total_tokens=4000,
                          k_stride_head=4000 * d, k_stride_tok=d, v_stride_head=4000 * d, v_stride_tok=d,
                          dtype=lava.LAVA_F32 if dtype == "f32" else lava.LAVA_BF16)
    out = torch.full((1, hkv * group, d), 9.0, device="cuda")
    work = torch.empty(lava.lava_decode_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
    lava.lava_decode_attention(desc, q, k, v, off, torch.zeros(2, dtype=torch.int64, device="cuda"), out, work)
    for h in range(hkv * group):
        a, b = int(off[0, h // group]), int(off[0, h // group + 1])
        want = torch.zeros(d, dtype=torch.float64, device="cuda")
        if b > a:
            want = (k[a:b].double() @ q[0, h].double() / d ** 0.5).softmax(0) @ v[a:b].double()
        torch.testing.assert_close(out[0, h].double(), want, rtol=1e-4, atol=1e-6)
