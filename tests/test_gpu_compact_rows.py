"""Compaction of calls large enough for two rows on their way per thread: heads of a window only, of one
row more, of odd and of many rows.  Bytes: compared exactly with an indexed copy."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,n", [(torch.bfloat16, 128, 80001), (torch.float32, 64, 80003)])
def test_rows_of_large_calls(dtype, d, n):
    layers, hkv, w = 2, 8, 32                       # more than 300 MB of K
    g = torch.Generator(device="cuda").manual_seed(5)
    k, v = (torch.randn((layers, hkv, n, d), generator=g, device="cuda").to(dtype) for _ in range(2))
    desc = lava.LayerDesc(n_q_heads=hkv, n_kv_heads=hkv, head_dim=d, window=w, total_tokens=n,
                          dtype=lava.LAVA_BF16 if dtype == torch.bfloat16 else lava.LAVA_F32,
                          k_stride_head=n * d, k_stride_tok=d, v_stride_head=n * d, v_stride_tok=d)
    counts = [[0, 1, 15, 16, 17, 4097, 20011, 1], [n - w, 0, 31, 33, 1000, 511, 513, 7]]
    keep = torch.full((layers, desc.total_scores), -1, dtype=torch.int32, device="cuda")
    hoff = torch.zeros((layers, hkv + 1), dtype=torch.int32)
    want = []
    for l in range(layers):
        at = 0
        for h, c in enumerate(counts[l]):
            pos = torch.randperm(n - w, generator=g, device="cuda")[:c].sort().values
            keep[l, at:at + c] = pos.int()
            at += c
            hoff[l, h + 1] = hoff[l, h] + c + w
            rows = torch.cat([pos, torch.arange(n - w, n, device="cuda")])
            want.append((k[l, h, rows], v[l, h, rows]))
    roff = torch.tensor([0, int(hoff[0, -1]), int(hoff[0, -1] + hoff[1, -1])], dtype=torch.int64, device="cuda")
    out = [torch.zeros((int(roff[-1]) + 1, d), dtype=dtype, device="cuda") for _ in range(2)]
    lava.lava_compact_kv_layers(desc, layers, k, v, k.stride(0), v.stride(0), keep, hoff.cuda(), roff, *out)
    for got, rows in zip(out, zip(*want)):
        assert torch.equal(got[:-1], torch.cat(rows))
        assert not got[-1].any()                    # nothing beyond the last row
