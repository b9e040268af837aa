"""Decode attention's split of the packed rows over warps: heads without rows, of one row, on both
sides of a 16-row block and of a chunk, inside one warp's range and spread over many, for both head
dimensions and several query group sizes, in both paths (a long max_seqlen chooses the listed one); the workspace holds garbage at first and is used again."""
import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


def _reference(q, k, v, rows, group):
    out = torch.zeros(q.shape, dtype=torch.float64, device="cuda")
    mag = torch.zeros_like(out)
    at = 0
    for h, n in enumerate(rows):
        if n:
            p = torch.softmax(q[h * group:(h + 1) * group].double() @ k[at:at + n].double().T / k.shape[1] ** 0.5, dim=1)
            out[h * group:(h + 1) * group] = p @ v[at:at + n].double()
            mag[h * group:(h + 1) * group] = p @ v[at:at + n].double().abs()
        at += n
    return out, mag


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("group,rows", [
    (1, [1, 0]), (4, [16, 17, 15, 33]), (8, [0, 0, 5, 0]),
    (4, [128] * 32 + [129] * 32),               # one chunk, and a row more
    (7, [40000, 3, 0, 700]),                    # one head over many warps, chunks of more than 128 rows
    (4, [2048 + 16 * i for i in range(32)]),    # boundaries everywhere
    (2, [31] * 2000),                           # more heads than threads
    (4, [512, 513, 0, 5] + [511] * 4 + [1, 2048, 1500, 16] * 30),   # enough for the listed path
])
def test_split_over_warps(d, group, rows):
    heads, kv = len(rows), min(len(rows), 4)
    layers = heads // kv
    assert layers * kv == heads
    g = torch.Generator(device="cuda").manual_seed(7)
    total = max(1, sum(rows))
    k = torch.randn((total, d), generator=g, device="cuda").bfloat16()
    v = torch.randn((total, d), generator=g, device="cuda").bfloat16()
    q = (2.0 * torch.randn((heads * group, d), generator=g, device="cuda")).bfloat16()
    n = torch.tensor(rows, dtype=torch.int64).view(layers, kv)
    hoff = torch.zeros((layers, 1, kv + 1), dtype=torch.int64)
    hoff[:, 0, 1:] = n.cumsum(dim=1)
    roff = torch.zeros(layers + 1, dtype=torch.int64)
    roff[1:] = n.sum(dim=1).cumsum(dim=0)
    hoff, roff = hoff.int().cuda(), roff.cuda()
    longest = max(64, max(rows)) if heads != 128 else 40000
    desc = lava.LayerDesc(n_q_heads=kv * group, n_kv_heads=kv, head_dim=d, window=16, max_seqlen=longest,
                          total_tokens=longest, k_stride_head=longest * d, k_stride_tok=d,
                          v_stride_head=longest * d, v_stride_tok=d)
    ws = torch.randint(0, 256, (lava.lava_decode_workspace_bytes(desc, layers),), dtype=torch.uint8, device="cuda")
    want, mag = _reference(q, k, v, rows, group)
    # d 128 rounds the probabilities to bf16, d 64 carries them in two bf16 terms; the rest is fp32
    tol = (2.0 ** -8 if d == 128 else 2.0 ** -15) * mag + 1e-6
    for _ in range(3):
        out = torch.full((heads * group, d), float("nan"), device="cuda")
        lava.lava_decode_attention_layers(desc, layers, q, k, v, hoff, roff, out, ws)
        assert bool(((out.double() - want).abs() <= tol).all())
