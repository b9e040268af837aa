"""Decode attention at the limits of its arguments: head dimension 64 without a workspace and with
its full precision, and heads that hold more rows than max_seqlen says."""
import ctypes

import pytest
import torch

import paper_2509_09754_b200 as lava

pytestmark = pytest.mark.gpu


def _setup(d, rows, group, longest):
    g = torch.Generator(device="cuda").manual_seed(9)
    total, kv = sum(rows), len(rows)
    k, v = (torch.randn((total, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = (2.0 * torch.randn((kv * group, d), generator=g, device="cuda")).bfloat16()
    hoff = torch.tensor([[0] + torch.tensor(rows).cumsum(0).tolist()], dtype=torch.int32, device="cuda")
    roff = torch.tensor([0, total], dtype=torch.int64, device="cuda")
    desc = lava.LayerDesc(n_q_heads=kv * group, n_kv_heads=kv, head_dim=d, window=16, max_seqlen=longest,
                          total_tokens=longest, k_stride_head=longest * d, k_stride_tok=d,
                          v_stride_head=longest * d, v_stride_tok=d)
    return desc, q, k, v, hoff, roff, torch.full((kv * group, d), float("nan"), device="cuda")


def _close(out, q, k, v, rows, group, tol):
    at = 0
    for h, n in enumerate(rows):
        p = torch.softmax(q[h * group:(h + 1) * group].double() @ k[at:at + n].double().T / k.shape[1] ** 0.5, dim=1)
        err = (out[h * group:(h + 1) * group].double() - p @ v[at:at + n].double()).abs()
        assert bool((err <= tol * (p @ v[at:at + n].double().abs()) + 1e-6).all()), h
        at += n


@pytest.mark.parametrize("n_bytes", [None, 0, 64])
def test_head_dimension_64_needs_no_workspace(n_bytes):
    rows, group = [300, 17, 1000, 5], 4
    desc, q, k, v, hoff, roff, out = _setup(64, rows, group, 1024)
    room = torch.empty(256, dtype=torch.uint8, device="cuda")
    lib, c = lava.load_library(), desc.to_c()
    rc = lib.lava_decode_attention(ctypes.byref(c), q.data_ptr(), k.data_ptr(), v.data_ptr(), hoff.data_ptr(),
                                   roff.data_ptr(), out.data_ptr(), None if n_bytes is None else room.data_ptr(),
                                   n_bytes or 0, torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    _close(out, q, k, v, rows, group, 2.0 ** -15)


@pytest.mark.parametrize("d", [128, 64])
def test_heads_longer_than_max_seqlen_stay_inside_the_workspace(d):
    # a workspace of one chunk of 512 rows per head: up to there all rows count, and nothing is written past it
    rows, group = [500, 40000, 512, 513], 4
    desc, q, k, v, hoff, roff, out = _setup(d, rows, group, 300)
    n = lava.lava_decode_workspace_bytes(desc, 1)
    buf = torch.full((n + 65536,), 85, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        lava.lava_decode_attention(desc, q, k, v, hoff, roff, out, buf[:n])
    assert bool((buf[n:] == 85).all())
    tol = 2.0 ** -8 if d == 128 else 2.0 ** -15
    _close(out[:group], q[:group], k[:500], v[:500], [500], group, tol)
    at = 500 + 40000
    _close(out[2 * group:3 * group], q[2 * group:3 * group], k[at:at + 512], v[at:at + 512], [512], group, tol)
    assert bool(torch.isfinite(out).all())


@pytest.mark.parametrize("longest", [1024, 1 << 20])   # the one kernel, the listed path
@pytest.mark.parametrize("n", [40, 100, 300])
def test_head_dimension_64_rounds_nothing_to_bf16(longest, n):
    rows, group = [n] * 8, 4
    desc, q, k, v, hoff, roff, out = _setup(64, rows, group, longest)
    ws = torch.empty(lava.lava_decode_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
    lava.lava_decode_attention(desc, q, k, v, hoff, roff, out, ws)
    kh, vh = k.view(8, n, 64).double(), v.view(8, n, 64).double()
    p = torch.softmax(torch.einsum("hgd,hnd->hgn", q.view(8, group, 64).double(), kh) / 8, dim=-1)
    want = torch.einsum("hgn,hnd->hgd", p, vh).view(8 * group, 64)
    # per block of 16 rows the sums are cut off once (2^-24 on average), and about four roundings of the
    # logits (of a few units), the exponential, the sum and the quotient; two bf16 terms would give 1.8e-6
    assert float((out - want).norm() / want.norm()) <= (n / 16 + 5) * 2.0 ** -24
