"""A workspace sized for a call serves every call of fewer layers and shorter sequences: the sizes do not
fall anywhere, across the lengths at which the kernels' blocks and paths change (no GPU needed)."""
import dataclasses

import pytest

import paper_2509_09754_b200 as lava

LENGTHS = sorted({n + e for n in (129, 300, 512, 1000, 1984, 2048, 3000, 4096, 6000, 8192, 12000, 16384, 19642, 32768,
                                  58682, 65536, 100000, 131072, 300000) for e in (-1, 0, 1, 100)})
LAYERS = (1, 2, 3, 7, 8, 16, 20, 31, 32, 47, 48, 64)


def _desc(n, **kw):
    base = dict(n_q_heads=32, n_kv_heads=8, head_dim=128, window=32, max_seqlen=n, total_tokens=n, dtype=lava.LAVA_BF16)
    base.update(kw)
    d = base["head_dim"]
    return lava.LayerDesc(**base, k_stride_head=n * d, k_stride_tok=d, v_stride_head=n * d, v_stride_tok=d)


@pytest.mark.parametrize("kw", [
    dict(), dict(head_dim=64), dict(dtype=lava.LAVA_F32), dict(dtype=lava.LAVA_F32, head_dim=64, n_q_heads=4, n_kv_heads=4),
    dict(n_q_heads=28, n_kv_heads=4), dict(window=64), dict(window=24), dict(pool_kernel=63), dict(pool_kernel=5, n_kv_heads=32),
    dict(dtype=lava.LAVA_F32, pool_kernel=31, window=16), dict(pool_kind=lava.LAVA_POOL_NONE),
])
def test_sizes_never_fall(kw):
    for size in (lava.lava_workspace_bytes, lava.lava_decode_workspace_bytes):
        by_length = [[size(_desc(n, **kw), layers) for layers in LAYERS] for n in LENGTHS]
        for row in by_length:
            assert row == sorted(row)
        for column in zip(*by_length):
            assert list(column) == sorted(column)


@pytest.mark.parametrize("dtype", [lava.LAVA_BF16, lava.LAVA_F32])
def test_a_host_arena_sized_without_max_seqlen_serves_shorter_sequences(dtype):
    # two sequences: without max_seqlen the arena is sized as if one of them held all tokens
    for total in (1000, 4100, 8200, 9000, 16500, 20000):
        d = _desc(total, dtype=dtype, batch=2, max_seqlen=0)
        sized = lava.lava_host_arena_bytes(d, 4, 4096)
        for longest in (total // 2 + 1, total // 2 + 40, total - 100):
            assert lava.lava_host_arena_bytes(dataclasses.replace(d, max_seqlen=longest), 4, 4096) <= sized
