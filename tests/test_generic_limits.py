"""The largest query group of the CUDA-core score path does not depend on the prompt's length: what is too
large is refused on the host, before any launch (no GPU needed; test_gpu_generic_split.py runs 66 heads)."""
import ctypes

import pytest

import paper_2509_09754_b200 as lava


@pytest.mark.parametrize("n", [300, 5000, 20000])
@pytest.mark.parametrize("d,w,group", [(64, 16, 78), (128, 128, 32), (64, 128, 53)])
def test_groups_beyond_the_limit_are_refused_at_any_length(d, w, group, n):
    desc = lava.LayerDesc(n_q_heads=group, n_kv_heads=1, head_dim=d, window=w, dtype=lava.LAVA_F32, total_tokens=n,
                          k_stride_head=n * d, k_stride_tok=d, v_stride_head=n * d, v_stride_tok=d)
    need = lava.lava_workspace_bytes(desc, 1)
    lib, c = lava.load_library(), desc.to_c()
    assert lib.lava_score_layer(ctypes.byref(c), 16, 16, 16, None, 16, None, 16, 16, need, None) == 2
    assert "too large for the generic score kernel" in lava.lava_last_error()
