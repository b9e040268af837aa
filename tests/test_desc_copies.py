"""The descriptor's C structure is kept between calls: it has to follow every change of a field, and
copies and pickles of a descriptor that has been used must work and be independent."""
import copy
import dataclasses
import pickle

import torch

import paper_2509_09754_b200 as lava


def _fields(c):
    return {n: getattr(c, n) for n, _ in c._fields_}


def test_the_structure_of_a_call_follows_its_descriptor():
    d = lava.LayerDesc(n_q_heads=8, n_kv_heads=2, head_dim=128, window=32, total_tokens=512, k_stride_tok=128,
                       cu_seqlens=torch.tensor([0, 200, 512], dtype=torch.int32), batch=2)
    first = d._for_call()
    assert _fields(first) == _fields(d.to_c()) and d._for_call() is first
    for name, value in dict(window=64, sm_scale=0.5, flags=2, cu_seqlens=torch.zeros(3, dtype=torch.int32),
                            total_tokens=600).items():
        old = d._for_call()
        setattr(d, name, value)
        assert d._for_call() is not old and _fields(d._for_call()) == _fields(d.to_c())
    d.cu_seqlens.set_(torch.tensor([0, 1, 2], dtype=torch.int32))     # the storage moves under the tensor
    assert _fields(d._for_call()) == _fields(d.to_c())
    d.cu_seqlens = None
    assert d._for_call().cu_seqlens is None
    for other in (copy.copy(d), copy.deepcopy(d), pickle.loads(pickle.dumps(d)), dataclasses.replace(d)):
        assert other == d and _fields(other._for_call()) == _fields(d._for_call())
        other.window = 16
        assert d._for_call().window == 64 and other._for_call().window == 16
