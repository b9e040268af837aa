"""The descriptor's kept C structure when something happens between two steps of a call, as another thread
may do: a field is set while the structure is being filled, the lengths move while a call uses it."""
import pytest
import torch

import paper_2509_09754_b200 as lava


def _desc(cls=lava.LayerDesc):
    return cls(n_q_heads=8, n_kv_heads=2, head_dim=128, window=32, total_tokens=512, k_stride_tok=128,
               cu_seqlens=torch.tensor([0, 200, 512], dtype=torch.int32), batch=2)


@pytest.mark.parametrize("first", [True, False])
def test_a_field_set_while_the_structure_is_filled(first):
    class Overtaken(lava.LayerDesc):
        def to_c(self):
            c = super().to_c()
            if armed.pop("now", False):
                self.window = 64            # what another thread does after the fields have been read
            return c

    armed = {}
    d = _desc(Overtaken)
    if not first:
        d._for_call()
        d.flags = 0
    armed["now"] = True
    d._for_call()                           # may have either window
    assert d._for_call().window == 64 and d._for_call().window == 64


def test_a_structure_in_use_is_not_written():
    d = _desc()
    used = d._for_call()
    before = used.cu_seqlens
    d.cu_seqlens.set_(torch.tensor([0, 1, 2], dtype=torch.int32))
    assert d._for_call().cu_seqlens == d.cu_seqlens.data_ptr() != before
    assert used.cu_seqlens == before


def test_a_used_descriptor_holds_nothing_but_its_fields():
    d = _desc()
    d._for_call()
    assert lava.LayerDesc(**vars(d)) == d
    del d.flags                             # back to the class's default
    assert d._for_call().flags == 0
