"""Argument marshalling of the binding's extension module: what it must reject before any call is made (no GPU needed)."""
import pytest
import torch

import paper_2606_18394_b200 as jet
from paper_2606_18394_b200 import binding


def _layer_call(layer, **kw):
    q = torch.zeros((2, 1, 4, 2, 64), dtype=torch.bfloat16)
    i32 = torch.zeros(4, dtype=torch.int32)
    args = dict(q=q, k_cache=q, v_cache=q, page_table=None, max_pages_per_seq=0, page_size=0, num_pages=0, seq_len=i32,
                max_seq_len=-1, tree_k=q, tree_v=q, anc_mask=i32, n_nodes=i32, batch=1, B=4, Hq=2, Hkv=2, D=64,
                kv_batch_stride=0, softmax_scale=1.0, out=q, lse=None, device_status=None, workspace=i32, flags=0, tail=False,
                stream=0)
    args.update(kw)
    binding.verify_attn_layer(layer, **args)


@pytest.mark.parametrize("layer", [2, -3, 1 << 40])
def test_a_layer_outside_the_stack_is_an_index_error(layer):
    with pytest.raises(IndexError):
        _layer_call(layer)


@pytest.mark.parametrize("layer", [0, 1, -1])
def test_a_rejected_call_names_the_entry_point_and_its_status(layer):
    with pytest.raises(jet.JetError) as e:           # max_seq_len = -1: refused by the library's own checks, nothing is launched
        _layer_call(layer)
    assert e.value.status == jet.JET_ERR_INVALID_ARG and "jet_tree_verify_attn_ex" in str(e.value)


def test_conversion_errors():
    with pytest.raises(TypeError):
        _layer_call(0, batch="one")
    with pytest.raises(OverflowError):
        _layer_call(0, B=1 << 40)
    with pytest.raises(TypeError):                   # an address alone does not say how large the workspace is
        _layer_call(0, workspace=4096)
    with pytest.raises(TypeError):
        binding.native().kv_compact(1, 2, 3)
