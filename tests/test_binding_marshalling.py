"""Argument marshalling of the binding's extension module: what it must reject before any call is made (no GPU needed)."""
import os
import subprocess
import sys

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


# Tensors that have no address raise what their own data_ptr() raises; the process goes on.  (One child process each: an
# exception that escapes the extension ends it.)
CHILD = """
import sys
import torch
import paper_2606_18394_b200 as jet
from paper_2606_18394_b200 import binding

def wrapped():
    kept = []
    torch.vmap(lambda x: (kept.append(x), x)[1])(torch.zeros(3, 4))
    return kept[0]

t = {"sparse": lambda: torch.zeros(4, 4, 4).to_sparse(), "csr": lambda: torch.eye(4).to_sparse_csr(),
     "nested": lambda: torch.nested.nested_tensor([torch.zeros(2), torch.zeros(3)]), "vmap": wrapped}[sys.argv[1]]()
z = torch.zeros(4, 4, 4)
calls = [lambda: jet.jet_kv_compact(t, z, z, z, 0, 0, None, 0, 0, z, z, z, 1, 1, 1, 1, 1, 1, stream=0),
         lambda: jet.jet_tree_build(t, z, 1, 4, 4, 2, 4, z, z, z, z, z, z, z, stream=0),
         lambda: jet.jet_tree_build(z, z, 1, 4, 4, 2, 4, z, z, z, z, z, z, t, stream=0),
         lambda: binding.verify_attn_layer(0, t, z, z, None, 0, 0, 0, z, 0, z, z, z, z, 1, 1, 1, 1, 64, 0, 1.0, z, None, None, z,
                                           0, False, stream=0)]
for call in calls:
    try:
        call()
    except Exception as e:
        print("raised", type(e).__name__)
"""


@pytest.mark.parametrize("kind", ["sparse", "csr", "nested", "vmap"])
def test_a_tensor_without_an_address_raises(kind):
    r = subprocess.run([sys.executable, "-c", CHILD, kind], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.count("raised") == 4, r.stdout + r.stderr[-2000:]


def test_a_tensor_subclass_is_asked_through_its_own_methods():
    class Elsewhere(torch.Tensor):
        def data_ptr(self):
            raise LookupError("no address here")

    with pytest.raises(LookupError):
        _layer_call(0, seq_len=torch.zeros(4, dtype=torch.int32).as_subclass(Elsewhere))
    with pytest.raises(LookupError):
        _layer_call(0, q=torch.zeros((2, 1, 4, 2, 64), dtype=torch.bfloat16).as_subclass(Elsewhere))
    with pytest.raises(IndexError):
        _layer_call(2, q=torch.zeros((2, 1, 4, 2, 64), dtype=torch.bfloat16).as_subclass(Elsewhere))
