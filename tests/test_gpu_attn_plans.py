"""Launch plans of small ragged batches: the host knows the longest sequence only, so the plan must not count on all of them
being that long and leave a third of the SMs without a key slice (the library's plan query; nothing is launched)."""
import pytest
import torch

import paper_2606_18394_b200 as jet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,B,Hq,Hkv,D,L", [(3, 15, 32, 8, 128, 19896), (4, 10, 32, 4, 128, 16371), (2, 22, 32, 8, 128, 23941),
                                                (4, 16, 32, 8, 128, 9774)])
def test_slices_cover_the_sms(batch, B, Hq, Hkv, D, L):
    p = jet.jet_tree_verify_attn_plan(batch, B, Hq, Hkv, D, L)
    ctas = batch * Hkv * p["tile_groups"] * p["key_slices"]
    assert 0.85 * torch.cuda.get_device_properties(0).multi_processor_count <= ctas, p
