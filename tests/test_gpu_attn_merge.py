"""GPU parity of the attention's slice merge in a second launch, at the edges of its forms: the slice counts its code is
written out for, one wave of small CTAs (up to 9 query tiles) or large ones, both head sizes, ragged rows."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import sys
sys.path.insert(0, "tests")
from test_gpu_tree_attn import _run_contiguous
import paper_2606_18394_b200 as jet
ns = int(sys.argv[1])
for B, Hq, Hkv, D, L, n in ((5, 8, 1, 64, 128 * ns, 5), (16, 8, 1, 128, 128 * ns - 60, 13), (16, 9, 9, 64, 128 * ns + 1, 16),
                            (16, 20, 10, 128, 128 * ns, 11), (61, 32, 8, 128, 128 * ns, 61)):
    tiles = Hkv * (-(-B * (Hq // Hkv) // 128))
    if tiles * ns > 148:
        continue
    p = jet.jet_tree_verify_attn_plan(1, B, Hq, Hkv, D, L + 40)
    assert p["merge"] == "second launch" and p["key_slices"] == ns, p
    _run_contiguous(B, Hq, Hkv, D, L, 70 + ns, n=n)
"""


@pytest.mark.parametrize("ns", [2, 4, 5, 8, 9, 10, 11, 12, 13, 20])
def test_second_launch_merge(ns):
    env = dict(os.environ, JET_FORCE_MT="1", JET_FORCE_SPLIT=f"{ns},h")
    r = subprocess.run([sys.executable, "-c", CHILD, str(ns)], env=env, capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]


@pytest.mark.parametrize("ns", ["2", "3", "5", "8"])
def test_fp32_rows_through_a_cluster(ns):
    """Two query tiles per CTA: every number of rounds that the exchange of the fp32 rows takes, ragged paged batches and
    rows without a key in some slice (the random shapes of test_gpu_attn_random_shapes, in a child process: the
    library reads the forced plan once)."""
    env = dict(os.environ, JET_FORCE_MT="2", JET_FORCE_SPLIT=ns)
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(here, "test_gpu_attn_random_shapes.py"), "-m", "gpu", "-x", "-q", "-k",
                        "random_configurations and 1"], env=env, capture_output=True, text=True, cwd=os.path.dirname(here), timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
