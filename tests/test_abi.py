"""The C-ABI library builds, loads and exports every symbol the header declares (no GPU needed)."""
import ctypes
import os
import re

import paper_2606_18394_b200 as jet
from paper_2606_18394_b200 import build as jet_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    names = []
    for fn in sorted(os.listdir(os.path.join(ROOT, "include"))):
        text = open(os.path.join(ROOT, "include", fn)).read()
        names += re.findall(r"JET_API\s+[\w\s\*]+?\b(jet_\w+)\s*\(", text)
    return sorted(set(names))


def test_library_builds_and_exports_every_declared_symbol():
    path = jet_build.build()
    assert os.path.exists(path)
    lib = ctypes.CDLL(path)
    declared = _declared()
    assert len(declared) >= 8
    for name in declared:
        assert hasattr(lib, name), name
    assert set(declared) == set(jet.exported_symbols())


def test_status_strings_and_workspace_queries():
    assert jet.status_string(0) == "JET_OK"
    assert jet.status_string(-5) == "JET_ERR_TIMEOUT"
    assert jet.jet_tree_build_workspace_bytes(1, 8, 151936, 7) % 256 == 0
    assert jet.jet_tree_accept_workspace_bytes(32, 64, 151936) >= 32 * 64 * 8
    assert jet.jet_tree_build_workspace_bytes(0, 8, 10, 7) == 0


def test_launch_queries():
    assert [jet.jet_tree_build_launches(N, V) for N, V in ((1, 1), (6, 4096), (6, 4097), (3, 8192), (4, 8192), (1, 24577))] == [1, 1, 2, 1, 2, 2]
    assert [jet.jet_tree_build_launches(2, 100, mode, raw) for mode, raw in ((0, True), (1, False), (2, True))] == [2, 2, 3]
    assert [jet.jet_tree_accept_launches(*a) for a in ((1, 16, 1024), (1, 16, 1025), (1, 17, 64), (1, 4, 2049), (20, 64, 512), (20, 64, 513),
                                                      (19, 64, 512), (20, 512, 64))] == [1, 2, 2, 2, 1, 2, 2, 1]
    assert [jet.jet_kv_compact_launches(*a, tail) for tail in (False, True) for a in
            ((1, 1, 8, 128, 31), (1, 1, 8, 128, 32), (36, 4, 8, 128, 8), (36, 2000, 8, 128, 8))] == [1, 2, 2, 1] + [1, 1, 2, 1]
    assert jet.jet_kv_compact_launches(1, 1, 8, 128, 0) == 0
    assert jet.jet_tree_build_launches(0, 10) == jet.jet_tree_build_launches(1, 10, 3) == jet.jet_tree_accept_launches(1, 0, 10) == 0
