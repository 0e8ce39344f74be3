"""The binding's extension is rebuilt, and refused at load time, when it was built for another torch (no GPU needed)."""
import json

import pytest
import torch

from paper_2606_18394_b200 import binding
from paper_2606_18394_b200 import build as jet_build


def test_a_build_for_another_torch_is_stale(tmp_path, monkeypatch):
    jet_build.build()
    assert not jet_build.needs_build()
    stamp = json.load(open(jet_build.STAMP))
    assert stamp["torch"] == torch.__version__
    other = tmp_path / "stamp.json"
    monkeypatch.setattr(jet_build, "STAMP", str(other))
    assert jet_build.needs_build()                   # no stamp: nothing is known about the files that are there
    other.write_text(json.dumps(dict(stamp, torch="1.0.0")))
    assert jet_build.needs_build()
    other.write_text("not json")
    assert jet_build.needs_build()
    other.write_text(json.dumps(stamp))
    assert not jet_build.needs_build()


def test_an_extension_for_another_torch_is_refused(monkeypatch):
    ext = binding.native()
    assert ext.torch_version == torch.__version__
    monkeypatch.setattr(binding, "_ext", None)
    monkeypatch.setattr(torch, "__version__", "1.0.0")
    with pytest.raises(RuntimeError, match="built for torch"):
        binding.native()
