"""The scan module reads torch tensors at the offsets that the headers it was built against give: one built for
another torch or Python is not taken, and is built anew.  No GPU needed."""
import sysconfig

import pytest
import torch

import __graft_entry__ as entry
from paper_2406_17660_b200 import binding, build


@pytest.mark.parametrize("other", ["torch", "python"])
def test_a_scan_built_for_another_torch_or_python_is_neither_taken_nor_kept(monkeypatch, other):
    entry.build()
    binding._accepted()
    assert not build._stale()
    if other == "torch":
        monkeypatch.setattr(torch, "__version__", "1.0.0")
    else:
        real = sysconfig.get_config_var
        monkeypatch.setattr(sysconfig, "get_config_var", lambda name: "cpython-30" if name == "SOABI" else real(name))
    monkeypatch.setattr(binding, "_SCAN", None)
    assert build._stale()
    with pytest.raises(RuntimeError, match="is missing: build it"):
        binding._accepted()


def test_a_scan_that_does_not_load_says_why(monkeypatch, tmp_path):
    broken = tmp_path / "_scan.so"
    broken.write_bytes(b"not a module")
    monkeypatch.setattr(build, "scan_path", lambda: str(broken))
    monkeypatch.setattr(binding, "_SCAN", None)
    with pytest.raises(ImportError, match="_scan.so"):
        binding._accepted()
