"""_s2a_torch.so belongs to the torch it was built with: another version is built for again, and refused if it is loaded."""
import os

import pytest
import torch

from paper_2309_12307_b200 import binding, build

needs_library = pytest.mark.skipif(not os.path.exists(build.TORCH_LIB), reason="not built")


@needs_library
def test_another_torch_means_another_build(monkeypatch, tmp_path):
    lib = tmp_path / "_s2a_torch.so"
    monkeypatch.setattr(build, "TORCH_LIB", str(lib))
    commands = []
    monkeypatch.setattr(build.subprocess, "run", lambda cmd, **kw: (commands.append(cmd), lib.write_bytes(b"")))
    build.build_torch()
    build.build_torch()
    assert len(commands) == 1  # up to date
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    build.build_torch()
    assert len(commands) == 2 and any('="0.0.0"' in a for a in commands[1])
    build.build_torch(force=True)
    assert len(commands) == 3


@needs_library
def test_a_module_of_another_torch_is_refused(monkeypatch):
    monkeypatch.setattr(binding, "_hot", None)
    assert binding.load_hot().torch_version == torch.__version__
    monkeypatch.setattr(binding, "_hot", None)
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    with pytest.raises(ImportError, match="built for torch"):
        binding.load_hot()
