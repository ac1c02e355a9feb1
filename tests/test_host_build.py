"""The native calls fit one interpreter and one torch: another build of them is refused, and built again when asked (no GPU needed)."""
import os
import types

import pytest

from paper_2604_26209_b200 import binding, build


def test_extension_is_built_again_for_another_torch(monkeypatch, tmp_path):
    runs = []

    def compiler(cmd, **_):
        runs.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()
        return types.SimpleNamespace(returncode=0, stdout="", stderr="")

    monkeypatch.setattr(build, "HOST", str(tmp_path / "_host.so"))
    monkeypatch.setattr(build, "OBJ", str(tmp_path))
    monkeypatch.setattr(build.subprocess, "run", compiler)
    build._build_host()
    build._build_host()                                  # up to date: newer than the sources, same torch
    assert len(runs) == 1
    monkeypatch.setattr(build, "host_key", lambda: "another torch")
    build._build_host()
    build._build_host()
    assert len(runs) == 2
    os.remove(tmp_path / "_host.key")                    # built by nobody knows what
    build._build_host()
    assert len(runs) == 3


def test_extension_of_another_torch_is_refused(monkeypatch):
    build.build()
    binding.load()
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(build, "host_key", lambda: "another torch")
    with pytest.raises(binding.HpdError, match="another torch"):
        binding.load()
    assert binding._lib is None


def test_file_name_carries_the_interpreter():
    import sysconfig
    assert build.HOST.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
