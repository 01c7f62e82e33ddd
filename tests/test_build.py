"""The built tensor side of the binding is tied to the torch and the interpreter that it was compiled against."""
import subprocess

import pytest

import paper_2609_36601_b200 as P
from paper_2609_36601_b200 import binding, build


def test_another_torch_means_another_build(monkeypatch):
    build.build()
    assert build.host_matches() and not build._host_needs_build()
    assert build.host_tag() in next(a for a in build._host_command() if "SAKI_BUILT_FOR" in a)
    monkeypatch.setattr(build, "host_tag", lambda: "saki tensor side for torch 0.0.0, python 3.0;")
    assert not build.host_matches() and build._host_needs_build()
    monkeypatch.setattr(binding, "_lib", None)
    with pytest.raises(P.SakiError, match="another torch"):
        binding.load_library()


def test_the_tensor_side_compiles_without_warnings(tmp_path):
    cmd = [str(tmp_path / "out.so") if a == build.TORCH_LIB else a for a in build._host_command()]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0 and "warning" not in r.stderr, r.stderr[-2000:]
