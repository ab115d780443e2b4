"""The padding of an instance is a whole number of the face-value kernels' items (64 or 256 cells) however
the library is compiled: items would else straddle instances and leave cells out."""
import subprocess

import pytest

from paper_1812_00394_gb300 import build


@pytest.mark.parametrize("option", [[], ["-DFVLBM_FUSED_BLOCK=128"], ["-DFVLBM_FUSED_BLOCK=384"]],
                         ids=["default", "128", "384"])
def test_instances_are_whole_items(option, tmp_path):
    src = tmp_path / "padding.cpp"
    src.write_text('#include "fvlbm_internal.h"\n'
                   "static_assert(fvlbm::kBlock % 256 == 0 && fvlbm::kBlock % 64 == 0, \"\");\n")
    r = subprocess.run(["g++", "-std=c++17", "-fsyntax-only", *option, "-I", build.INCLUDE, "-I", build.CSRC,
                        str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def test_no_build_option_changes_the_padding(monkeypatch, tmp_path):
    """The environment does not reach the compiler's options."""
    seen = []

    class Done(Exception):
        pass

    def popen(cmd, **kw):
        seen.append(cmd)
        raise Done

    monkeypatch.setenv("FVLBM_FUSED_BLOCK", "128")
    monkeypatch.setattr(build, "BUILD", str(tmp_path))
    monkeypatch.setattr(build, "_nvcc", lambda: "nvcc")
    monkeypatch.setattr(subprocess, "Popen", popen)
    with pytest.raises(Done):
        build.build(force=True)
    assert not [x for cmd in seen for x in cmd if x.startswith("-D")]
