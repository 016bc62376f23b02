"""When the binding's host calls (csrc/host_calls.cpp) are compiled again, and against which declarations."""
import os
import re
import subprocess
import sys

import pytest
import torch

from paper_2502_20586_b200 import build


@pytest.fixture
def compiled(monkeypatch, tmp_path):
    """A copy of the built file that is newer than its sources, and the list of the compilers that build_host starts."""
    host = tmp_path / os.path.basename(build.HOST)
    host.write_bytes(open(build.HOST, "rb").read())
    for name in ("HOST_SOURCE", "HEADER"):
        copy = tmp_path / name
        copy.write_bytes(open(getattr(build, name), "rb").read())
        os.utime(copy, (1000, 1000))
        monkeypatch.setattr(build, name, str(copy))
    monkeypatch.setattr(build, "HOST", str(host))
    monkeypatch.setattr(build, "HOST_UNTAGGED", str(tmp_path / "_host_calls.so"))
    started = []

    def run(command, check):
        started.append(command)
        open(command[command.index("-o") + 1], "wb").close()
    monkeypatch.setattr(build.subprocess, "run", run)
    return started


@pytest.mark.parametrize("newer", [None, "HOST_SOURCE", "HEADER"])
def test_built_again_when_what_it_is_made_of_is_newer(compiled, newer):
    if newer is not None:
        os.utime(getattr(build, newer), (4e9, 4e9))
    build.build_host()
    assert len(compiled) == (newer is not None)


@pytest.mark.parametrize("what", ["torch", "python"])
def test_built_again_for_another_torch_or_python(compiled, monkeypatch, what):
    if what == "torch":
        monkeypatch.setattr(torch, "__version__", "99.0")
    else:
        monkeypatch.setattr(build.sys.implementation, "cache_tag", "cpython-99")
    open(build.HOST_UNTAGGED, "wb").close()
    build.build_host()
    assert len(compiled) == 1 and not os.path.exists(build.HOST_UNTAGGED)


@pytest.mark.parametrize("version,said", [("torch.__version__", None), ("'99.0'", "torch 99.0")])
def test_the_import_refuses_a_build_for_another_torch(version, said):
    code = f"import torch; torch.__version__ = {version}\nfrom paper_2502_20586_b200 import binding"
    done = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=os.path.dirname(build.INCLUDE))
    assert (done.returncode != 0) == (said is not None)
    assert said is None or ("ImportError" in done.stderr and said in done.stderr and "paper_2502_20586_b200.build" in done.stderr)


def test_a_changed_prototype_does_not_compile(tmp_path):
    header = open(build.HEADER).read()
    changed, n = re.subn(r"(mxfp4_linear_backward_ex\([^;]*?), int accumulate,", r"\1,", header)
    assert n == 1
    (tmp_path / "mxfp4.h").write_text(changed)
    done = subprocess.run([*build.host_command(os.devnull, str(tmp_path)), "-fsyntax-only"], capture_output=True, text=True)
    assert done.returncode != 0 and "too many arguments" in done.stderr


def test_links_no_cuda_library_of_torchs():
    """A torch that was built without CUDA imports the binding too (its calls then refuse every tensor)."""
    libraries = [flag for flag in build.host_command("out") if flag.startswith("-l")]
    assert "-lc10" in libraries and not any("cuda" in flag for flag in libraries)
