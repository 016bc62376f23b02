"""When the binding's host calls (csrc/host_calls.cpp) are compiled again, and against which declarations."""
import os
import re
import subprocess

import pytest

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


def test_a_changed_prototype_does_not_compile(tmp_path):
    header = open(build.HEADER).read()
    changed, n = re.subn(r"(mxfp4_linear_backward_ex\([^;]*?), int accumulate,", r"\1,", header)
    assert n == 1
    (tmp_path / "mxfp4.h").write_text(changed)
    done = subprocess.run([*build.host_command(os.devnull, str(tmp_path)), "-fsyntax-only"], capture_output=True, text=True)
    assert done.returncode != 0 and "too many arguments" in done.stderr
