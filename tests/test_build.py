"""The C-ABI library is built by nvcc alone; the binding's native calls come after it and belong to one Python and one torch."""
import os
import shutil
import stat
import subprocess
import sys

import pytest

from paper_2510_19705_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE_NVCC = """#!/bin/sh
while [ $# -gt 0 ]; do if [ "$1" = -o ]; then echo built > "$2"; fi; shift; done
"""


def _build(tree, code, **env):
    """Runs `code` in a copy of the sources whose nvcc only writes its output files."""
    shutil.copytree(os.path.join(ROOT, "include"), str(tree / "include"))
    shutil.copytree(build.HERE, str(tree / "paper_2510_19705_b200"), ignore=shutil.ignore_patterns("*.so", "build", "__pycache__"))
    nvcc = tree / "nvcc"
    nvcc.write_text(FAKE_NVCC)
    nvcc.chmod(nvcc.stat().st_mode | stat.S_IXUSR)
    r = subprocess.run([sys.executable, "-c", "import sys; sys.path.insert(0, %r)\n%s" % (str(tree), code)], env=dict(os.environ, NVCC=str(nvcc), **env),
                       capture_output=True, text=True)
    return r, sorted(f for f in os.listdir(str(tree / "paper_2510_19705_b200")) if f.endswith(".so"))


def test_the_library_is_built_without_torch(tmp_path):
    r, built = _build(tmp_path, "sys.modules['torch'] = None\nfrom paper_2510_19705_b200 import build\n"
                                "assert build.build(force=True) == build.LIB and build.build() == build.LIB and not build.needs_build()")
    assert r.returncode == 0, r.stderr
    assert built == ["libhsd.so"]


@pytest.mark.parametrize("compiler", ["false", "/no/such/compiler"])
def test_the_library_is_there_when_the_native_calls_cannot_be_built(tmp_path, compiler):
    r, built = _build(tmp_path, "from paper_2510_19705_b200 import build\nbuild.build()", CXX=compiler)
    assert r.returncode != 0 and built == ["libhsd.so"]


def test_native_calls_of_another_torch_are_not_taken(monkeypatch):
    import torch
    build.build()
    here = build.host_path()
    assert os.path.exists(here) and not build.needs_build()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert build.host_path() != here and build.needs_build()
