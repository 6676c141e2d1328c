"""What the build needs: the C library nvcc alone, the binding's extension module PyTorch and a C++ compiler as well."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BUILD = """
import os, sys
if %(hide)r:
    sys.modules["torch"] = None            # `import torch` raises ImportError
from paper_2604_16855_b200 import build as b
b.OBJ, b.LIB, b.HOST = (os.path.join(%(tmp)r, n) for n in ("obj", "libtdq.so", "_tdq_host.so"))
open(b.HOST, "w").close()
os.utime(b.HOST, (0, 0))                   # of older sources
try:
    print(b.build(), os.path.exists(b.LIB), os.path.exists(b.HOST))
    print(b.build(), os.path.exists(b.LIB), os.path.exists(b.HOST))
except RuntimeError as e:
    print("RuntimeError", e)
"""


def _run(tmp_path, hide, cxx):
    nvcc = tmp_path / "nvcc"                # writes the file its -o names, and a line for the call
    nvcc.write_text('#!/bin/sh\necho call >> %s/calls\nwhile [ "$1" != -o ]; do shift; done\n: > "$2"\n' % tmp_path)
    nvcc.chmod(0o755)
    env = dict(os.environ, NVCC=str(nvcc), CXX=cxx)
    r = subprocess.run([sys.executable, "-c", BUILD % dict(hide=hide, tmp=str(tmp_path))], cwd=ROOT, env=env, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return r, len((tmp_path / "calls").read_text().split())


@pytest.mark.parametrize("hide,cxx", [(True, "g++"), (False, "no-such-compiler")])
def test_library_builds_without_pytorch_or_compiler(tmp_path, hide, cxx):
    r, calls = _run(tmp_path, hide, cxx)
    want = "%s True False" % (tmp_path / "libtdq.so")
    assert r.stdout.split("\n")[:2] == [want, want]         # no extension module, and none of older sources left
    assert "is not built" in r.stderr
    sys.path.insert(0, ROOT)
    from paper_2604_16855_b200 import build as b
    assert calls == len(b.SOURCES) + 1                      # the second build finds the library up to date


def test_a_compiler_that_fails_is_reported(tmp_path):
    r, _ = _run(tmp_path, False, "false")
    assert r.stdout.startswith("RuntimeError")
