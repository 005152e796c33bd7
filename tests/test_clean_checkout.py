"""The build entry point on a tree in which nothing has been built yet."""
import os
import shutil
import subprocess
import sys

from tests.conftest import ROOT


def test_build_starts_without_a_built_library(tmp_path):
    """A copy of the sources without any built file: build() has to reach the compiler (a stand-in that writes what it is asked
    for) before anything needs the library."""
    for name in ("__graft_entry__.py", "paper_2411_17525_b200", "include"):
        src = os.path.join(ROOT, name)
        if os.path.isdir(src):
            shutil.copytree(src, tmp_path / name, ignore=shutil.ignore_patterns("*.so", "build", "__pycache__"))
        else:
            shutil.copy(src, tmp_path / name)
    nvcc = tmp_path / "nvcc"
    nvcc.write_text("#!/bin/sh\nwhile [ $# -gt 0 ]; do [ \"$1\" = -o ] && : > \"$2\"; shift; done\n")
    nvcc.chmod(0o755)
    code = ("import __graft_entry__, os\n"
            "try: __graft_entry__.build()\n"
            "except ImportError as e: print('after the compiler:', e)\n"       # (the oracle is not copied)
            "assert os.path.exists('paper_2411_17525_b200/libhiggs_b200.so')\n")
    env = dict(os.environ, NVCC=str(nvcc))
    env.pop("PYTHONPATH", None)
    done = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, env=env, capture_output=True, text=True)
    assert done.returncode == 0, done.stderr
