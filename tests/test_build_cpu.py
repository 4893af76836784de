"""The C library builds with nvcc alone: neither torch nor a host compiler for the Python binding is asked for."""
import os
import shutil
import stat
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_builds_without_torch(tmp_path):
    pkg = tmp_path / "pkg"
    os.makedirs(pkg)
    shutil.copy(os.path.join(ROOT, "paper_2501_16385_b200", "build.py"), pkg)
    shutil.copytree(os.path.join(ROOT, "paper_2501_16385_b200", "csrc"), pkg / "csrc")
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    nvcc = tmp_path / "nvcc"                       # stands in for the compiler: writes what -o names
    nvcc.write_text('#!/bin/sh\nwhile [ $# -gt 0 ]; do if [ "$1" = -o ]; then echo object > "$2"; fi; shift; done\n')
    nvcc.chmod(nvcc.stat().st_mode | stat.S_IXUSR)
    code = ("import sys; sys.modules['torch'] = None; sys.path.insert(0, %r); import build; "
            "print(build.build()); print(build.build())" % str(pkg))
    env = {"NVCC": str(nvcc), "PATH": "/bin:/usr/bin"}
    res = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stderr
    assert (pkg / "libfbq.so").exists() and not (pkg / "_fbq_torch.so").exists()
