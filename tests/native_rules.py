"""The library's plain C++ rules (csrc/tds_rules.cuh) compiled for the host, so
that they can be tested without a GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def compile_rules(tmp_path, exports: str):
    """A ctypes library of extern "C" functions over the rules."""
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    src, lib = tmp_path / "rules.cpp", tmp_path / "rules.so"
    src.write_text('#include "tds_rules.cuh"\n' + exports)
    subprocess.run([gxx, "-std=c++17", "-O2", "-Wall", "-Werror", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2011_00459_gb300", "csrc"), "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(str(lib))
