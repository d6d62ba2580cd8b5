"""Runs a function of a test module in a process of its own with refuse_launch.cpp ahead of the library."""
import os
import subprocess
import sys

from paper_2408_00930_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def child(what, tmp_path, *args, module):
    """module.what(rt, *args), rt the stand-in library (refuse_launch, launches_seen); raises if it does."""
    lib = str(tmp_path / "refuse.so")
    inc = os.path.join(os.path.dirname(build.nvcc()), "..", "include")
    subprocess.run(["g++", "-shared", "-fPIC", "-I", inc, os.path.join(HERE, "refuse_launch.cpp"), "-o", lib, "-ldl"],
                   check=True)
    code = ("import ctypes, importlib, sys; rt = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)\n"
            "sys.path.insert(0, sys.argv[2])\n"
            "from tests.gpu_common import need_gpu; need_gpu()\n"
            "getattr(importlib.import_module('tests.' + sys.argv[3]), sys.argv[4])(rt, *eval(sys.argv[5]))\n")
    subprocess.run([sys.executable, "-c", code, lib, os.path.dirname(HERE), module, what, repr(args)], check=True,
                   timeout=600)
