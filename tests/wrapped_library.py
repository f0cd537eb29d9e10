"""The library's objects linked once more with some CUDA runtime functions wrapped (the linker's
--wrap), for child processes that see a runtime call fail, or answer otherwise, on purpose."""

import json
import os
import subprocess
import sys

from paper_1401_0427_gb300 import build as libbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import ctypes, json, sys
import numpy as np
from paper_1401_0427_gb300 import inputs, lbm_sw
lib = lbm_sw.load(sys.argv[1])
"""
ON_GPU = """
import torch
torch.zeros(1, device="cuda")
"""


def link(folder, hook: str, wrapped) -> str:
    """Shared library of the library's objects and the hook's source; returns its path."""
    libbuild.build()
    objs = [os.path.join(libbuild.BUILD, os.path.basename(s)[:-3] + ".o") for s in libbuild.sources()]
    src, so = os.path.join(folder, "hook.cu"), os.path.join(folder, "liblbm_sw_wrapped.so")
    with open(src, "w") as f:
        f.write(hook)
    r = subprocess.run([libbuild.nvcc(), *libbuild.ARCH, "-Xcompiler", "-fPIC", "-shared", "-cudart", "static", "-o", so,
                        src, *objs, *[x for w in wrapped for x in ("-Xlinker", f"--wrap={w}")]],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return so


def run(library: str, script: str, on_gpu: bool = True):
    """The JSON value of the last line that the script prints in a child process with the library."""
    r = subprocess.run([sys.executable, "-c", PRELUDE + (ON_GPU if on_gpu else "") + script, library], capture_output=True, text=True, cwd=ROOT,
                       env={**os.environ, "PYTHONPATH": ROOT}, timeout=300)
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.splitlines()[-1])
