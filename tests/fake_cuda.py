"""Runs the library on the stand-in CUDA runtime of fake_cudart.c, to see on the CPU which kernels a call launches, in
which launch shape and with which device current.

run_fake(body) runs the statements of `body` in a new process, where `ccmf` is the binding module, `np` is numpy,
`launches()` returns and clears the log as (device, kernel, grid x, block x), `buf(n)` is n zeroed bytes on a 256-byte
boundary and `set_device(d)` makes a device current. What the statements put in the dict `out` is returned."""

import json
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

needs_toolchain = pytest.mark.skipif(
    shutil.which("gcc") is None or (shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc")),
    reason="needs gcc and nvcc")

_HEAD = """
import ctypes, json, sys
fake = ctypes.CDLL({so!r}, mode=ctypes.RTLD_GLOBAL)
fake.fake_log.restype = ctypes.c_char_p
import numpy as np
from paper_2103_05968_gb300 import ccmf
lib = ccmf.load_library()
out, _keep = {{}}, []

def launches():
    rows = [r.split() for r in fake.fake_log().decode().splitlines()]
    fake.fake_clear()
    return [(int(d), k, int(g), int(b)) for d, k, g, b in rows]

def buf(n, offset=0):
    a = np.zeros(int(n) + 512, dtype=np.uint8)
    _keep.append(a)
    return ctypes.c_void_p((a.ctypes.data + 255) // 256 * 256 + offset)

def set_device(d):
    fake.fake_set_device(int(d))
"""


def run_fake(body, tmp_path, env=None):
    so = os.path.join(str(tmp_path), "libfakecudart.so")
    versions = os.path.join(str(tmp_path), "versions")
    with open(versions, "w") as f:
        f.write("libcudart.so.13 { global: *; };\n")
    subprocess.run(["gcc", "-O1", "-w", "-shared", "-fPIC", "-Wl,-soname,libcudart.so.13",
                    f"-Wl,--version-script={versions}", os.path.join(HERE, "fake_cudart.c"), "-o", so], check=True)
    code = _HEAD.format(so=so) + body + "\nprint('OUT ' + json.dumps(out))\n"
    e = {k: v for k, v in os.environ.items() if not k.startswith("CCMF_")}
    e.update(env or {}, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=e, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return json.loads([x for x in r.stdout.splitlines() if x.startswith("OUT ")][-1][4:])
