"""The library's host code on the CPU: a child process with fake_cudart.c preloaded in place of libcudart, so that
a test can make chosen CUDA calls fail and see what the C entry points do."""
import json
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

_PRELUDE = """
import ctypes, json, sys
sys.path.insert(0, {root!r})
import numpy as np
from paper_0710_5470_gb300 import lb
from tests.helpers import A_VDW, B_VDW
fake = ctypes.CDLL({so!r})
fake.fake_used.restype = ctypes.c_longlong
fake.fake_capacity.argtypes = [ctypes.c_longlong]
def status(f, *a, **k):
    try:
        f(*a, **k)
        return 0
    except lb.LBError as e:
        return e.status
"""


def run(code, tmp_path, env=None):
    """Runs `code` (which ends with print(json.dumps(result))) in the child; returns the result."""
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler")
    from tests.helpers import library
    library()
    so = str(tmp_path / "fake_cudart.so")
    subprocess.run([cc, "-O1", "-shared", "-fPIC", "-o", so, os.path.join(HERE, "fake_cudart.c")], check=True)
    root = os.path.dirname(HERE)
    r = subprocess.run([sys.executable, "-c", _PRELUDE.format(root=root, so=so) + code], cwd=root,
                       env=dict(os.environ, LD_PRELOAD=so, **(env or {})), capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
    return json.loads(r.stdout.strip().splitlines()[-1])
