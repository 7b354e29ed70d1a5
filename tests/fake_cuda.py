"""The library's host code without a device: its object files linked with
fake_cudart.cpp, a call made in a process of its own (`call.py` text), and the
runtime calls that it made as a list."""
import json
import os
import subprocess
import sys
from pathlib import Path

import pytest

from paper_1905_08394_gb300 import build

ROOT = Path(__file__).resolve().parents[1]

PRELUDE = """
import ctypes, json
import numpy as np
from paper_1905_08394_gb300 import binding as B
from rqc_inputs import make_circuit, make_circuit_general, prefix_group_bitstrings, uniform_bitstrings
lib = B.load()
lib.fake_log.restype = ctypes.c_char_p

def context(circ):
    h, C = B.peps_create(circ.R, circ.C), circ.C
    for g in circ.gates:
        a, b = g.qubits[0], g.qubits[-1]
        if g.kind == "1q":
            B.peps_apply_1q(h, a // C, a % C, g.U)
        elif g.kind == "2q":
            B.peps_apply_2q(h, a // C, a % C, b // C, b % C, g.U)
        else:
            B.peps_apply_cz(h, a // C, a % C, b // C, b % C)
    return h

def call(h, bits, device=0, out=None, align=0, **kw):
    # one host call in host memory; its log, one list of words per line
    o, keep = B.make_opts(**kw)
    need = B.peps_workspace_bytes(h, len(bits), o)
    ws = np.zeros(need + 1024, dtype=np.uint8)
    base = (ws.ctypes.data + 511) // 512 * 512 + align
    out = np.zeros(len(bits), dtype=np.complex128) if out is None else out
    lib.fake_set_device(device)
    lib.fake_clear()
    rc = lib.peps_amplitudes(h, bits.ctypes.data, len(bits), out.ctypes.data, o, base, need, None)
    log = [l.split() for l in lib.fake_log().decode().splitlines()]
    return rc, log, ws, out
"""


@pytest.fixture(scope="session")
def fake_lib(tmp_path_factory):
    """The library with the fake runtime in place of CUDA's."""
    objs = [build.BUILD / (Path(s).stem + ".o") for s in build.SOURCES]
    if not all(o.exists() for o in objs):
        pytest.skip("object files missing: build the library first")
    so = tmp_path_factory.mktemp("fake") / "libpeps_fake.so"
    cuda = Path(build.nvcc()).resolve().parents[1] / "include"
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", str(cuda),
                    str(ROOT / "tests" / "fake_cudart.cpp"), *map(str, objs), "-o", str(so)],
                   check=True, capture_output=True, text=True)
    return so


def run(fake_lib, script):
    """`script`'s own last line of output, as JSON."""
    env = dict(os.environ, PEPS_GB300_LIB=str(fake_lib), PYTHONPATH=str(ROOT))
    r = subprocess.run([sys.executable, "-c", PRELUDE + script], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-4000:]
    return json.loads(r.stdout.splitlines()[-1])
