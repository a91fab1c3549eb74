"""The particle buffers a handle allocates cover what the filtered search writes
for a last tile that is not full.  CPU only: the library's host code runs on a
stand-in for the CUDA runtime (host_cudart.cpp) that records the allocations and
looks at the buffers every launch is given."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1210_8084_gb300")

CHILD = r"""
import ctypes, json, math, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import paper_1210_8084_gb300 as k
lib = ctypes.CDLL(sys.argv[2])
lib.host_shortfall.restype = ctypes.c_long
for f in ("kmc_init", "kmc_step"):
    getattr(lib, f).restype = ctypes.c_int
out = {}
for prec in (32, 64):
    dtype = np.float32 if prec == 32 else np.float64
    for n in list(range(0, 42)) + [255, 1001]:
        pos, vel = np.full((n, 3), 0.5, dtype), np.zeros((n, 3), dtype)
        # a contact distance just under half a c-bin: a binary32 batch takes the filtered search
        one = dict(sigma=math.pi * (0.48 / 6) ** 2, lam=1.0, dt=1e-3)
        cfg = k.make_config(dim_pos=2, n_cells=(6, 6, 1), instances=[dict(one, n=n), dict(one, n=0)], precision=prec,
                            flags=k.KMC_FLAG_NO_GRAPH)
        h = ctypes.c_void_p()
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        rc = lib.kmc_init(ctypes.byref(cfg), ctypes.c_int64(n), ptr(pos), ptr(vel), 0, ctypes.byref(h))
        assert rc == 0, (n, rc)
        before = lib.host_launches(b"filter_prep_kernel")
        assert lib.kmc_step(h, 1, 0) == 0
        filtered = lib.host_launches(b"filter_prep_kernel") - before
        lib.kmc_free(h)
        out["%d/%d" % (prec, n)] = (filtered, lib.host_shortfall())
print(json.dumps(out))
"""


@pytest.fixture(scope="module")
def host_lib(tmp_path_factory):
    import __graft_entry__ as g
    g.build()
    from paper_1210_8084_gb300 import build
    home = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    out = str(tmp_path_factory.mktemp("host") / "libkmc_host.so")
    objs = [os.path.join(build.OBJ, s.replace(".cu", ".o")) for s in build.SOURCES]
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", os.path.join(home, "include"), "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "host_cudart.cpp"), *objs, "-o", out], check=True)
    return out


def test_buffers_cover_whole_tiles(host_lib):
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, host_lib], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout)
    assert all(v[0] == 1 for key, v in out.items() if key.startswith("32/") and key != "32/0")
    short = {key: v[1] for key, v in out.items() if v[1] > 0}
    assert not short, short
