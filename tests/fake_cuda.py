"""Runs a script against the library with fake_cudart.cpp in place of the CUDA runtime (no GPU)."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = r'''
import ctypes as C, json, os, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import workloads as W
from paper_0911_0459_gb300 import lb, mlp
fake = C.CDLL(os.environ["LD_PRELOAD"])
fake.fake_take_log.restype = C.c_char_p
fake.fake_cost.argtypes = [C.c_char_p, C.c_uint, C.c_uint, C.c_float]

def log():
    return [l.split(" ", 5) for l in fake.fake_take_log().decode().splitlines()]

def launches(part):
    """(grid, block, name) of the launches of kernels whose name holds part."""
    return [(int(l[2]), int(l[3]), l[5]) for l in log() if l[0] == "launch" and part in l[5]]

def ptr(a):
    return a.ctypes.data_as(C.c_void_p)

def lattice(nx, ny, model, storage, **kw):
    p = W.lg_params(storage=storage) if model == W.LG else W.binary_params(nu_l=0.5, nu_g=0.05, storage=storage)
    g, w, q = lb._structs_for(W.Capillary("t", nx, ny, nx // 2, nx - nx // 2, 1, ny - 3, 8, 3, p, wall_grad=-0.1))
    h = C.c_void_p()
    assert L.lb_create(C.byref(g), C.byref(w), C.byref(q), None, None, C.byref(h)) == 0, L.lb_last_error(None)
    return h

def tile(h):
    a, b = C.c_int(), C.c_int()
    assert L.lb_get_tile(h, C.byref(a), C.byref(b)) == 0
    return a.value, b.value

def kernel(h):
    v = C.c_int()
    assert L.lb_get_kernel(h, C.byref(v)) == 0
    return v.value

def network(nin, nh, nout, members, batch):
    h = C.c_void_p()
    assert M.lb_mlp_create(nin, nh, nout, members, batch, 1, None, None, C.byref(h)) == 0, M.lb_mlp_last_error(None)
    return h

L, M = lb.library(), mlp._lib()
'''


def run(tmp, script):
    """The JSON value that script prints last.  tmp: a folder for the stand-in."""
    from paper_0911_0459_gb300 import build
    build.build()
    lib = os.path.join(str(tmp), "fake_cudart.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", cuda, "-o", lib,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp")], check=True)
    env = dict(os.environ, LD_PRELOAD=lib)
    env.pop("LB_GB300_LIBRARY", None)
    r = subprocess.run([sys.executable, "-c", PRELUDE + script, ROOT], capture_output=True, text=True, env=env,
                       timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])
