"""The bounds-checked debug build on the kernels that tall tiles leave out (needs a GPU).

FP64 runs the warp strips in bands of one or two rows only; planes run the shared window where its
tiles fit in one wave of CTAs and the strips don't; FP16-block batches have a body for tiles just
over one wave.  Each runs in a child process that loads the checked library: no access outside its
buffer, and the states of the normal build."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = r'''
import hashlib, json, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import workloads as W
from paper_0911_0459_gb300 import Batch, Lattice
out = {}

def digest(a):
    return hashlib.sha256(np.ascontiguousarray(a).tobytes()).hexdigest()[:16]

def lattice(name, cap, storage, tiles):
    lat = Lattice.from_workload(cap, storage=storage)
    lat.step(70)                 # the default tile, a replayed graph
    lat.set_kernel(1)
    for tx, ty in tiles:
        lat.set_tile(tx, min(ty, cap.ny))
        lat.step(5)
    d = lat.filled_length()
    out[name] = {"check": lat.check_report(), "state": digest(lat.save_state()[0]), "l": d["l"]}
    lat.close()

bp = W.binary_params(nu_l=0.5, nu_g=0.05)
caps = {"c8": W.Capillary("c8", 200, 37, 64, 120, 5, 27, 12, 8, bp, theta_deg=50.0),
        "cw": W.Capillary("cw", 144, 30, 104, 90, 27, 20, 0, 0, bp, wall_grad=-0.1),     # tube through x = 0
        "cr": W.Capillary("cr", 203, 37, 61, 120, 5, 27, 12, 8, bp, wall_grad=-0.11),    # ragged nx
        "nw": W.Capillary("nw", 20, 12, 6, 10, 2, 7, 2, 3, bp, wall_grad=-0.2),
        "ct": W.Capillary("ct", 513, 9, 100, 300, 1, 6, 20, 10, bp, wall_grad=-0.1)}
strips = ((64, 1), (64, 2), (128, 1), (128, 2), (256, 1), (256, 2))
for nm, c in caps.items():
    lattice(f"f64_{nm}", c, 0, strips)
lg = W.config_lg_256x32()
for st in (0, 1):
    lattice(f"lg{st}", lg, st, strips)
wide = W.Capillary("w", 2304, 128, 1000, 1304, 1, 125, 8, 3, bp, wall_grad=-0.1)
for st in (0, 1, 2):             # one wave of the shared window's tiles, two of the strips
    lattice(f"window{st}", wide, st, ((64, 4), (128, 4), (256, 4)))
for nx in (1280, 1276):
    b = Batch([W.Capillary("b", nx, 24, 160, nx - 160, 1, 22, 32, 10, bp, theta_deg=45.0)] * 17, storage=7)
    b.set_tile(128, 8)           # 510 tiles on 456 CTAs
    for v in (2, 3):
        b.set_kernel(v)
        b.step(7)
    out[f"batch{nx}"] = {"check": b.check_report(), "state": digest(b.save_state()[0])}
    b.close()
print(json.dumps(out))
'''


def run(lib=None):
    env = dict(os.environ)
    env.pop("LB_GB300_LIBRARY", None)
    if lib:
        env["LB_GB300_LIBRARY"] = lib
    r = subprocess.run([sys.executable, "-c", RUN, ROOT], capture_output=True, text=True, env=env,
                       timeout=900, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_strips_windows_and_the_second_batch_body_stay_inside_their_buffers():
    from paper_0911_0459_gb300 import build
    checked = run(build.build(variant="check"))
    plain = run()
    assert len(checked) == 12
    for name, rec in checked.items():
        enabled, bad, first = rec["check"]
        assert enabled == 1, name
        assert bad == 0, (name, bad, first - 1)
        assert plain[name]["check"][0] == 0, name
        assert rec["state"] == plain[name]["state"], name
