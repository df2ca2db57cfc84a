"""The resident step of the checked debugging build (LBM_CHECKED) records no offset
outside the population arrays: single steps and many per launch, periodic and
walled and sliding-walled grids, with and without the ghost band, down to extents
of one node.  Against the default build: FP64 to 1e-12, FP32 to 1e-6."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
import numpy as np
sys.path.insert(0, ROOT)
from paper_1812_00118_gb300 import lbm as L, inputs as I
lib = L.load()
P, W = L.PERIODIC, L.WALL
out = {"checked_build": int(lib.lbm_is_checked_build()), "runs": []}
CASES = [((40, 70), (P, P)), ((33, 9), (W, W)), ((1, 40), (P, W)), ((300, 200), (W, P)), ((13, 21, 37), (P, P, P)),
         ((19, 11, 35), (W, P, W)), ((4, 64, 4), (P, W, P)), ((1, 1, 30), (P, P, P)), ((40, 38, 36), (W, W, W))]
for shape, bc in CASES:
    d = len(shape)
    nx, ny = shape[:2]
    nz = shape[2] if d == 3 else 1
    phi, u, Pr = I.smooth_random((nz, ny, nx), 5, dim=d, u_amp=0.01, P_amp=1e-4)
    for store in (L.F64, L.F32):
        for band in (False, True):
            prm = L.make_params(M=0.1, W=3.0, sigma=0.001, rho_L=0.5, rho_H=1.0, nu_L=0.05, nu_H=0.05, store=store)
            s = L.Simulation(L.D2Q9 if d == 2 else L.D3Q19, shape, prm, bc=bc, ghost_band=band)
            for a in range(d):
                if bc[a] == W:
                    v = [0.01, -0.02, 0.005][:d]
                    v[a] = 0.0
                    s.set_wall_velocity(a, 0, v)
            s.init_fields(*[np.ascontiguousarray(q.reshape(-1)) for q in (phi, u[:d], Pr)])
            n0 = s.launch_count()
            s.step(1)
            s.step(6)
            assert s.launch_count() - n0 == 2      # the resident form
            h, g = s.get_populations()
            s.close()
            out["runs"].append([h[::max(1, h.size // 50)].tolist(), g[::max(1, g.size // 50)].tolist(),
                                1e-12 if store == L.F64 else 1e-6])
out["status"] = int(lib.lbm_checked_status(None))
print("RESULT" + json.dumps(out))
"""


def run_child(checked):
    r = subprocess.run([sys.executable, "-c", CHILD.replace("ROOT", repr(ROOT))],
                       env=dict(os.environ, LBM_CHECKED=checked), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads([l for l in r.stdout.splitlines() if l.startswith("RESULT")][-1][len("RESULT"):])


def test_checked_resident_step():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00118_gb300 import build
    build.build()
    build.build(checked=True)
    plain, checked = run_child("0"), run_child("1")
    assert plain["checked_build"] == 0 and checked["checked_build"] == 1
    assert plain["status"] == 0 and checked["status"] == 0
    for a, b in zip(plain["runs"], checked["runs"]):
        for x, y in zip(a[:2], b[:2]):
            assert np.allclose(x, y, rtol=a[2], atol=a[2] * np.abs(x).max())
