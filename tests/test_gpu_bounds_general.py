"""The bounds-checked build on the GPU over the general warp passes and the warp pass C (test_gpu_bounds.py has
the block passes and the clusters): every class count of kx and ky, partly filled blocks, regions with empty
cells, two sublattices with elastodynamics, grids above two row pairs an SM, batch members, and the demag field
without allocations.  Fields and torques against the oracle, adaptive steps without a failed check."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import json, sys
sys.path.insert(0, "tests")
import numpy as np, torch
from inputs import config_small
from gpu_util import field_tolerance, torque_tolerance, make_magnet, gpu_eval, oracle_eval
import paper_2411_18194_gb300 as pkg
assert pkg.library_path().endswith("libmmp_checked.so"), pkg.library_path()
FM = ("DEMAG", "EXCH", "ANIS", "DMI", "ZEEMAN")
AF = ("DEMAG", "EXCH", "ANIS", "AFM", "MEL", "ELASTIC", "ZEEMAN")
CASES = [((33, 27, 3), 1, 0.0, 1, FM), ((49, 65, 5), 1, 0.0, 1, FM), ((130, 33, 1), 3, 0.1, 1, FM),
         ((200, 101, 7), 2, 0.1, 1, FM), ((515, 6, 1), 1, 0.0, 1, FM), ((1030, 5, 1), 1, 0.0, 1, FM),
         ((1030, 6, 1), 3, 0.1, 1, FM), ((6, 700, 2), 1, 0.0, 1, FM), ((64, 64, 1), 1, 0.0, 1, FM),
         ((40, 30, 2), 1, 0.0, 2, AF), ((300, 7, 1), 1, 0.0, 2, AF), ((30, 620, 1), 1, 0.0, 1, FM),
         ((1000, 613, 1), 1, 0.0, 1, FM)]
out = []
for i, (shape, nreg, empty, nsub, terms) in enumerate(CASES):
    w = config_small(shape, (2e-9, 2e-9, 1e-9), 190 + i, terms=terms, n_regions=nreg, empty_fraction=empty, n_sub=nsub)
    p = w.problem
    u = None
    if "ELASTIC" in terms:
        u = (np.random.default_rng(i).normal(size=(3,) + shape[::-1]) * 2e-12).astype(np.float32)
    mag = make_magnet(p, w.m0, u, None if u is None else np.zeros_like(u))
    Bg, Tg = gpu_eval(mag, p)
    Bo, To = oracle_eval(p, w.m0, u)
    ok = True
    for s in range(nsub):
        tolB = field_tolerance(p, Bo[s], s)
        ok = ok and bool(np.all(np.abs(Bg[s] - Bo[s]) <= tolB))
        ok = ok and bool(np.all(np.abs(Tg[s] - To[s]) <= torque_tolerance(p, Bo[s], tolB)))
    mag.set_solver(adaptive=True, dt=1e-16 if nsub == 2 else 1e-14)
    mag.step(6)          # direct attempts, then a graph
    mag.close()
    out.append([list(shape), ok])
mags = []
with pkg.Batch() as b:
    for i, shape in enumerate([(33, 27, 3), (130, 40, 1), (200, 31, 6), (600, 12, 1), (20, 20, 2)]):
        w = config_small(shape, (2e-9, 2e-9, 1e-9), 290 + i, terms=("DEMAG", "EXCH", "ZEEMAN"))
        mag = make_magnet(w.problem, w.m0)
        mag.set_shape(R=1, stage_kernel=0, engine=0)
        mag.set_solver(adaptive=True, dt=1e-14)
        mags.append(mag)
        b.add(mag, "steps", 4)
    b.advance()
    out.append(["batch", all(b.status(m) == (True, 0) for m in mags)])
for mag in mags:
    mag.close()
for shape in [(33, 27, 3), (600, 9, 1)]:
    w = config_small(shape, (2e-9, 2e-9, 1e-9), 390, terms=("DEMAG",))
    w.problem.set("MS", 1.0)
    M = torch.from_numpy(w.m0[0]).cuda()
    B = pkg.demag_noalloc(shape, (2e-9, 2e-9, 1e-9), M, torch.empty_like(M)).cpu().numpy()
    Bo, _ = oracle_eval(w.problem, w.m0)
    out.append(["noalloc %s" % (shape,), bool(np.all(np.abs(B - Bo[0]) <= field_tolerance(w.problem, Bo[0])))])
print(json.dumps(out))
'''


def test_checked_build_over_the_general_passes():
    from paper_2411_18194_gb300 import build
    if not os.path.exists(build.CHECKED_LIB):
        build.build(checked=True)
    env = dict(os.environ, MMP_CHECK_BOUNDS="1")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=1800)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(res) == 16 and all(ok for _, ok in res), res
