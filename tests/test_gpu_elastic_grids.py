"""GPU: the elastic kernels where their cells fill no block or have few rows in the 4th-order bulk: narrow
rows, extents of 1 to 9 along any axis, rows just above a block; with and without the demag term.  Three fixed
steps from a random displacement against the FP64 oracle.

Tolerance of u and v: sums of 36 products over two stencil levels (strain, then force) of FP32 values, in seven
stage combinations: 2 * 36 * 2^-23 * 2 = 2e-5 of the largest value."""
import numpy as np
import pytest

from gpu_util import make_magnet
from inputs import config_small

pytestmark = pytest.mark.gpu

SHAPES = [(8, 40, 1), (17, 9, 2), (129, 6, 1), (5, 4, 3), (3, 3, 3), (2, 5, 1), (1, 20, 2), (260, 1, 1), (9, 130, 1),
          (6, 7, 9), (11, 10, 12)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n_sub,demag,regions", [(2, False, 1), (1, True, 3)])
def test_elastic_steps_match_oracle(shape, n_sub, demag, regions):
    import torch
    from oracle.dp45 import Oracle, State
    terms = {"EXCH", "ANIS", "MEL", "ELASTIC"} | ({"AFM"} if n_sub == 2 else set()) | ({"DEMAG"} if demag else set())
    w = config_small(shape, (2e-9, 3e-9, 2.5e-9), 40 + sum(shape), terms=terms, n_sub=n_sub, n_regions=regions)
    w.problem.glob.update(ETA=2e-14)
    nx, ny, nz = shape
    rng = np.random.default_rng(sum(shape))
    u = (rng.normal(size=(3, nz, ny, nx)) * 2e-12).astype(np.float32)
    v = (rng.normal(size=(3, nz, ny, nx)) * 1e-4).astype(np.float32)
    dt = 1e-16
    mag = make_magnet(w.problem, w.m0, u, v)
    mag.set_solver(adaptive=False, dt=dt)
    mag.step(3)
    ug, vg = (torch.empty((3, nz, ny, nx), dtype=torch.float32, device="cuda") for _ in range(2))
    mag.get_elastic(ug, vg)
    st = Oracle(w.problem).run_fixed(State([m.astype(np.float64) for m in w.m0], u, v), dt, 3)
    assert np.abs(st.v - v).max() > 1e-4    # the force moves the cells
    for got, ref in ((ug, st.u), (vg, st.v)):
        assert np.abs(got.cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()
    mag.close()
