"""GPU: kernels that other tests' grids no longer reach, against the FP64 oracle element by element: the warp
pass C (k_field_w: one sublattice, one region, Px = 2048, more than two row pairs an SM) at its edges, and the
general passes on an explicit shape, where only the shape itself may be refused."""
import numpy as np
import pytest

from gpu_util import field_tolerance, gpu_eval, make_magnet, oracle_eval, torque_tolerance
from inputs import config_small
from test_gpu_general_passes import LENGTHS, ROWS

pytestmark = pytest.mark.gpu

FM = ("DEMAG", "EXCH", "ANIS", "DMI", "ZEEMAN")


def agree(mag, p, m0, u=None):
    Bg, Tg = gpu_eval(mag, p)
    Bo, To = oracle_eval(p, m0, u)
    tolB = field_tolerance(p, Bo[0])
    assert np.all(np.abs(Bg[0] - Bo[0]) <= tolB), np.abs(Bg[0] - Bo[0]).max()
    assert np.all(np.abs(Tg[0] - To[0]) <= torque_tolerance(p, Bo[0], tolB)), np.abs(Tg[0] - To[0]).max()
    mag.close()


# more than 304 row pairs: odd ny (a last pair of one row), nx not a multiple of 4 (cell by cell), nx = 1024 with
# an open boundary over three layers, cubic anisotropy, the magnetoelastic field
FIELD_W = [((1000, 613, 1), FM, False), ((999, 612, 1), FM, False), ((1024, 206, 3), FM, True),
           ((772, 615, 1), ("DEMAG", "EXCH", "CUBIC", "ZEEMAN"), False),
           ((1024, 310, 2), ("DEMAG", "EXCH", "ANIS", "DMI", "MEL", "ELASTIC"), False)]


@pytest.mark.parametrize("shape,terms,open_bc", FIELD_W)
def test_warp_pass_c(shape, terms, open_bc):
    w = config_small(shape, (2e-9, 2.5e-9, 1.5e-9), 1000 + shape[1], terms=terms)
    p = w.problem
    p.open_bc = open_bc
    u = None
    if "ELASTIC" in terms:
        u = (np.random.default_rng(shape[1]).normal(size=(3,) + shape[::-1]) * 2e-12).astype(np.float32)
    mag = make_magnet(p, w.m0, u, None if u is None else np.zeros_like(u))
    assert mag.get_shape()["engine"] & 2 and (shape[1] + 1) // 2 * shape[2] > 304
    agree(mag, p, w.m0, u)


@pytest.mark.parametrize("shape", [(5 if ny > 128 else 21, ny, nz) for ny, nz in LENGTHS] + ROWS)
def test_general_passes_of_an_explicit_shape(shape):
    from paper_2411_18194_gb300 import MmpError
    w = config_small(shape, (2e-9, 2.5e-9, 1.5e-9), sum(shape), terms=FM)
    mag = make_magnet(w.problem, w.m0)
    try:
        mag.set_shape(R=1, stage_kernel=0, engine=0)
    except MmpError as e:
        assert e.status == -1     # refused (MMP_E_INVAL); the creation default runs
    agree(mag, w.problem, w.m0)
