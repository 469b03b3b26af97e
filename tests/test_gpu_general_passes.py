"""GPU: the general warp passes (passb_g.cuh) at the sizes where they can go
wrong: every padded y length of the engine at its smallest and largest ny,
every half z length, planes that fill a block only in part, and one or two
ky classes; against the FP64 oracle, element by element, within the field bar."""
import numpy as np
import pytest

from gpu_util import field_tolerance, gpu_eval, make_magnet, oracle_eval, torque_tolerance
from inputs import config_small

pytestmark = pytest.mark.gpu

FM = ("DEMAG", "EXCH", "ANIS", "DMI", "ZEEMAN")


def check(shape, seed, nreg=1, empty=0.0, terms=FM, n_sub=1, **launch_shape):
    w = config_small(shape, (2e-9, 2.5e-9, 1.5e-9), seed, terms=terms, n_regions=nreg, empty_fraction=empty,
                     n_sub=n_sub)
    p = w.problem
    mag = make_magnet(p, w.m0)
    if launch_shape:
        mag.set_shape(**launch_shape)
    Bg, Tg = gpu_eval(mag, p)
    Bo, To = oracle_eval(p, w.m0)
    for s in range(p.n_sub):
        tolB = field_tolerance(p, Bo[s], s)
        assert np.all(np.abs(Bg[s] - Bo[s]) <= tolB), np.abs(Bg[s] - Bo[s]).max()
        assert np.all(np.abs(Tg[s] - To[s]) <= torque_tolerance(p, Bo[s], tolB)), np.abs(Tg[s] - To[s]).max()
    mag.close()


# (ny, nz): padded y lengths 64, 96, 128, 192, 256, 384, 512, 768, 1024 (one class), 1536 and 2048 (two),
# smallest and largest ny of each; nz over every half z length 1, 2, 3, 4, 6 (5 and 6), 8 (7 and 8)
LENGTHS = [(25, 1), (32, 2), (33, 3), (48, 4), (49, 5), (64, 6), (65, 7), (96, 8), (97, 1), (128, 3), (129, 2),
           (192, 4), (193, 5), (256, 7), (257, 1), (384, 6), (385, 3), (512, 4), (513, 1), (768, 2), (769, 3),
           (1024, 1), (700, 4), (400, 8), (60, 1), (120, 1), (380, 1), (511, 2)]


@pytest.mark.parametrize("ny,nz", LENGTHS)
def test_pass_b_lengths(ny, nz):
    # engine 0, R = 1 where the shape fits; the creation default otherwise
    from paper_2411_18194_gb300 import MmpError
    nx = 5 if ny > 128 else 21
    try:
        check((nx, ny, nz), 300 + ny + nz, R=1, stage_kernel=0, engine=0)
    except MmpError:
        check((nx, ny, nz), 300 + ny + nz)


@pytest.mark.parametrize("ny,nz", [(120, 1), (200, 2), (500, 1), (900, 1), (1000, 2)])
def test_pass_b_default_shapes(ny, nz):
    """The creation defaults that run the general pass B under the warp engine."""
    check((6, ny, nz), 400 + ny, nreg=2, empty=0.05)
