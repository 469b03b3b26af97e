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


# passes A and C (xfft_g.cuh): padded x lengths 64 .. 1024 (one class of kx), 1536 and 2048 (two), 3072 and
# 4096 (four): smallest and largest nx of each, odd ones and ones of 2 mod 4 among them, ny odd, even and 1
ROWS = [(25, 4, 2), (32, 5, 1), (33, 6, 1), (48, 1, 3), (49, 7, 1), (64, 8, 2), (66, 3, 2), (96, 4, 1), (97, 2, 1),
        (128, 5, 3), (130, 6, 1), (192, 3, 1), (193, 4, 1), (256, 9, 2), (258, 2, 1), (384, 4, 1), (387, 3, 2),
        (512, 6, 1), (514, 5, 1), (768, 4, 2), (771, 2, 1), (1024, 3, 1), (1025, 4, 1), (1536, 2, 1), (1538, 3, 1),
        (2047, 2, 1), (2048, 5, 1)]


@pytest.mark.parametrize("nx,ny,nz", ROWS)
def test_passes_a_and_c_lengths(nx, ny, nz):
    from paper_2411_18194_gb300 import MmpError
    try:   # engine 0: the general passes at Px = 2048 too
        check((nx, ny, nz), 500 + nx + ny, R=1, stage_kernel=0, engine=0)
    except MmpError:
        check((nx, ny, nz), 500 + nx + ny)


@pytest.mark.parametrize("nx,ny,nz", [(31, 6, 2), (100, 7, 1), (300, 4, 2), (700, 3, 1), (1030, 4, 1), (2000, 2, 1)])
def test_passes_a_and_c_materials(nx, ny, nz):
    """Several regions with empty cells, and two sublattices."""
    check((nx, ny, nz), 600 + nx, nreg=3, empty=0.1)
    check((nx, ny, nz), 700 + nx, n_sub=2, terms=("DEMAG", "EXCH", "ANIS", "AFM", "ZEEMAN"))


@pytest.mark.parametrize("nx,ny,nz", [(28, 620, 1), (62, 611, 1), (150, 306, 2), (250, 205, 3), (300, 612, 1)])
def test_passes_a_and_c_many_rows(nx, ny, nz):
    """More than two row pairs per SM: blocks of at most 128 threads, four cells an item."""
    check((nx, ny, nz), 800 + nx)


@pytest.mark.parametrize("shape,cell", [
    ((3, 2, 1), (2e-9, 2e-9, 2e-9)),        # fewer cells than lattice points: the differences point by point
    ((12, 11, 3), (2e-9, 2e-9, 2e-9)),      # offsets on both sides of the cutoff along x and y
    ((40, 9, 16), (4e-9, 4e-9, 5e-10)),     # every layer below the cutoff
    ((70, 50, 2), (1e-9, 4e-9, 2e-9)),      # unequal cells
    ((33, 200, 1), (2e-9, 3e-9, 2e-9)),     # lengths 96 and 512: a radix-3 pass, line counts that fill no block
])
def test_kernel_build(shape, cell):
    """The near-field lattice and the line-pair transforms of the demag kernel, demag field alone."""
    w = config_small(shape, cell, 900 + shape[0], terms=("DEMAG",))
    p = w.problem
    mag = make_magnet(p, w.m0)
    Bg, _ = gpu_eval(mag, p)
    Bo, _ = oracle_eval(p, w.m0)
    assert np.all(np.abs(Bg[0] - Bo[0]) <= field_tolerance(p, Bo[0], 0)), np.abs(Bg[0] - Bo[0]).max()
    mag.close()


@pytest.mark.parametrize("batch", [False, True])
def test_autotune_times_each_set_of_kernels_once(batch):
    """96 x 64 x 2 runs the general passes: one candidate of passes A and C, and of pass B the general kernel and
    (not in a batch) four block shapes for each of R = 2, 4 and 8.  Five evaluations a candidate and round, 36 for
    the final comparison, after a warm-up of 200 times five."""
    w = config_small((96, 64, 2), (2e-9, 2e-9, 2e-9), 31, terms=("DEMAG", "EXCH"))
    mag = make_magnet(w.problem, w.m0)
    start = mag.get_shape()
    before = mag.time()["evals"]
    shape, _ = mag.autotune(batch=batch, force=True)
    if not batch:
        assert [shape[k] for k in ("ty", "tyc", "radix_x")] == [start[k] for k in ("ty", "tyc", "radix_x")]
    assert mag.time()["evals"] - before <= 1000 + 2 * 5 * (2 if batch else 1 + 13) + 36
    mag.close()
