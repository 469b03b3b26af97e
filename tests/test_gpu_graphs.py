"""GPU: the forms of one computation that differ only in how it is launched are
bitwise equal: adaptive attempts from a graph and one by one (tracing launches
one by one), of a context and of a batch; and a batch member whose pass C is
one kernel with its own context, where the inverse x transforms and the local
field are two kernels."""
import numpy as np
import pytest

from gpu_util import make_magnet
from inputs import Problem, random_unit_vectors, stable_dt

pytestmark = pytest.mark.gpu


def _magnet(shape, seed, alpha=0.3):
    p = Problem(shape, (4e-9, 4e-9, 2e-9), 1, frozenset({"DEMAG", "EXCH", "ZEEMAN"}))
    p.set("MS", 8e5).set("AEX", 1.3e-11).set("ALPHA", alpha).set("B_EXT", (0.02, 0.0, 0.03))
    return p, make_magnet(p, [random_unit_vectors(seed, shape)])


def _m(mag):
    import torch
    nx, ny, nz = mag.shape
    out = torch.empty((3, nz, ny, nx), dtype=torch.float32, device="cuda")
    mag.get_m(0, out)
    return out.cpu().numpy()


@pytest.mark.parametrize("shape", [(48, 40, 1), (200, 24, 2), (1000, 16, 1), (1100, 10, 1), (7, 40, 2)])
@pytest.mark.parametrize("method", ["DP45", "BS23"])
def test_adaptive_graph_equals_direct_launches(shape, method):
    res = []
    for traced in (False, True):
        p, mag = _magnet(shape, 11)
        mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5, method=method)
        if traced:
            mag.profile(True)
        mag.step(7)          # the graph from the fifth attempt on
        mag.step(6)          # captured before, both sides of the buffer swap
        mag.set_param("ALPHA", 0.2, 0, -1)
        mag.step(3)          # the coefficients' contents change, the graph stays
        t = mag.time()
        res.append((_m(mag), t["t"], t["dt"], t["steps"], t["rejected"], t["evals"]))
        mag.close()
    assert np.array_equal(res[0][0], res[1][0])
    assert res[0][1:] == res[1][1:]


def test_adaptive_graph_two_sublattices():
    from inputs import config_small
    w = config_small((1000, 6, 1), (2e-9, 2e-9, 2e-9), 5, terms=("DEMAG", "EXCH", "ANIS", "AFM", "MEL", "ELASTIC"), n_sub=2)
    w.problem.glob.update(ETA=1e-15)
    res = []
    for traced in (False, True):
        mag = make_magnet(w.problem, w.m0)
        mag.set_solver(adaptive=True, dt=1e-15, tol=1e-4)
        if traced:
            mag.profile(True)
        mag.step(12)
        res.append((_m(mag), mag.time()))
        mag.close()
    assert np.array_equal(res[0][0], res[1][0])
    assert res[0][1] == res[1][1]


def test_batch_graph_and_split_pass_c_equal_solo():
    import paper_2411_18194_gb300 as pkg
    shapes = [(200, 30, 1), (300, 20, 2), (500, 9, 1), (700, 12, 1), (64, 64, 1), (1200, 6, 1)]
    solo = []
    for i, sh in enumerate(shapes):
        p, mag = _magnet(sh, 40 + i)
        mag.set_shape(R=1, stage_kernel=0, engine=0)
        mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5)
        mag.run(3e-13)
        solo.append((_m(mag), [mag.time()[k] for k in ("t", "dt", "steps", "rejected")]))
        mag.close()
    for traced in (False, True):
        mags = []
        with pkg.Batch() as b:
            for i, sh in enumerate(shapes):
                p, mag = _magnet(sh, 40 + i)
                mag.set_shape(R=1, stage_kernel=0, engine=0)
                mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5)
                mags.append(mag)
                b.add(mag, "run", 3e-13)
            if traced:
                b.profile(True)
            b.advance()
        for mag, (m, t) in zip(mags, solo):
            assert np.array_equal(_m(mag), m)
            assert [mag.time()[k] for k in ("t", "dt", "steps", "rejected")] == t
            mag.close()


def test_adaptive_graph_after_steps_of_other_methods():
    """Steps of methods with other stage counts swap k_1 with other buffers: after one fixed step each of
    Heun, Bogacki-Shampine, Dormand-Prince and Heun, y and k_1 are where the attempt graphs were captured and
    the buffer of the last stage is not."""
    res = []
    for traced in (False, True):
        p, mag = _magnet((48, 40, 1), 21)
        mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5)
        if traced:
            mag.profile(True)
        mag.step(8)          # both graphs captured
        for method in ("HEUN", "BS23", "DP45", "HEUN"):
            mag.set_solver(adaptive=False, dt=1e-14, method=method)
            mag.step(1)
        mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5)
        out = []
        for _ in range(6):
            mag.step(1)
            t = mag.time()
            out.append((_m(mag), t["t"], t["dt"], t["steps"], t["rejected"], t["evals"]))
        mag.relax(torque_tol=1e-9, max_time=1.5e-13)   # the other torque, then the first one again
        mag.step(7)
        t = mag.time()
        out.append((_m(mag), t["t"], t["dt"], t["steps"], t["rejected"], t["evals"]))
        res.append(out)
        mag.close()
    for a, b in zip(*res):
        assert np.array_equal(a[0], b[0])
        assert a[1:] == b[1:]


def test_batch_keeps_its_graph_between_advances():
    """Lock steps of one set of members replay one graph however the calls divide them; another set, or another
    shape of a member between calls, makes a new one.  Bitwise the runs of the members alone."""
    import paper_2411_18194_gb300 as pkg
    shapes = [(64, 48, 1), (100, 60, 2), (40, 130, 1)]

    def magnet(i):
        p, mag = _magnet(shapes[i], 60 + i)
        mag.set_shape(R=1, stage_kernel=0, engine=0)
        mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5)
        return mag

    mags, solo = ([magnet(i) for i in range(3)] for _ in range(2))
    with pkg.Batch() as b:
        for mag in mags:
            b.add(mag, "steps", 24)
        for _ in range(4):
            assert b.advance(4) == 3
        assert b.graphs() == 1
        sh = mags[1].get_shape()
        mags[1].set_shape(ty=4 if sh["ty"] == 2 else 2)
        assert b.advance(4) == 3 and b.graphs() == 2
        while b.advance(4):
            pass
        assert all(b.status(m) == (True, 0) for m in mags)
    for i, (mag, s) in enumerate(zip(mags, solo)):
        s.step(24)
        t, ts = mag.time(), s.time()
        if i != 1:   # member 1's change of shape drops its first stage: its own trajectory to rounding only
            assert np.array_equal(_m(mag), _m(s))
            assert [t[k] for k in ("t", "dt", "steps", "rejected")] == [ts[k] for k in ("t", "dt", "steps", "rejected")]
        mag.close()
        s.close()


def test_batch_fixed_steps_keep_their_graph_between_advances():
    import paper_2411_18194_gb300 as pkg
    (p, mag), (_, solo) = _magnet((64, 48, 2), 71), _magnet((64, 48, 2), 71)
    for x in (mag, solo):
        x.set_shape(R=1, stage_kernel=0, engine=0)
        x.set_solver(adaptive=False, dt=stable_dt(p))
    with pkg.Batch() as b:
        b.add(mag, "steps", 15)
        while b.advance(4):
            pass
        assert b.graphs() == 1
    solo.step(15)
    assert np.array_equal(_m(mag), _m(solo))
    for x in (mag, solo):
        x.close()
