"""Timing cases of the micromagnetic library, through its Python entry points.

Each case is a piece of a simulation that a program does again and again: a
few time steps of one magnet from a given state, a relaxation, the effective
field of a state, a batch of independent magnets advanced together, the demag
field alone, or the set-up and first field of a new geometry.  Sizes and
materials are those of the seeded workloads in `inputs/`, of the tests, or
generic.

`exact` is a plain FP64 restatement in torch of what the calls return (demag
tensor, field terms, torque, elastodynamics, Dormand-Prince steps); it uses
none of the library's code.
"""
import math

import numpy as np
import torch

import paper_2411_18194_gb300 as mmp
from inputs import Problem, stable_dt

MU0 = 4e-7 * math.pi
GAMMA = 1.7595e11

AFM_DT = 5e-15   # the fixed step of the antiferromagnet workload


# ------------------------------------------------------------------- cases --
def listed():
    return [
        # A small plain ferromagnet, fixed steps: launches and latency (the 64 x 64 workload).
        dict(name="steps 64x64x1", kind="steps", nx=64, ny=64, nz=1, material="plain", steps=10),
        # A relaxation request of the served workload: one error read-back per attempt.
        dict(name="relax 256x256x2", kind="relax", nx=256, ny=256, nz=2, material="film", time=1e-12),
        # A single-layer film, adaptive steps over a short time: the ordinary interactive size.
        dict(name="run 512x512x1", kind="run", nx=512, ny=512, nz=1, material="film", time=3e-13),
        # A multilayer of 3 * 2^k cells per side, fixed steps (sizes of the batched workload, alone).
        dict(name="steps 384x192x4", kind="steps", nx=384, ny=192, nz=4, material="plain", steps=4),
        # A long racetrack strip: the longest x transforms.
        dict(name="run 2048x128x1", kind="run", nx=2048, ny=128, nz=1, material="dmi", time=1.5e-13),
        # The large ferromagnet of the benchmark: anisotropy, interfacial DMI, adaptive steps.
        dict(name="run 1024x1024x8", kind="run", nx=1024, ny=1024, nz=8, material="dmi", time=1e-13),
        # The two-sublattice antiferromagnet with magnetoelastic coupling and elastodynamics.
        dict(name="afm 1024x256x1", kind="afm", nx=1024, ny=256, nz=1, steps=4),
        # Field and torque of a patterned sample: odd sizes, several regions, empty cells, every local term.
        dict(name="field 300x213x3", kind="field", nx=300, ny=213, nz=3, regions=4, empty=0.1),
        # Independent magnets of uneven sizes advanced together, ten fixed steps each.
        dict(name="batch 24 fixed", kind="batch", members=24, pick=3, goal="steps", steps=10),
        # Served relaxations advanced together: one read-back per lock step for all of them.
        dict(name="batch 8 relax", kind="batch", members=8, pick=4, goal="relax", time=5e-13),
        # The demag field of a caller's magnetisation, without allocations.
        dict(name="demag 128x100x4", kind="demag", nx=128, ny=100, nz=4),
        # A new geometry: context, demag kernel spectrum, first field.
        dict(name="new 256x256x4", kind="new", nx=256, ny=256, nz=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi, cells, nzs):
    """Extents spread over the logarithm of lo .. hi, of at most `cells` cells; every third one a round size."""
    while True:
        nx, ny, nz = _log_int(rng, lo, hi), _log_int(rng, lo, hi), rng.choice(nzs)
        if rng.random() < 1 / 3:
            round_sizes = [s for s in (32, 64, 96, 128, 192, 256, 384, 512, 768, 1024) if lo <= s <= hi]
            nx, ny = rng.choice(round_sizes), rng.choice(round_sizes)
        if nx * ny * nz <= cells:
            return dict(nx=nx, ny=ny, nz=nz)


def draw(rng):
    kind = rng.choice(["steps", "steps", "run", "relax", "afm", "field", "batch", "demag", "new"])
    if kind in ("steps", "run"):
        g = _grid(rng, 32, 1024, 1 << 21, (1, 1, 2, 3, 4, 8))
        if rng.random() < 0.15:   # a strip
            g = dict(nx=_log_int(rng, 1025, 2048), ny=_log_int(rng, 32, 256), nz=1)
        material = rng.choice(["plain", "film", "dmi"])
        if kind == "run":
            return dict(kind="run", **g, material=material, time=1e-13 if material == "dmi" else 3e-13)
        return dict(kind="steps", **g, material=material, steps=rng.choice([2, 4]))
    if kind == "relax":
        return dict(kind="relax", **_grid(rng, 64, 1024, 1 << 20, (1, 2, 4)), material="film", time=1e-12)
    if kind == "afm":
        return dict(kind="afm", **_grid(rng, 64, 1024, 1 << 19, (1, 1, 2)), steps=2)
    if kind == "field":
        return dict(kind="field", **_grid(rng, 20, 700, 1 << 20, (1, 2, 3, 5)), regions=rng.choice([2, 3, 6]),
                    empty=rng.choice([0.0, 0.1, 0.3]))
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind="batch", members=rng.randint(4, 40), pick=rng.randint(0, 1 << 20), goal="steps",
                        steps=rng.choice([2, 4, 10]))
        return dict(kind="batch", members=rng.randint(2, 12), pick=rng.randint(0, 1 << 20), goal="relax", time=5e-13)
    if kind == "demag":
        return dict(kind="demag", **_grid(rng, 16, 256, 52000, (1, 2, 3, 4)))
    return dict(kind="new", **_grid(rng, 64, 512, 1 << 19, (1, 2, 4)))


# ---------------------------------------------------------------- problems --
def _ferromagnet(nx, ny, nz, material):
    if material == "plain":
        p = Problem((nx, ny, nz), (4e-9, 4e-9, 4e-9), 1, frozenset({"DEMAG", "EXCH", "ZEEMAN"}))
        p.set("MS", 8e5).set("AEX", 1.3e-11).set("ALPHA", 0.02).set("B_EXT", (0.0, 0.0, 0.01))
    elif material == "film":   # the served relaxation requests
        p = Problem((nx, ny, nz), (4e-9, 4e-9, 2e-9), 1, frozenset({"DEMAG", "EXCH", "ZEEMAN"}))
        p.set("MS", 8e5).set("AEX", 1.3e-11).set("ALPHA", 0.5).set("B_EXT", (0.02, 0.0, 0.03))
    else:   # "dmi"
        p = Problem((nx, ny, nz), (2e-9, 2e-9, 1e-9), 1, frozenset({"DEMAG", "EXCH", "ANIS", "DMI"}))
        p.set("MS", 1.1e6).set("AEX", 1.6e-11).set("ALPHA", 0.1)
        p.set("KU1", 8e5).set("ANIS_U", (0.0, 0.0, 1.0)).set("DIND", 3e-3)
    return p


def _antiferromagnet(nx, ny, nz):
    p = Problem((nx, ny, nz), (2e-9, 2e-9, 2e-9), 2,
                frozenset({"DEMAG", "EXCH", "ANIS", "AFM", "MEL", "ELASTIC"}))
    p.set("MS", 4e5).set("AEX", 1e-11).set("ALPHA", 0.01)
    p.set("KU1", 8.57e4).set("ANIS_U", (1.0, 0.0, 0.0)).set("KB1", -8.57e5).set("ANIS_UB", (0.0, 0.0, 1.0))
    p.set("B1", -1e7).set("B2", -1e7)
    p.glob.update(A0=-4e-11, A12=-1e-12, LATTICE_A=0.42e-9, C11=2.5e11, C12=1.5e11, C44=1e11, RHO=7e3, ETA=0.0)
    return p


def _patterned(case, seed):
    """Several regions of different material in columns through the layers, some of them empty."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(seed)
    p = Problem((nx, ny, nz), (2e-9, 2.5e-9, 1.5e-9), 1,
                frozenset({"DEMAG", "EXCH", "ANIS", "DMI", "ZEEMAN", "CUBIC"}))
    size = 16
    blocks = rng.integers(0, case["regions"], (ny // size + 1, nx // size + 1))
    blocks[rng.random(blocks.shape) < case["empty"]] = 255
    plane = np.kron(blocks, np.ones((size, size), dtype=np.int64))[:ny, :nx]
    p.regions = np.ascontiguousarray(np.broadcast_to(plane, (nz, ny, nx))).astype(np.uint8)
    for r in range(case["regions"]):
        v = rng.random(6)
        p.set("MS", 4e5 + 8e5 * v[0], 0, r).set("AEX", 5e-12 + 1.5e-11 * v[1], 0, r)
        p.set("ALPHA", 0.01 + 0.3 * v[2], 0, r).set("KU1", 1e5 + 5e5 * v[3], 0, r).set("KU2", 2e4, 0, r)
        p.set("KC1", 5e4 * (v[4] - 0.3), 0, r).set("DIND", 3e-3 * (v[5] - 0.3), 0, r)
        p.set("B_EXT", (0.02, -0.01, 0.05), 0, r)
    p.set("MS", 0.0, None, 255)
    return p


def _batch_problems(case):
    """Uneven sizes and materials of the batch, from the case's own pick (the states come from the seed)."""
    rng = np.random.default_rng(case["pick"])
    out = []
    for _ in range(case["members"]):
        if case["goal"] == "steps":
            nx, ny = (int(v) for v in rng.choice([32, 64, 96, 128, 192, 256, 384, 512], 2))
            p = Problem((nx, ny, int(rng.choice([1, 2, 4]))), (2e-9, 2e-9, 2e-9), 1, frozenset({"DEMAG", "EXCH"}))
            p.set("MS", 4e5 + 1e6 * rng.random()).set("AEX", 5e-12 + 1.5e-11 * rng.random())
            p.set("ALPHA", 0.01 + 0.49 * rng.random())
        else:
            n = (64, 128, 256, 512)[int(rng.random() ** 2 * 4)]
            p = _ferromagnet(n, n, int(rng.choice([1, 2, 4])) if n <= 256 else 1, "film")
            p.set("B_EXT", (0.05 * (rng.random() - 0.5), 0.0, 0.05 * rng.random()))
        out.append(p)
    return out


def _unit_vectors(shape, seed):
    """Random directions, float32 [3][nz][ny][nx] on the GPU."""
    nx, ny, nz = shape
    gen = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn((3, nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    return (v / v.norm(dim=0)).float()


def _noisy_axis(shape, sign, seed):
    """Directions within about a degree of +-x."""
    nx, ny, nz = shape
    gen = torch.Generator(device="cuda").manual_seed(seed)
    v = 0.01 * torch.randn((3, nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    v[0] = sign
    return (v / v.norm(dim=0)).float()


def _problems(case, seed):
    kind = case["kind"]
    if kind in ("steps", "run", "relax"):
        return [_ferromagnet(case["nx"], case["ny"], case["nz"], case["material"])]
    if kind == "new":
        return [_ferromagnet(case["nx"], case["ny"], case["nz"], "film")]
    if kind == "afm":
        return [_antiferromagnet(case["nx"], case["ny"], case["nz"])]
    if kind == "field":
        return [_patterned(case, seed)]
    if kind == "batch":
        return _batch_problems(case)
    p = Problem((case["nx"], case["ny"], case["nz"]), (4e-9, 4e-9, 2e-9), 1, frozenset({"DEMAG"}))
    p.set("MS", 8e5)
    return [p]


def _states(case, seed, problems):
    if case["kind"] == "afm":
        p = problems[0]
        return [_noisy_axis(p.shape, 1.0, seed), _noisy_axis(p.shape, -1.0, seed + 7919)]
    return [_unit_vectors(p.shape, seed + 7919 * i) for i, p in enumerate(problems)]


# --------------------------------------------------------------- the passes --
def prepare(case, seed):
    problems = _problems(case, seed)
    m0 = _states(case, seed, problems)
    s = dict(case=case, problems=problems, m0=m0, out=[torch.empty_like(m) for m in m0])
    kind = case["kind"]
    if kind == "demag":
        s["M"] = m0[0] * 8e5
    elif kind != "new":
        s["mags"] = [mmp.Magnet.from_problem(p) for p in problems]
        if kind == "batch":
            for mag in s["mags"]:
                mag.set_shape(R=1, stage_kernel=0, engine=0)
        if kind == "field":
            s["mags"][0].set_m(0, m0[0])
            s["tau"] = torch.empty_like(m0[0])
        if kind == "afm":
            s["u0"] = torch.zeros_like(m0[0])
            s["u"], s["v"] = torch.empty_like(m0[0]), torch.empty_like(m0[0])
    return s


def run(s):
    case, m0, out = s["case"], s["m0"], s["out"]
    kind = case["kind"]
    if kind == "demag":
        p = s["problems"][0]
        return mmp.demag_noalloc(p.shape, p.cell, s["M"], out[0])
    if kind == "new":
        tau = torch.empty_like(out[0])
        with mmp.Magnet.from_problem(s["problems"][0]) as mag:
            mag.set_m(0, m0[0])
            mag.eval_field(0, out[0], tau)
        return dict(B=out[0], tau=tau)
    if kind == "batch":
        with mmp.Batch() as batch:
            for p, mag, m in zip(s["problems"], s["mags"], m0):
                mag.set_m(0, m)
                if case["goal"] == "steps":
                    mag.set_solver(adaptive=False, dt=stable_dt(p))
                    batch.add(mag, "steps", case["steps"])
                else:
                    mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5)
                    batch.add(mag, "relax", 1e-4, case["time"])
            batch.advance()
        for mag, o in zip(s["mags"], out):
            mag.get_m(0, o)
        return out
    mag = s["mags"][0]
    if kind == "field":
        mag.set_m(0, m0[0])
        mag.eval_field(0, out[0], s["tau"])
        return dict(B=out[0], tau=s["tau"])
    for i, m in enumerate(m0):
        mag.set_m(i, m)
    if kind == "afm":
        mag.set_elastic(s["u0"], s["u0"])
        mag.set_solver(adaptive=False, dt=AFM_DT)
        mag.step(case["steps"])
        for i, o in enumerate(out):
            mag.get_m(i, o)
        mag.get_elastic(s["u"], s["v"])
        return dict(m=out, u=s["u"], v=s["v"])
    if kind == "steps":
        mag.set_solver(adaptive=False, dt=stable_dt(s["problems"][0]))
        mag.step(case["steps"])
    else:
        mag.set_solver(adaptive=True, dt=2e-14, tol=1e-5)
        if kind == "run":
            mag.run(case["time"])
        else:
            mag.relax(torque_tol=1e-4, max_time=case["time"])
    return mag.get_m(0, out[0])


# ---------------------------------------------------------------- the floor --
_STAGE_READS = (2, 3, 4, 5, 6, 6)   # vectors that stages 2 .. 7 of Dormand-Prince read: y and the k_j they use


def _padded(n):
    return 1 if n == 1 else 2 * n


def _field_work(p):
    """One field and torque: the kernel octant read once; transforms of the zero-padded grid, multiply, local terms."""
    nx, ny, nz = p.shape
    px, py, pz = (_padded(v) for v in p.shape)
    n = nx * ny * nz
    octant = 24.0 * (px // 2 + 1) * (py // 2 + 1) * (pz // 2 + 1)
    kx = px // 2 + 1
    lg = lambda v: math.log2(v) if v > 1 else 0.0   # noqa: E731
    flops = 2 * 3 * (2.5 * px * lg(px) * ny * nz + 5.0 * py * lg(py) * nz * kx + 5.0 * pz * lg(pz) * kx * py)
    flops += 36.0 * kx * py * pz + 150.0 * n * p.n_sub
    return octant, flops


def _steps_work(p, steps, adaptive):
    """First stage, then `steps` steps of six evaluations: state and stage vectors in and out, kernel octant."""
    n = p.n_cells
    parts = p.n_sub + (2 if "ELASTIC" in p.terms else 0)
    vec = 12.0 * n * parts
    octant, flops = _field_work(p)
    per_step = sum(_STAGE_READS) + 6 + 1 + (6 if adaptive else 0)
    return 2 * vec + octant + steps * (per_step * vec + 6 * octant), (1 + 6 * steps) * flops


def work(case):
    kind = case["kind"]
    total = np.zeros(2)
    for p in _problems(case, 0):
        if "steps" in case:
            total += _steps_work(p, case["steps"], False)
        elif "time" in case:
            # the fastest exchange mode sets the adaptive step (2e-14 s the first one)
            total += _steps_work(p, 2 + int(case["time"] / (2.5 * stable_dt(p))), True)
        else:
            octant, flops = _field_work(p)
            outputs = 1 if kind == "demag" else 2
            # a new geometry makes its octant itself, six FP64 transforms of the offsets
            total += (12.0 * p.n_cells * (1 + outputs) + octant, flops * (2.0 if kind == "new" else 1.0))
    return dict(bytes=float(total[0]), flops=float(total[1]))


# ------------------------------------------------------- the FP64 statement --
def exact(case, seed):
    problems = _problems(case, seed)
    states = [m.double() for m in _states(case, seed, problems)]
    kind = case["kind"]
    if kind == "demag":
        return _Fields(problems[0]).demag((states[0] * 8e5).float().double())
    if kind in ("field", "new"):
        f = _Fields(problems[0])
        B = f.effective([states[0]], None)
        return dict(B=B[0], tau=f.torque(0, states[0], B[0]))
    if kind == "afm":
        f = _Fields(problems[0])
        zero = torch.zeros_like(states[0])
        y = _advance(f, states + [zero, zero.clone()], AFM_DT, steps=case["steps"])
        return dict(m=y[:2], u=y[2], v=y[3])
    out = []
    for p, m in zip(problems, states):
        f = _Fields(p)
        if "steps" in case:
            y = _advance(f, [m], stable_dt(p), steps=case["steps"])
        else:
            y = _advance(f, [m], 2e-14, adaptive=True, until=case["time"], relax=kind != "run")
        out.append(y[0])
    return out if kind == "batch" else out[0]


def _newell_f(x, y, z):
    x, y, z = x.abs(), y.abs(), z.abs()
    r = torch.sqrt(x * x + y * y + z * z)
    tiny = 1e-300
    rxz, rxy = torch.sqrt(x * x + z * z), torch.sqrt(x * x + y * y)
    out = (2 * x * x - y * y - z * z) * r / 6
    out = out + torch.where(rxz > 0, 0.5 * y * (z * z - x * x) * torch.asinh(y / (rxz + tiny)), 0 * x)
    out = out + torch.where(rxy > 0, 0.5 * z * (y * y - x * x) * torch.asinh(z / (rxy + tiny)), 0 * x)
    return out - torch.where(x * r > 0, x * y * z * torch.atan(y * z / (x * r + tiny)), 0 * x)


def _newell_g(x, y, z):
    sign = torch.sign(x) * torch.sign(y)
    x, y, z = x.abs(), y.abs(), z.abs()
    r = torch.sqrt(x * x + y * y + z * z)
    tiny = 1e-300
    rxy, ryz, rxz = torch.sqrt(x * x + y * y), torch.sqrt(y * y + z * z), torch.sqrt(x * x + z * z)
    out = -x * y * r / 3
    out = out + torch.where(rxy > 0, x * y * z * torch.asinh(z / (rxy + tiny)), 0 * x)
    out = out + torch.where(ryz > 0, y / 6 * (3 * z * z - y * y) * torch.asinh(x / (ryz + tiny)), 0 * x)
    out = out + torch.where(rxz > 0, x / 6 * (3 * z * z - x * x) * torch.asinh(y / (rxz + tiny)), 0 * x)
    out = out - torch.where(z * r > 0, z ** 3 / 6 * torch.atan(x * y / (z * r + tiny)), 0 * x)
    out = out - torch.where(y * r > 0, z * y * y / 2 * torch.atan(x * z / (y * r + tiny)), 0 * x)
    return sign * (out - torch.where(x * r > 0, z * x * x / 2 * torch.atan(y * z / (x * r + tiny)), 0 * x))


def _second_difference(fun, x, y, z, a, b, c):
    w, acc = {-1: -1.0, 0: 2.0, 1: -1.0}, 0.0
    for i in w:
        for j in w:
            for k in w:
                acc = acc + w[i] * w[j] * w[k] * fun(x + i * a, y + j * b, z + k * c)
    return acc / (4 * math.pi * a * b * c)


def _triangular_nodes(count=5):
    """Gauss nodes and weights of the density 1 - |s| on [-1, 1] (difference of two uniform points)."""
    mom = [2.0 / ((k + 1) * (k + 2)) if k % 2 == 0 else 0.0 for k in range(2 * count + 1)]
    chol = np.linalg.cholesky(np.array([[mom[i + j] for j in range(count + 1)] for i in range(count + 1)])).T
    off = [chol[k + 1, k + 1] / chol[k, k] for k in range(count - 1)]
    nodes, vec = np.linalg.eigh(np.diag(off, 1) + np.diag(off, -1))
    return nodes, vec[0] ** 2


def _tensor_octant(shape, cell):
    """Cell-to-cell demag tensor (xx, yy, zz, xy, xz, yz) at the offsets i, j, k >= 0: Newell's formula near, the
    dipole kernel averaged over the difference of the two cells' points (Gauss quadrature) from ten cells on."""
    L = max(cell)
    a, b, c = (v / L for v in cell)
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) * d for n, d in zip(shape, (a, b, c))]
    Z, Y, X = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    out = torch.zeros((6,) + X.shape, device="cuda", dtype=torch.float64)
    nodes, weights = _triangular_nodes()
    origin = X * X + Y * Y + Z * Z < 1.0
    for sx, wx in zip(nodes, weights):
        for sy, wy in zip(nodes, weights):
            for sz, wz in zip(nodes, weights):
                x, y, z = X + sx * a, Y + sy * b, Z + sz * c
                r2 = torch.where(origin, torch.ones_like(X), x * x + y * y + z * z)
                k3 = (wx * wy * wz * a * b * c / (4 * math.pi)) * r2.pow(-1.5)
                k5 = 3 * k3 / r2
                for q, (u, v) in enumerate(((x, x), (y, y), (z, z), (x, y), (x, z), (y, z))):
                    out[q] -= k5 * u * v
                out[:3] += k3
    m = [min(n, int(10.0 / d) + 2) for n, d in zip(shape, (a, b, c))]
    X, Y, Z = (v[:m[2], :m[1], :m[0]].contiguous() for v in (X, Y, Z))
    near = torch.stack([_second_difference(_newell_f, X, Y, Z, a, b, c), _second_difference(_newell_f, Y, X, Z, b, a, c),
                        _second_difference(_newell_f, Z, Y, X, c, b, a), _second_difference(_newell_g, X, Y, Z, a, b, c),
                        _second_difference(_newell_g, X, Z, Y, a, c, b), _second_difference(_newell_g, Y, Z, X, b, c, a)])
    part = out[:, :m[2], :m[1], :m[0]]
    part.copy_(torch.where(X * X + Y * Y + Z * Z < 100.0, near, part))
    return out


def _gradient_matrix(n, h):
    """First derivative along an axis: 4th order in the bulk, 2nd order one cell in, one-sided at the edges."""
    G = np.zeros((n, n))
    if n == 2:
        G[:, 0], G[:, 1] = -1.0, 1.0
    elif n > 2:
        for i in range(n):
            if i == 0:
                G[i, :3] = (-1.5, 2.0, -0.5)
            elif i == n - 1:
                G[i, -3:] = (0.5, -2.0, 1.5)
            elif i in (1, n - 2):
                G[i, i - 1], G[i, i + 1] = -0.5, 0.5
            else:
                G[i, i - 2:i + 3] = np.array((1.0, -8.0, 0.0, 8.0, -1.0)) / 12.0
    return torch.from_numpy(G / h).cuda()


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


class _Fields:
    """Effective field, torque and elastic force of a Problem in FP64, arrays [3][nz][ny][nx]."""

    def __init__(self, p):
        self.p = p
        reg = torch.from_numpy(p.regions.astype(np.int64)).cuda()
        self.scal = {k: [torch.from_numpy(np.ascontiguousarray(v[s])).cuda()[reg] for s in range(p.n_sub)]
                     for k, v in p.scal.items()}
        self.vec = {k: [torch.from_numpy(np.ascontiguousarray(v[s])).cuda()[reg].movedim(-1, 0)
                        for s in range(p.n_sub)] for k, v in p.vec.items()}
        self.G = None
        if "ELASTIC" in p.terms:
            self.G = [_gradient_matrix(n, h) for n, h in zip(p.shape, p.cell)]
        self.K = self._spectrum() if "DEMAG" in p.terms else None

    # ------------------------------------------------------------- demag --
    def _spectrum(self):
        self.P = [_padded(n) for n in self.p.shape]
        octant = _tensor_octant(self.p.shape, self.p.cell)
        odd = ((0, 0, 0), (0, 0, 0), (0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1))
        out = []
        for comp, signs in zip(octant, odd):
            full = comp
            for axis in range(3):   # x, y, z on dimensions 2, 1, 0
                n, P, dim = self.p.shape[axis], self.P[axis], 2 - axis
                if P == 1:
                    continue
                back = full.narrow(dim, 1, n - 1).flip(dim) * (-1.0 if signs[axis] else 1.0)
                gap = list(full.shape)
                gap[dim] = P - 2 * n + 1
                full = torch.cat([full, torch.zeros(gap, device="cuda", dtype=torch.float64), back], dim)
            out.append(torch.fft.rfftn(full))
        return out

    def demag(self, M):
        nx, ny, nz = self.p.shape
        F = [torch.fft.rfftn(M[c], s=(self.P[2], self.P[1], self.P[0])) for c in range(3)]
        K = self.K
        H = (K[0] * F[0] + K[3] * F[1] + K[4] * F[2], K[3] * F[0] + K[1] * F[1] + K[5] * F[2],
             K[4] * F[0] + K[5] * F[1] + K[2] * F[2])
        size = (self.P[2], self.P[1], self.P[0])
        return torch.stack([-MU0 * torch.fft.irfftn(h, s=size)[:nz, :ny, :nx] for h in H])

    # ------------------------------------------------------- local terms --
    @staticmethod
    def _neighbour(a, axis, d, fill):
        dim = a.dim() - 1 - axis
        n = a.shape[dim]
        edge = torch.full_like(a.narrow(dim, 0, 1), fill)
        if d > 0:
            return torch.cat([a.narrow(dim, 1, n - 1), edge], dim)
        return torch.cat([edge, a.narrow(dim, 0, n - 1)], dim)

    def _axes(self):
        for axis in range(3):
            for d in (-1, 1):
                yield axis, d, self.p.cell[axis]

    def effective(self, ms, u):
        p, t = self.p, self.p.terms
        eps = self._strain(u) if "MEL" in t else None
        bd = self.demag(sum(self.scal["MS"][s] * ms[s] for s in range(p.n_sub))) if "DEMAG" in t else 0.0
        return [self._local(s, ms, eps) + bd if p.scal["MS"].all() else
                (self._local(s, ms, eps) + bd) * (self.scal["MS"][s] > 0) for s in range(p.n_sub)]

    def _local(self, s, ms, eps):
        t, g, m = self.p.terms, self.p.glob, ms[s]
        q = {k: v[s] for k, v in self.scal.items()}
        inv = torch.where(q["MS"] > 0, 1.0 / q["MS"], torch.zeros_like(q["MS"]))
        B = torch.zeros_like(m)
        for axis, d, h in self._axes():
            there = self._neighbour(q["MS"], axis, d, 0.0) > 0
            nb = self._neighbour(m, axis, d, 0.0)
            dmi = "DMI" in t and axis < 2
            if dmi:   # the boundary value m + h d_n m, d_n m = -(D / 2A) (z x n) x m
                zero = torch.zeros_like(m[0])
                w = torch.stack([m[2], zero, -m[0]] if axis == 0 else [zero, m[2], -m[1]])
                ghost = m - d * h * q["DIND"] / (2 * q["AEX"] + 1e-300) * w
            else:
                ghost = m
            if "EXCH" in t:
                A = self._neighbour(q["AEX"], axis, d, 0.0)
                pair = torch.where(there, 2 * q["AEX"] * A / (q["AEX"] + A + 1e-300), q["AEX"])
                B = B + 2 * pair * inv / (h * h) * (torch.where(there, nb, ghost) - m)
            if dmi:
                D = torch.where(there, 0.5 * (q["DIND"] + self._neighbour(q["DIND"], axis, d, 0.0)), q["DIND"])
                v = torch.where(there, nb, ghost)
                B[axis] += d * D * inv / h * v[2]
                B[2] -= d * D * inv / h * v[axis]
        if "ANIS" in t:
            e, eb = self.vec["ANIS_U"][s], self.vec["ANIS_UB"][s]
            c = (m * e).sum(0)
            B = B + (2 * q["KU1"] * c + 4 * q["KU2"] * c ** 3) * inv * e + 2 * q["KB1"] * inv * (m * eb).sum(0) * eb
        if "CUBIC" in t:
            c1 = self.vec["ANIS_C1"][s]
            c1 = c1 / c1.norm(dim=0)
            c2 = self.vec["ANIS_C2"][s]
            c2 = c2 - (c1 * c2).sum(0) * c1
            c2 = c2 / c2.norm(dim=0)
            c3 = _cross(c1, c2)
            a, b, c = ((m * e).sum(0) for e in (c1, c2, c3))
            B = B - 2 * q["KC1"] * inv * (a * (b * b + c * c) * c1 + b * (a * a + c * c) * c2 + c * (a * a + b * b) * c3)
        if "ZEEMAN" in t:
            B = B + self.vec["B_EXT"][s]
        if "AFM" in t:
            o = ms[1 - s]
            for axis, d, h in self._axes():
                there = self._neighbour(torch.ones_like(m[0]), axis, d, 0.0)
                B = B + g["A12"] * inv / (h * h) * there * (self._neighbour(o, axis, d, 0.0) - o)
            B = B + 4 * g["A0"] * inv / g["LATTICE_A"] ** 2 * o
        if eps is not None:
            b1, b2 = -2 * q["B1"] * inv, -2 * q["B2"] * inv
            B = B + torch.stack([
                b1 * eps[0] * m[0] + b2 * (eps[3] * m[1] + eps[4] * m[2]),
                b1 * eps[1] * m[1] + b2 * (eps[3] * m[0] + eps[5] * m[2]),
                b1 * eps[2] * m[2] + b2 * (eps[4] * m[0] + eps[5] * m[1])])
        return B

    def torque(self, s, m, B, relax=False):
        al = self.scal["ALPHA"][s]
        mxb = _cross(m, B)
        return -GAMMA / (1 + al * al) * (al * _cross(m, mxb) + (0.0 if relax else mxb))

    # ----------------------------------------------------------- elastic --
    def _along(self, f, axis, transpose=False):
        G = self.G[axis].T if transpose else self.G[axis]
        dim = f.dim() - 1 - axis
        return (f.movedim(dim, -1) @ G.T).movedim(-1, dim)

    def _strain(self, u):
        D = [[self._along(u[j], a) for j in range(3)] for a in range(3)]
        return [D[0][0], D[1][1], D[2][2], 0.5 * (D[0][1] + D[1][0]), 0.5 * (D[0][2] + D[2][0]),
                0.5 * (D[1][2] + D[2][1])]

    def acceleration(self, ms, u):
        g, e = self.p.glob, self._strain(u)
        sig = [g["C11"] * e[i] + g["C12"] * (e[(i + 1) % 3] + e[(i + 2) % 3]) for i in range(3)]
        sig += [2 * g["C44"] * e[i] for i in (3, 4, 5)]
        at = ((0, 3, 4), (3, 1, 5), (4, 5, 2))
        f = [-sum(self._along(sig[at[a][b]], a, True) for a in range(3)) for b in range(3)]
        for s, m in enumerate(ms):
            b1, b2 = self.scal["B1"][s], self.scal["B2"][s]
            D = [[self._along(m[j], a) for j in range(3)] for a in range(3)]
            for i in range(3):
                j, k = (i + 1) % 3, (i + 2) % 3
                f[i] = f[i] + 2 * b1 * m[i] * D[i][i] + b2 * (m[i] * (D[j][j] + D[k][k]) + m[j] * D[j][i] + m[k] * D[k][i])
        return torch.stack(f) / g["RHO"]

    def derivative(self, y, relax):
        ns = self.p.n_sub
        u = y[ns] if "ELASTIC" in self.p.terms else None
        B = self.effective(y[:ns], u)
        k = [self.torque(s, y[s], B[s], relax) for s in range(ns)]
        return k if u is None else k + [y[ns + 1].clone(), self.acceleration(y[:ns], u)]


_A = ((1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
      (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
      (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
      (35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
_B4 = (5179 / 57600, 0.0, 7571 / 16695, 393 / 640, -92097 / 339200, 187 / 2100, 1 / 40)


def _advance(f, y, dt, adaptive=False, steps=0, until=None, relax=False, tol=1e-5):
    """Dormand-Prince steps (m renormalised at the 5th-order stage, whose derivative is the next first stage)."""
    ns, t, done = f.p.n_sub, 0.0, 0
    k1 = f.derivative(y, relax)
    while t < until * (1 - 1e-15) if until is not None else done < steps:
        h = dt if until is None else min(dt, until - t)
        ks = [k1]
        for i, row in enumerate(_A):
            yi = [a + h * sum(c * k[j] for c, k in zip(row, ks) if c) for j, a in enumerate(y)]
            if i == 5:
                yi = [v / v.norm(dim=0) if j < ns else v for j, v in enumerate(yi)]
            ks.append(f.derivative(yi, relax))
        ok = True
        if adaptive:
            err = h * max(float(sum((a - b) * k[s] for a, b, k in zip(_A[5] + (0.0,), _B4, ks)).abs().max())
                          for s in range(ns))
            ok = err <= tol
            dt = min(max(h * min(max(0.9 * (tol / err) ** 0.2, 0.2), 5.0), 1e-18), 1e-11)
        if ok:
            y, k1, t, done = yi, ks[6], t + h, done + 1
    return y
