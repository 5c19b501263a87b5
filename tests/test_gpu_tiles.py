"""One step from a seeded non-equilibrium state against the FP64 oracle at grid
sizes around the step kernels' tile edges (one node short of a tile, a whole
tile, one node over; grids smaller than a tile), with walls inside the grid and
at its ends, stepped alone and in a batch.  Bounds: tests/parity_util.py, whose
rounding budget is derived there from the step's sums."""
import math
import os
import sys

import numpy as np
import pytest

import oracle
from paper_2605_30878_gb300 import lbm
from paper_2605_30878_gb300 import workloads as wl

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
import parity_util as pu  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_30878_gb300 import build
    build.build()
    lbm.load()


def _case(shape, ratio):
    """Two solid spheres (circles in 2D), one across the periodic ends."""
    nz, ny, nx = shape
    Q = 9 if nz == 1 else 19
    r = 0.18 * min(n for n in shape if n > 1)
    centers = [(0.52 * nx, 0.47 * ny, 0.5 * nz if nz > 1 else 0.0), (0.0, 0.1 * ny, 0.0)]
    solid, ghosts = wl.multi_sphere_domain(Q, shape, centers, [r, 0.8 * r])
    params = dict(lattice=Q, nx=nx, ny=ny, nz=nz, periodic=7, rho_l=ratio, rho_g=1.0,
                  mu_l=0.1 * (100.0 if ratio > 1 else 1.0), mu_g=0.1, sigma=0.005, W=4.0, M_phi=0.02,
                  theta=math.radians(70.0), g=(1e-6, -2e-6, 0.0))
    return dict(params=params, solid=solid, ghosts=ghosts, center=(0.52 * nx, 0.47 * ny, 0.5 * nz), R0=2.0 * r)


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32, lbm.FP16])
@pytest.mark.parametrize("ratio", [1.0, 1000.0])
@pytest.mark.parametrize("shape", [(1, 9, 11), (1, 31, 63), (1, 32, 64), (1, 33, 65), (1, 20, 131), (6, 7, 9),
                                   (15, 16, 63), (16, 16, 64), (17, 18, 65), (12, 34, 130)])
def test_one_step_at_tile_edges(shape, ratio, precision):
    cfg = _case(shape, ratio)
    P = dict(cfg["params"], precision=precision)
    fluid = cfg["solid"].reshape(-1) == 0
    o = oracle.Oracle(cfg["params"], cfg["solid"], cfg["ghosts"])
    o.init_droplet(cfg["center"], cfg["R0"])
    chi = o.get("N")[:, np.nonzero(fluid)[0][0]]
    Q = cfg["params"]["lattice"]
    N, _, u, p = wl.random_state(Q, fluid.size, fluid, seed=sum(shape), base=chi, amp=1e-4)
    phi = o.get("phi")
    B = np.where(fluid, phi, 0.0)[None, :] * N
    state = dict(N=N, B=B, u=u, p=p, phi=phi)
    alone = lbm.Domain(P, cfg["solid"], cfg["ghosts"])
    mate = lbm.Domain(P, cfg["solid"], cfg["ghosts"])
    for f, v in state.items():
        o.set(f, v)
        alone.write(f, v)
        mate.write(f, v)
    o.step(1)
    alone.step(1)
    want = pu.read_oracle(o)
    pu.check(pu.read_gpu(alone), want, cfg["params"], precision, fluid, 1, "%s ratio %g" % (shape, ratio))
    with lbm.Batch([mate]) as b:
        for v in range(lbm.BATCH_TILE_SHAPES):
            for f in ("N", "B", "u", "p", "phi"):
                mate.write(f, state[f])
            b.set_variant(v)
            b.step(1)
            b.sync()
            got = {f: mate.read(f) for f in want}
            for f in got:
                assert np.array_equal(got[f], alone.read(f)), (v, f)


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32])
@pytest.mark.parametrize("shape", [(1, 1500, 1021), (3, 700, 1024), (1, 5, 1200001), (1, 1, 1)])
def test_fields_read_back_whole(shape, precision):
    """Fields of several read-back pieces (4 MiB each), ragged and dense rows, a
    row longer than a piece (FP64), and one value: the values as written, in the
    domain's precision."""
    nz, ny, nx = shape
    params = dict(lattice=9 if nz == 1 else 19, nx=nx, ny=ny, nz=nz, periodic=7, rho_l=1.0, rho_g=1.0, mu_l=0.1,
                  mu_g=0.1, sigma=0.01, W=4.0, M_phi=0.02, theta=1.0, g=(0, 0, 0), precision=precision)
    d = lbm.Domain(params, np.zeros(shape, np.uint8), (np.zeros(0, np.int64), np.zeros((0, 3))))
    rng = np.random.default_rng(nx)
    kind = np.float64 if precision == lbm.FP64 else np.float32
    for f, n in (("phi", 1), ("u", 3), ("p", 1)):
        v = rng.uniform(0, 1, n * nx * ny * nz)
        if f == "u" and nz == 1:
            v[2 * nx * ny:] = 0.0
        d.write(f, v)
        assert np.array_equal(d.read(f).reshape(-1), v.astype(kind).astype(np.float64)), f


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32, lbm.FP16])
@pytest.mark.parametrize("ratio", [1.0, 1000.0])
@pytest.mark.parametrize("shape", [(1, 33, 65), (17, 18, 70)])
def test_steps_in_one_call_equal_single_steps(shape, ratio, precision):
    """A run of steps in one call (captured eight at a time, from either buffer
    parity) leaves the state of as many single steps, every field, alone and in
    a batch."""
    cfg = _case(shape, ratio)
    P = dict(cfg["params"], precision=precision)
    doms = [lbm.Domain(P, cfg["solid"], cfg["ghosts"]) for _ in range(3)]
    for d in doms:
        d.init_droplet(cfg["center"], cfg["R0"])
    one, many, mate = doms
    b = lbm.Batch([mate])
    for n in (8, 1, 19):
        for _ in range(n):
            one.step(1)
        many.step(n)
        b.step(n)
        b.sync()
        for f in ("N", "B", "phi", "u", "p"):
            want = one.read(f)
            assert np.array_equal(many.read(f), want), (n, f)
            assert np.array_equal(mate.read(f), want), (n, f, "batch")
    b.close()
