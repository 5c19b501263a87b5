"""Every tile list that LBM_BATCH_PHI_SHAPE gives a batch's color kernel, against
the domains stepped alone."""
import math

import numpy as np
import pytest

from paper_2605_30878_gb300 import lbm
from paper_2605_30878_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_30878_gb300 import build
    build.build()
    lbm.load()


def _domain(shape, ratio, precision):
    nz, ny, nx = shape
    Q = 9 if nz == 1 else 19
    small = min(n for n in shape if n > 1)
    center = (0.5 * nx, 0.45 * ny, 0.5 * nz if nz > 1 else 0.0)
    solid, ghosts = wl.sphere_domain(Q, shape, center, 0.2 * small)
    params = dict(lattice=Q, nx=nx, ny=ny, nz=nz, periodic=7, rho_l=ratio, rho_g=1.0, mu_l=0.1 * ratio ** 0.5, mu_g=0.1,
                  sigma=0.005, W=4.0, M_phi=0.02, theta=math.radians(110.0), g=(1e-6, 0.0, 0.0), precision=precision)
    d = lbm.Domain(params, solid, ghosts)
    d.init_droplet((center[0], center[1] + 0.25 * small, center[2]), 0.2 * small)
    return d


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32, lbm.FP16])
@pytest.mark.parametrize("shapes", [[(1, 33, 65), (1, 24, 131)], [(15, 17, 33), (18, 16, 65)]])
def test_color_tile_lists_give_the_same_bits(shapes, precision, monkeypatch):
    ratios = (1.0, 100.0)
    alone = [_domain(s, r, precision) for s, r in zip(shapes, ratios)]
    for d in alone:
        d.step(9)
    want = [{f: d.read(f) for f in ("N", "B", "phi", "u", "p")} for d in alone]
    for tiles in ["rows", "step"] + [str(v) for v in range(lbm.BATCH_TILE_SHAPES)]:
        monkeypatch.setenv("LBM_BATCH_PHI_SHAPE", tiles)
        doms = [_domain(s, r, precision) for s, r in zip(shapes, ratios)]
        with lbm.Batch(doms) as b:
            b.step(9)
            b.sync()
        for d, w in zip(doms, want):
            for f in w:
                assert np.array_equal(d.read(f), w[f]), (tiles, f)
