"""FP64 grids around the tallest that the step kernel's tiles cover: 65535 tiles of
4 rows, then of 8."""
import numpy as np
import pytest

from paper_2605_30878_gb300 import lbm

pytestmark = pytest.mark.gpu

NX, PERIOD = 4, 60


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_30878_gb300 import build
    build.build()
    lbm.load()


def _domain(ny, ratio, precision=lbm.FP64):
    params = dict(lattice=9, nx=NX, ny=ny, nz=1, periodic=7, rho_l=ratio, rho_g=1.0, mu_l=0.1 * ratio ** 0.5, mu_g=0.1,
                  sigma=0.01, W=4.0, M_phi=0.02, theta=1.0, g=(0, 0, 0), precision=precision)
    return lbm.Domain(params, np.zeros((1, ny, NX), np.uint8), (np.zeros(0, np.int64), np.zeros((0, 3))))


@pytest.mark.parametrize("ratio", [1.0, 10.0])
@pytest.mark.parametrize("ny", [4369 * PERIOD, 4370 * PERIOD, 8738 * PERIOD])      # 262140, 262200, 524280
def test_tall_grid_repeats_its_period(ny, ratio):
    """A state of period 60 along y steps as a grid of 60 rows does, to the bit."""
    y, x = np.mgrid[0:PERIOD, 0:NX]
    phi = 0.5 + 0.4 * np.sin(2 * np.pi * y / PERIOD) + 0.05 * np.cos(np.pi * x / 2 + y)
    one, tall = _domain(PERIOD, ratio), _domain(ny, ratio)
    one.init_phi(phi)
    tall.init_phi(np.tile(phi, (ny // PERIOD, 1)))
    one.step(9)
    tall.step(9)
    tall.sync()
    for f in ("phi", "u", "p"):
        got, want = tall.read(f).reshape(-1, ny // PERIOD, PERIOD * NX), one.read(f).reshape(-1, 1, PERIOD * NX)
        assert np.array_equal(got, np.broadcast_to(want, got.shape)), f


@pytest.mark.parametrize("precision,ny", [(lbm.FP64, 524281), (lbm.FP32, 262141)])
def test_taller_grid_is_refused_and_leaves_no_error_behind(precision, ny):
    with pytest.raises(lbm.LbmError, match="step launch: invalid"):
        _domain(ny, 1.0, precision)
    _domain(PERIOD, 1.0, precision).init_phi(np.full(PERIOD * NX, 0.5))
