"""State taken out of a domain and put back, and reads from several threads."""
import math
import threading
import time

import numpy as np
import pytest

from paper_2605_30878_gb300 import lbm
from paper_2605_30878_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

FIELDS = ("N", "B", "phi", "u", "p")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_30878_gb300 import build
    build.build()
    lbm.load()


def _drop(shape, ratio, precision, **where):
    nz, ny, nx = shape
    Q = 9 if nz == 1 else 19
    small = min(n for n in shape if n > 1)
    center = (0.5 * nx, 0.45 * ny, 0.5 * nz if nz > 1 else 0.0)
    solid, ghosts = wl.sphere_domain(Q, shape, center, 0.2 * small)
    params = dict(lattice=Q, nx=nx, ny=ny, nz=nz, periodic=7, rho_l=ratio, rho_g=1.0, mu_l=0.1 * ratio ** 0.5, mu_g=0.1,
                  sigma=0.005, W=4.0, M_phi=0.02, theta=math.radians(70.0), g=(1e-6, -2e-6, 0.0), precision=precision)
    d = lbm.Domain(params, solid, ghosts, **where)
    d.init_droplet((center[0], center[1] + 0.25 * small, center[2]), 0.2 * small)
    return d


@pytest.mark.parametrize("ratio", [1.0, 1000.0])
@pytest.mark.parametrize("shape", [(1, 33, 41), (18, 19, 22)])
def test_fp64_state_written_back_goes_on_to_the_bit(shape, ratio):
    """A run stopped, its fields written into a fresh domain and gone on with
    (either buffer parity) is the run that was not stopped."""
    one = _drop(shape, ratio, lbm.FP64)
    for n in (5, 12):
        one.step(n)
        two = _drop(shape, ratio, lbm.FP64)
        for f in FIELDS:
            two.write(f, one.read(f))
        one.step(7)
        two.step(7)
        for f in FIELDS:
            assert np.array_equal(one.read(f), two.read(f)), (n, f)


@pytest.mark.parametrize("precision", [lbm.FP64, lbm.FP32])
def test_read_of_an_idle_domain_does_not_wait_for_another_domain(precision):
    """One thread reads a domain with a second or so of steps queued; meanwhile the
    read of an idle domain on another stream returns, with the right values."""
    import torch
    busy_stream, idle_stream = torch.cuda.Stream(), torch.cuda.Stream()
    shape = (160, 160, 160)                      # few launches in a second: none blocks on a full queue
    busy, idle = _drop(shape, 10.0, precision, stream=busy_stream), _drop(shape, 10.0, precision, stream=idle_stream)
    idle.step(8)
    want = {f: idle.read(f) for f in ("phi", "u")}
    busy.step(8)
    for f in want:
        assert np.array_equal(busy.read(f), want[f])
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record(busy_stream)
    busy.step(80)
    end.record(busy_stream)
    busy.sync()
    busy.step(int(80 * 1200.0 / start.elapsed_time(end)))          # about 1.2 s
    reader = threading.Thread(target=busy.read, args=("phi",))
    reader.start()
    time.sleep(0.2)
    got = {f: idle.read(f) for f in want}
    still_running = not busy_stream.query()
    reader.join()
    assert still_running
    for f in want:
        assert np.array_equal(got[f], want[f])
