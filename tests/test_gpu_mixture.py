"""FP64 mixture viscosity against exact rationals where the phases differ widely."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_2605_30878_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_30878_gb300 import build
    build.build()
    lbm.load()


@pytest.mark.parametrize("Q", [9, 19])
@pytest.mark.parametrize("nu_l,nu_g,phi", [(0.7, 0.077, 0.93), (0.7, 7.7e-4, 1 - 1e-6), (0.7, 7.7e-7, 1 - 1e-9),
                                           (7.7e-7, 0.7, 1e-9)])
def test_relaxation_of_a_uniform_shear_stress(Q, nu_l, nu_g, phi):
    """Uniform color and N = chi + a c_x c_y: no gradient, no force, u = p = 0, so a
    step multiplies the xy stress by 1 - 1/tau, tau = 1/2 + 3 nu.  Rounding, in units
    of 2^-53 (u) of the result: the mixture, nu, tau and 1 - 1/tau have 12 operations
    or rounded parameters (12 u); the stress is 4 stored values below 2^-7, each off by
    at most one unit in its last place (2^-60), against |m| > 0.45 x 0.0046 after the
    step: 4 x 2^-60 / 0.0021 = 15 u, and as much again going in: 42 u in all."""
    n = 4
    shape = (n, n, n) if Q == 19 else (1, n, n)
    params = dict(lattice=Q, nx=n, ny=n, nz=shape[0], periodic=7, rho_l=1.0, rho_g=1.0, mu_l=nu_l, mu_g=nu_g, sigma=0.01,
                  W=4.0, M_phi=0.02, theta=1.0, g=(0, 0, 0), precision=lbm.FP64)
    d = lbm.Domain(params, np.zeros(shape, np.uint8), (np.zeros(0, np.int64), np.zeros((0, 3))))
    d.init_phi(np.full(n * n * shape[0], phi))
    c = oracle.lattice_tables(Q)["c"]
    cxy = c[:, 0] * c[:, 1]
    N = d.read("N") + 0.3 * 2.0 ** -8 * cxy[:, None]
    d.write("N", N)
    d.write("B", phi * N)

    def stress(f):
        return sum(Fraction(int(k)) * Fraction(float(v)) for k, v in zip(cxy, f[:, 0]))

    before = stress(N)
    d.step(1)
    got = stress(d.read("N")) / before
    inv_nu = Fraction(phi) / Fraction(nu_l) + (1 - Fraction(phi)) / Fraction(nu_g)
    want = 1 - 1 / (Fraction(1, 2) + 3 / inv_nu)
    assert abs(got / want - 1) <= 42 * Fraction(1, 2 ** 53), float(got / want - 1)
