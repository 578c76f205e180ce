"""The mean of the potential that the FP32 multigrid solve removes.

The starting guess is 1 on three cells of four and 1 + 2^-23 on the fourth along
x, and the tolerance lets the guess pass: the solve only removes the mean, 1 +
2^-25 in rows of a multiple of four.  Sums that round to single precision before
they reach the double-float accumulator lose the last bit of every fourth cell
(3 + (1 + 2^-23) rounds to 4), and the mean comes out 2^-25 too small.  With
every cell's term in double-float a sum of n of them is off by at most 3 n 2^-48
of their magnitudes a thread, and the mean by at most 3 n 2^-48 with n the cells
of a thread: below 2^-40 up to n = 85, which these boxes stay far under."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [32, 8, 10])  # rows taken four cells at a time, and cell by cell
def test_mean_is_removed_to_double_float(lbeh, nx):
    ny, nz = 16, 24
    rng = np.random.default_rng(nx)
    p = synth.Params(nx=nx, ny=ny, nz=nz, prec="fp32", G=0.0, eps_r=(1.0, 0.5), E_ext=(0.01, 0.0, 0.02),
                     poisson_tol=1e30, poisson_max_iter=1, poisson_solver="multigrid")
    rho = rng.uniform(0.3, 0.4, size=(2, nz, ny, nx))
    ions = rng.uniform(0.005, 0.015, size=(2, nz, ny, nx))
    phi = np.ones((nz, ny, nx))
    phi[..., 3::4] += 2.0 ** -23
    s = lbeh.System(p)
    s.set_fields(rho=list(rho), n=list(ions), phi=phi)
    assert s.step(1) == lbeh.LBEH_OK
    o = s.observables()
    assert o.poisson_solver == lbeh.LBEH_POISSON_MULTIGRID and o.poisson_iters == 0
    got = s.get(("phi",))["phi"]
    s.close()
    assert abs(got.mean()) < 2.0 ** -40, got.mean()
    assert np.array_equal(got > 0, phi > phi.mean())
