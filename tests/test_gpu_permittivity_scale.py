"""Multigrid solves at permittivities far from one, whose products leave the range
of the compute type: the operator is linear in the permittivity, so the solve
takes as many cycles as at one (one more or less where the coarse faces round
differently) and leaves a potential whose FP64 residual is below the tolerance."""
import numpy as np
import pytest

import synth
from test_spectral_lengths import _residual

pytestmark = pytest.mark.gpu

# permittivity and field: the right-hand side and the force of the field on the
# permittivity's gradient, eps E^2, stay moderate
SCALES = {"fp32": ((66, -36), (-66, 30)), "fp64": ((600, -306), (-600, 294))}


def _solve(lbeh, prec, box, eps, E):
    nx, ny, nz = box
    rng = np.random.default_rng(nx + ny + nz)
    p = synth.Params(nx=nx, ny=ny, nz=nz, nions=0, prec=prec, G=0.0, eps_r=(eps, 0.25 * eps),
                     E_ext=(E, 0.5 * E, 2.0 * E), poisson_tol=1e-6, poisson_max_iter=60, poisson_solver="multigrid")
    rho = rng.uniform(0.04, 0.7, size=(2, nz, ny, nx))
    s = lbeh.System(p)
    s.set_fields(rho=list(rho))
    rc = s.step(1)
    o = s.observables()
    phi, e = s.get(("phi",))["phi"], s.aux(lbeh.LBEH_AUX_EPS)
    s.close()
    assert rc == lbeh.LBEH_OK
    # scaled by powers of two, so that the FP64 sums of squares stay in range
    top = 2.0 ** np.floor(np.log2(np.abs(e).max()))
    return o.poisson_iters, _residual(phi / E, e / top, np.zeros_like(phi), (1.0, 0.5, 2.0))


@pytest.mark.parametrize("box", [(32, 32, 32), (32, 16, 4), (12, 20, 36)])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_solve_at_far_permittivities(lbeh, prec, box):
    base, r = _solve(lbeh, prec, box, 1.0, 2.0 ** -10)
    assert 2 <= base <= 30 and r < 1.05e-6
    for e, f in SCALES[prec]:
        it, r = _solve(lbeh, prec, box, 2.0 ** e, 2.0 ** f)
        assert abs(it - base) <= 1, (e, it, base)
        assert r < 1.05e-6, (e, r)
