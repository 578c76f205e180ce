"""Failures inside lbeh_step_adjoint, in forms that fault and hang no GPU: a
barrier wait of one poll runs out in the first step; a non-finite density."""
import numpy as np
import pytest

import synth
from _common import gpu_for

pytestmark = pytest.mark.gpu


def _drop(n=32):
    return synth.droplet(n=n, r=0.28 * n, prec="fp32", Ez=0.01, charge=3.0)


@pytest.mark.parametrize("every", [1, 5, 12])
@pytest.mark.parametrize("solver", ["spectral", "multigrid"])
def test_wait_that_runs_out_ends_the_sweep(lbeh, solver, every):
    """The sweep stops at the step after the failing one at the latest; with the
    default limit restored and the state loaded again the gradients come."""
    w = _drop()
    w.params.poisson_solver = solver
    s = gpu_for(w, lbeh)
    lbeh.lbeh_set_wait_limit(s.h, 1)
    with pytest.raises(lbeh.LbehError) as e:
        s.step_adjoint(12, every, d_deformation=1.0)
    assert e.value.code == lbeh.LBEH_ERR_BARRIER_TIMEOUT
    assert 1 <= s.observables().steps <= 2
    lbeh.lbeh_set_wait_limit(s.h, 0)
    s.set_fields(rho=list(w.rho), n=list(w.n))
    g = s.step_adjoint(4, 2, d_deformation=1.0)
    ref = gpu_for(w, lbeh)
    r = ref.step_adjoint(4, 2, d_deformation=1.0)
    assert g["status"] == lbeh.LBEH_OK and r["status"] == lbeh.LBEH_OK
    assert np.array_equal(g["dE_ext"], r["dE_ext"]) and g["dG"] == r["dG"]
    s.close()
    ref.close()


def test_non_finite_state_ends_the_sweep(lbeh):
    w = _drop()
    n = w.n.copy()
    n[0, 1, 2, 3] = np.nan
    s = lbeh.System(w.params)
    s.set_fields(rho=list(w.rho), n=list(n))
    with pytest.raises(lbeh.LbehError) as e:
        s.step_adjoint(12, 4, d_deformation=1.0)
    assert e.value.code == lbeh.LBEH_ERR_NONFINITE
    assert 1 <= s.observables().steps <= 2
    s.close()
