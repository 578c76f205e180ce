"""The colour-split multigrid against the oracle at the box shapes where its
layouts change: half rows that are and are not a multiple of the vector width,
rows of a multiple of two but not of four cells, an axis of two cells (a level
whose rows run along y, then along z), levels of one colour pair per row.

Tolerances are those of the other parity tests: FP64 to the 1e-13 residual of
both solves (1e-11 after three steps), FP32 single rounding of the populations
and a 1e-9 residual.
"""
import numpy as np
import pytest

import synth
from _common import compare, gpu_for, oracle_for

pytestmark = pytest.mark.gpu

BOXES = [(40, 24, 16), (12, 16, 16), (20, 24, 28), (14, 8, 16), (2, 64, 64), (4, 4, 256), (64, 2, 16)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("box", BOXES)
def test_box_shapes(lbeh, box, prec):
    nx, ny, nz = box
    rng = np.random.default_rng(nx * 10007 + ny * 101 + nz)
    p = synth.Params(nx=nx, ny=ny, nz=nz, prec=prec, G=4.0, eps_r=(1.0, 0.1), E_ext=(0.01, 0.005, 0.02),
                     poisson_tol=1e-13 if prec == "fp64" else 1e-9, poisson_max_iter=400,
                     poisson_solver="multigrid")
    rho = rng.uniform(0.04, 0.7, size=(2, nz, ny, nx))
    ions = rng.uniform(0.005, 0.015, size=(2, nz, ny, nx))
    w = synth.Workload("box", p, rho, ions)
    so, sg = oracle_for(w), gpu_for(w, lbeh)
    for _ in range(3):
        so.step()
        assert sg.step(1) == lbeh.LBEH_OK
    assert sg.observables().poisson_solver == lbeh.LBEH_POISSON_MULTIGRID
    e = compare(sg, so, ("rho", "n", "phi"))
    lim = (1e-11, 1e-11, 1e-11) if prec == "fp64" else (2e-5, 2e-5, 2e-4)
    assert e["rho"] < lim[0] and e["n"] < lim[1] and e["phi"] < lim[2], e
    sg.close()
