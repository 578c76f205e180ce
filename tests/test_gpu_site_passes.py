"""The site passes at the sizes where their work is split differently.

Read-out: one pass writes the wanted fields in the caller's element type.  A
single-precision read is the double-precision read rounded once; the potential
of the FP32 modes is a pair of FP32 words, whose sum may round twice: one unit
of the 24-bit significand, 2^-23.  A density is the sum of the populations that
are read beside it: 19 terms summed in the compute type, at most 18 roundings
of at most the sum of their magnitudes.

Ion update and sites near colloids: rows that are and are not a multiple of
four sites, without spheres and with spheres that cross the faces, an edge and a
corner of the box or nearly touch.  Tolerances are those of the other parity
tests: FP64 1e-11 (Poisson 1e-13), FP32 2e-5 and 2e-4 for the potential.
"""
import numpy as np
import pytest

import synth
from _common import compare, gpu_for, oracle_for, step_both

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbeh():
    import paper_1712_08494_gb300 as pkg
    pkg.build()
    from paper_1712_08494_gb300 import lbeh as L
    return L


def _workload(box, ncomp, prec, spheres=()):
    nx, ny, nz = box
    rng = np.random.default_rng(nx * 10007 + ny * 101 + nz + ncomp)
    p = synth.Params(nx=nx, ny=ny, nz=nz, ncomp=ncomp, nions=2, prec=prec, G=4.0 if ncomp == 2 else 0.0,
                     eps_r=(1.0, 0.5) if ncomp == 2 else (1.0, 1.0), E_ext=(0.01, 0.0, 0.02),
                     poisson_tol=1e-13 if prec == "fp64" else 1e-9, poisson_max_iter=500, ncolloid_max=len(spheres))
    rho = rng.uniform(0.3, 0.4, size=(ncomp, nz, ny, nx))
    ions = rng.uniform(0.005, 0.015, size=(2, nz, ny, nx))
    if not spheres:
        return synth.Workload("box", p, rho, ions)
    x = np.array([s[:3] for s in spheres], dtype=float)
    return synth.Workload("spheres", p, rho, ions, x, np.zeros_like(x), np.full(len(spheres), -2.0),
                          np.array([s[3] for s in spheres], dtype=float))


@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("box", [(7, 5, 3), (8, 6, 10), (36, 20, 12)])
@pytest.mark.parametrize("ncomp", [1, 2])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_read_out(lbeh, prec, ncomp, box, where):
    import torch
    w = _workload(box, ncomp, prec)
    sg = gpu_for(w, lbeh)
    assert sg.step(2) in (lbeh.LBEH_OK, lbeh.LBEH_ERR_POISSON_NOT_CONVERGED)
    want = sg.get(("rho", "n", "phi", "u"), f=True)

    def read(f32):
        fl = lbeh.lbeh_fields()
        fl.dtype, fl.on_device = (lbeh.LBEH_F32 if f32 else lbeh.LBEH_F64), int(where == "device")
        dev = "cuda" if where == "device" else "cpu"
        out = {k: torch.full(want[k].shape, float("nan"), dtype=torch.float32 if f32 else torch.float64, device=dev)
               for k in ("rho", "n", "phi", "u")}
        for s in range(ncomp):
            fl.rho[s] = out["rho"][s].data_ptr()
        for s in range(2):
            fl.n[s] = out["n"][s].data_ptr()
        fl.phi, fl.u = out["phi"].data_ptr(), out["u"].data_ptr()
        torch.cuda.synchronize()
        assert lbeh.lbeh_get_fields(sg.h, fl) in (None, lbeh.LBEH_OK)
        torch.cuda.synchronize()
        return {k: v.cpu().numpy() for k, v in out.items()}

    d, s = read(False), read(True)
    for k in d:
        assert np.array_equal(d[k], want[k]), k
        if k == "phi" and prec != "fp64":
            assert np.all(np.abs(s[k] - want[k]) <= 2.0 ** -23 * np.abs(want[k]))
        else:
            assert np.array_equal(s[k], want[k].astype(np.float32)), k
    eps = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    bound = 20 * eps * (np.abs(want["f"]).sum(axis=1) + np.abs(want["rho"]))
    assert np.all(np.abs(want["f"].sum(axis=1) - want["rho"]) <= bound)
    sg.close()


SPHERES = {
    "none": (),
    "faces": ((0.4, 8.2, 8.1, 2.5), (8.3, 0.2, 15.7, 2.5)),        # across x; across an edge in y and z
    "corner_and_near": ((0.1, 0.2, 15.9, 2.5), (6.3, 0.2, 0.1, 2.5)),  # a corner; a gap of 1.2 between surfaces
}


@pytest.mark.parametrize("spheres", list(SPHERES))
@pytest.mark.parametrize("box", [(16, 16, 16), (18, 16, 16), (20, 16, 16)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_ion_update_and_sites_near_colloids(lbeh, prec, box, spheres):
    w = _workload(box, 2, prec, SPHERES[spheres])
    so, sg = oracle_for(w), gpu_for(w, lbeh)
    step_both(sg, so, 3)
    e = compare(sg, so, ("rho", "n", "phi"))
    lim = dict(rho=1e-11, n=1e-11, phi=1e-11) if prec == "fp64" else dict(rho=2e-5, n=2e-5, phi=2e-4)
    assert all(e[k] < lim[k] for k in e), e
    sg.close()
