"""Device buffers that a copy reaches but a kernel's stores of whole elements do
not: an FP64 buffer that starts off its natural alignment.  The results are the
bytes that the aligned buffer gets."""
import numpy as np
import pytest

import synth
from _common import gpu_for

pytestmark = pytest.mark.gpu


def _drop(prec):
    return synth.droplet(n=16, r=5.0, prec=prec, Ez=0.01, charge=2.0, salt=1e-3)


def _off_aligned(torch, count, off):
    """A device buffer for count FP64 values that starts `off` bytes past an aligned address."""
    raw = torch.full((8 * count + 8,), 0xA5, dtype=torch.uint8, device="cuda")
    return raw, raw.data_ptr() + off


def _values(raw, off, count):
    return np.frombuffer(raw.cpu().numpy().tobytes()[off:off + 8 * count], dtype=np.float64)


@pytest.mark.parametrize("off", [0, 4])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_fields(lbeh, prec, off):
    import torch
    w = _drop(prec)
    s = gpu_for(w, lbeh)
    assert s.step(2) == lbeh.LBEH_OK
    want = s.get(("rho", "n", "phi", "u"), f=True)
    N = w.rho[0].size
    fl = lbeh.lbeh_fields()
    fl.dtype, fl.on_device = lbeh.LBEH_F64, 1
    bufs = {}
    for name, count in (("rho0", N), ("rho1", N), ("n0", N), ("n1", N), ("phi", N), ("u", 3 * N), ("f", 38 * N)):
        raw, ptr = _off_aligned(torch, count, off)
        bufs[name] = (raw, count)
        if name[-1] in "01":
            getattr(fl, name[:-1])[int(name[-1])] = ptr
        else:
            setattr(fl, name, ptr)
    torch.cuda.synchronize()
    lbeh.lbeh_get_fields(s.h, fl)
    ref = {"rho0": want["rho"][0], "rho1": want["rho"][1], "n0": want["n"][0], "n1": want["n"][1],
           "phi": want["phi"], "u": want["u"], "f": want["f"]}
    for name, (raw, count) in bufs.items():
        assert np.array_equal(_values(raw, off, count), np.ravel(ref[name])), name
        assert int(raw[8 * count + off:].ne(0xA5).sum()) == 0 and int(raw[:off].ne(0xA5).sum()) == 0, name
    s.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_adjoint_state(lbeh, prec):
    import torch
    w = _drop(prec)
    N, got = w.rho[0].size, {}
    for off in (0, 4):
        s = gpu_for(w, lbeh)
        seed, g = lbeh.lbeh_obs_seed(), lbeh.lbeh_grads()
        seed.d_deformation = 1.0
        (f, fp), (n, np_) = _off_aligned(torch, 38 * N, off), _off_aligned(torch, 2 * N, off)
        g.f0_bar, g.n0_bar, g.on_device = fp, np_, 1
        torch.cuda.synchronize()
        lbeh.lbeh_step_adjoint(s.h, 3, 2, seed, g)
        got[off] = _values(f, off, 38 * N), _values(n, off, 2 * N)
        s.close()
    assert np.array_equal(got[0][0], got[4][0]) and np.array_equal(got[0][1], got[4][1])
    assert np.abs(got[0][0]).max() > 0
