"""Host paths of the library after a failure, on a CUDA runtime that has no
device (fake_cudart.cpp: memory of the host with a capacity, kernels that do
nothing, a status word that reads as a chosen failure).  Each test is a program
of its own, which loads that runtime in place of CUDA's."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
PRELUDE = """
import ctypes as C
import numpy as np
import synth
from paper_1712_08494_gb300 import lbeh
fake = C.CDLL("libcudart.so.13")
fake.fake_live.restype = C.c_size_t
fake.fake_capacity.argtypes = [C.c_size_t]
fake.fake_status.argtypes = [C.c_int, C.c_int]
ST_TIMEOUT = 4

def drop(n=8, prec="fp32"):
    w = synth.droplet(n=n, r=0.3 * n, prec=prec, Ez=0.01, charge=2.0)
    s = lbeh.System(w.params)
    s.set_fields(rho=list(w.rho), n=list(w.n))
    return s, w

def code(f, *a, **k):
    try:
        f(*a, **k)
    except lbeh.LbehError as e:
        return e.code
    return lbeh.LBEH_OK
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    inc = "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("g++ or the CUDA headers not found")
    import paper_1712_08494_gb300 as pkg
    try:
        pkg.build()
    except RuntimeError as e:
        pytest.skip(str(e))
    d = tmp_path_factory.mktemp("cudart")
    (d / "version").write_text("libcudart.so.13 { global: *; };\n")
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", inc, "-Wl,-soname,libcudart.so.13",
                    "-Wl,--version-script=%s" % (d / "version"), "-o", str(d / "libcudart.so.13"),
                    os.path.join(HERE, "fake_cudart.cpp")], check=True, capture_output=True)

    def run(body):
        env = dict(os.environ, LD_LIBRARY_PATH=str(d), PYTHONPATH=ROOT)
        r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(body)], env=env, cwd=ROOT, text=True,
                           capture_output=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr
    return run


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_adjoint_that_fails_gives_its_staging_back(program, prec):
    """A wait that runs out in the reverse sweep: the buffers of the host seeds
    serve the next call."""
    program("""
        s, w = drop(prec="%s")
        fbar = np.ones((2, 19) + w.rho.shape[1:])
        nbar = np.ones((2,) + w.rho.shape[1:])
        assert code(s.step_adjoint, 2, 1, f_bar=fbar, n_bar=nbar) == lbeh.LBEH_OK
        live = [fake.fake_live()]
        for _ in range(5):
            # two steps: their two words, the sweep's word, then the words of the reverse sweep
            fake.fake_status(4, ST_TIMEOUT)
            assert code(s.step_adjoint, 2, 1, f_bar=fbar, n_bar=nbar) == lbeh.LBEH_ERR_BARRIER_TIMEOUT
            assert s.observables().status == lbeh.LBEH_OK  # the forward sweep was fine
            live.append(fake.fake_live())
        assert len(set(live)) == 1, live
        s.close()
        assert fake.fake_live() == 0, fake.fake_live()
    """ % prec)


def test_idle_adjoint_memory_is_given_back(program):
    """The memory that a handle keeps after a gradient goes to another handle
    that finds no room, and comes back for the next gradient once there is."""
    program("""
        a, w = drop(n=16)
        before = fake.fake_live()
        assert code(a.step_adjoint, 6, 2) == lbeh.LBEH_OK
        kept = fake.fake_live() - before
        assert kept > 0
        b = lbeh.System(w.params)
        need = fake.fake_live() - kept - before  # of a second handle
        b.close()
        full = fake.fake_live() + need
        fake.fake_capacity(full - 1)  # one byte too few for the handle beside the block
        b = lbeh.System(w.params)
        assert need < fake.fake_live() < full
        assert code(a.step_adjoint, 6, 2) == lbeh.LBEH_ERR_OOM  # the handle in use keeps its own
        assert a.observables().steps == 6
        b.close()
        assert code(a.step_adjoint, 6, 2) == lbeh.LBEH_OK
        assert a.observables().steps == 12
        a.close()
        assert fake.fake_live() == 0
    """)
