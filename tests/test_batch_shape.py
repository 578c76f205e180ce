"""The default launch shape of a batch (csrc/batch_shape.h) against measured times
of every portable shape (us a step, clusters of 1, 2, 4 and 8 blocks, of which
152, 76, 36 and 15 run at once): the estimate picks a shape within 5% of the
fastest.  The smallest cluster that gives two waves of blocks, the rule before,
is up to 3.3 times slower there."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

import synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_08494_gb300", "csrc")
BLOCKS, SLOTS = (1, 2, 4, 8), (152, 76, 36, 15)
MEASURED = {  # (boxes, edge, precision): time per shape
    (1, 16, "fp32"): (217.8, 171.9, 142.8, 129.4), (16, 16, "fp32"): (217.0, 172.5, 143.8, 254.7),
    (32, 16, "fp32"): (215.7, 169.9, 145.2, 384.0), (64, 16, "fp32"): (239.3, 193.4, 285.6, 639.2),
    (128, 16, "fp32"): (286.5, 404.6, 570.2, 1154.9), (300, 16, "fp32"): (582.1, 855.5, 1290.5, 2561.2),
    (600, 16, "fp32"): (1163.0, 1710.0, 2469.5, 5116.6), (10, 24, "fp32"): (557.1, 385.9, 288.9, 244.0),
    (20, 24, "fp32"): (584.6, 414.2, 313.1, 484.0), (64, 24, "fp32"): (665.6, 478.2, 700.4, 1317.1),
    (100, 24, "fp32"): (688.3, 922.8, 1053.9, 1825.2), (8, 32, "fp32"): (965.4, 602.6, 422.2, 306.1),
    (19, 32, "fp32"): (1075.0, 662.2, 461.0, 586.6), (76, 32, "fp32"): (1143.3, 746.6, 1350.4, 1883.2),
    (160, 32, "fp32"): (2284.1, 2089.1, 2403.5, 3545.9), (30, 48, "fp32"): (3319.6, 1894.9, 1176.6, 1458.2),
    (76, 48, "fp32"): (3769.4, 2308.9, 3525.5, 4206.7), (1, 64, "fp32"): (6249.3, 3349.6, 1842.5, 1042.3),
    (40, 64, "fp32"): (8191.2, 4457.6, 4659.7, 3787.8), (80, 64, "fp32"): (8994.7, 9042.4, 7340.3, 7623.1),
    (16, 16, "fp64"): (1412.9, 775.2, 460.9, 599.3), (40, 16, "fp64"): (1432.9, 797.2, 939.9, 902.9),
    (300, 16, "fp64"): (2878.8, 3203.1, 4287.7, 5983.2), (40, 32, "fp64"): (10512.2, 5378.3, 5601.6, 4354.2),
    (100, 32, "fp64"): (10632.6, 10777.7, 8419.1, 10130.6),
}
SOURCE = """
#include "batch_shape.h"
extern "C" double estimate(int nbox, long long cells, int blocks, int slots, int fp64) {
  return lbeh::batch_estimate(std::vector<long long>(nbox, cells), blocks, slots,
                              fp64 ? lbeh::kBatchLatencyF64 : lbeh::kBatchLatency);
}
"""


def _two_waves(nbox):
    for i, b in enumerate(BLOCKS):
        if b * nbox >= 2 * SLOTS[0]:
            return i
    return len(BLOCKS) - 1


def test_estimate_picks_a_fast_shape(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    (tmp_path / "s.cpp").write_text(SOURCE)
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(tmp_path / "s.so"),
                    str(tmp_path / "s.cpp")], check=True, capture_output=True)
    lib = C.CDLL(str(tmp_path / "s.so"))
    lib.estimate.argtypes = [C.c_int, C.c_longlong, C.c_int, C.c_int, C.c_int]
    lib.estimate.restype = C.c_double
    before = 0.0
    for (nbox, edge, prec), t in MEASURED.items():
        est = [lib.estimate(nbox, edge ** 3, b, s, int(prec == "fp64")) for b, s in zip(BLOCKS, SLOTS)]
        got = t[est.index(min(est))]
        assert got <= 1.05 * min(t), (nbox, edge, prec, est)
        before = max(before, t[_two_waves(nbox)] / min(t))
    assert before > 3.0


@pytest.mark.gpu
@pytest.mark.parametrize("nbox,shape", [(1, 8), (32, 4), (64, 2), (128, 1)])
def test_default_shape(lbeh, nbox, shape):
    p = synth.Params(nx=16, ny=16, nz=16, G=4.0, E_ext=(0.0, 0.0, 1e-3))
    b = lbeh.Batch([p] * nbox)
    assert b.shape() == shape
    b.close()
