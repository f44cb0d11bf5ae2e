"""Step sizes of the explicit B_perp solver's conjugate gradients (csrc/pcg_scalars.h), on the host."""
import ctypes as C
import math
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_10277_gb300", "csrc")
SHIM = """
#include "pcg_scalars.h"
extern "C" void scalars(int first, const double* v, int bits, double* out) {
  const hq::PcgScalars s = hq::pcg_scalars(first != 0, v[0], v[1], v[2], v[3], v[4], bits);
  out[0] = s.alpha;
  out[1] = s.beta;
  out[2] = s.pq;
}
"""


@pytest.fixture(scope="module")
def scalars(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("pcg")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run([gxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)

    def call(rz, zaz, paz=0.0, rz_prev=0.0, pq_prev=0.0, first=False, bits=13):
        v, out = (C.c_double * 5)(rz, zaz, paz, rz_prev, pq_prev), (C.c_double * 3)()
        lib.scalars(int(first), v, bits, out)
        return tuple(out)

    return call


def test_regular_steps(scalars):
    assert scalars(2.0, 5.0, first=True) == (0.4, 0.0, 5.0)
    # conjugate directions: p'.Az = -beta p'.Ap', so p.Ap = z.Az - beta^2 p'.Ap'
    assert scalars(1.0, 3.0, -2.0, 2.0, 4.0) == (0.5, 0.5, 2.0)
    # and any others: 3 + 2 0.5 1 + 0.25 4
    assert scalars(1.0, 3.0, 1.0, 2.0, 4.0) == (0.2, 0.5, 5.0)


@pytest.mark.parametrize("paz", [-2.5, -2.5 + 1e-9, -2.5 - 1e-9, -2.6, -2.5 + 5e-5])
def test_cancelled_terms_start_over(scalars, paz):
    """z.Az + 2 beta p'.Az + beta^2 p'.Ap' = 5 + 2 paz at or below the rounding of its terms (here 2^-13 of
    them), zero and negative included: the step along z alone, never one of the wrong sign or of the size
    of 1 over that rounding."""
    assert scalars(4.0, 4.0, paz, 4.0, 1.0) == (1.0, 0.0, 4.0)


def test_zero_denominators_and_nan(scalars):
    assert scalars(1.0, 0.0, first=True) == (0.0, 0.0, 0.0)
    assert scalars(0.0, 0.0, 0.0, 0.0, 0.0) == (0.0, 0.0, 0.0)
    assert scalars(3.0, 2.0, 1.0, 0.0, 7.0) == (1.5, 0.0, 2.0)
    nan = math.nan
    assert math.isnan(scalars(1.0, math.inf, -1.0, 1.0, -math.inf)[0])
    for v in ((nan, 1.0, 0.0, 1.0, 1.0), (1.0, nan, 0.0, 1.0, 1.0), (1.0, 1.0, nan, 1.0, 1.0), (1.0, 1.0, 0.0, nan, 1.0)):
        assert math.isnan(scalars(*v)[0])
        assert math.isnan(scalars(*(-x for x in v))[0])   # (the other sign of NaN)
    # an operator that is not positive keeps its negative steps
    assert scalars(1.0, -2.0, first=True) == (-0.5, 0.0, -2.0)
