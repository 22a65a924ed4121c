"""Per-cell functions of the CUDA headers, compiled for the host (device_host/) and held against
extended-precision sums."""
import ctypes
import os
import subprocess

import pytest

from paper_2508_06911_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("device_host") / "checks.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.NVCC)), "include")
    src = os.path.join(HERE, "device_host", "checks.cpp")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-w", "-ffp-contract=off", "-shared", "-fPIC", "-I", cuda, "-I",
                        build.CSRC, src, "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def call(f, *args, n_out):
    out = (ctypes.c_double * n_out)()
    f(*[ctypes.c_double(a) if isinstance(a, float) else ctypes.c_int(a) for a in args], out)
    return list(out)


# The residual that the mixed path judges is that of the deposit.  Streaming from kept populations sums
# the change of the residual in FP32, off by up to 5.5 2^-24 of sums of at most 3e-6, of which the judge
# adds three fifths to what it finds: 0.45 of the default tolerance are left.  A smaller tolerance
# has to be judged by a fresh sum.
# 5e-14: the double-float floor of that sum (2^-48 of sums of |X|^3 f times 1 / sqrt(RT)^3).
@pytest.mark.parametrize("tol", [1e-12, 1e-13])
@pytest.mark.parametrize("fluon", [1, 0])
@pytest.mark.parametrize("RT", [0.22, 0.6, 4.0, 9.0])
def test_judged_residual_is_that_of_the_deposit(lib, RT, fluon, tol):
    some_kept = 0
    for noise in (3e-9, 1e-8, 3e-8, 6e-8, 1e-7):
        cells, worst, kept, _ = call(lib.check_judged, fluon, RT, noise, tol, 400, 5, n_out=4)
        assert cells > 100
        assert worst <= (1.45 if tol >= 1e-12 else 1.0) * tol + 5e-14, f"noise {noise}: {worst:.2e}"
        some_kept += kept
    assert (some_kept > 0) == (tol >= 1e-12)


# A phonon deposit that a failed fluon solve takes back leaves the rounding of the additions only: at most
# two times twenty additions to a cell, half an ulp each.  Also where the updated multipliers are out of
# the range of the pass that evaluates them, while the kept populations were streamed.
@pytest.mark.parametrize("edge", [0, 1])
@pytest.mark.parametrize("RT", [0.22, 0.6, 4.0])
def test_phonon_take_back(lib, RT, edge):
    cells, left, kept, at_edge = call(lib.check_take_back, RT, 3e-7, edge, 1500 if edge else 300, 6, n_out=4)
    assert cells > 50 and kept > 30 and (not edge or at_edge > 50)
    assert left <= 40 * 2.0 ** -53


# The lattice form's populations are no further off, weighted by the population, than the general stencil's,
# which starts every row from exponentials of its own: within a fifth and two roundings (2^-52).
@pytest.mark.parametrize("RT", [0.2, 0.35, 0.6, 1.5, 4.2, 8.0, 9.4, 10.2, 13.0, 16.0, 25.0, 32.0])
@pytest.mark.parametrize("D", [1, 2])
def test_lattice_form_populations(lib, D, RT):
    mean, _, mean_rows, _ = call(lib.check_populations, D, RT, 30 if D == 2 else 200, 7, n_out=4)
    assert 0 < mean <= 1.2 * mean_rows + 2.0 ** -52


# The scratch of the kept populations has a column for every thread of a mixed launch: a persistent batch of
# tubes however short (four blocks of 128 threads an SM, no more than tubes) and a cell update of one block an SM.
@pytest.mark.parametrize("n_inst,per_tube", [(1, 400), (7, 30), (700, 12), (760, 12), (4096, 12), (4096, 3000)])
def test_scratch_of_kept_populations_1d(lib, n_inst, per_tube, sms=152):
    f = lib.check_pop_threads
    f.restype = ctypes.c_longlong
    ncell = n_inst * per_tube
    got = f(1, ctypes.c_longlong(ncell), n_inst, sms)
    batch = min(n_inst, 4 * sms) * 128
    cells = min(ncell + 384, sms * 384)
    assert max(batch, min(cells, ncell)) <= got <= sms * 512


@pytest.mark.parametrize("ncell", [1, 1000, 60000, 399999, 400000, 1 << 24])
def test_scratch_of_kept_populations_2d(lib, ncell, sms=152):
    f = lib.check_pop_threads
    f.restype = ctypes.c_longlong
    block = 384 if ncell < 400000 else 512
    got = f(2, ctypes.c_longlong(ncell), 1, sms)
    assert min(ncell + block - 1, sms * block) <= got <= sms * block


# The exponential by integer instructions carries at least 59 bits and rounds once: half an ulp, a sixth for the
# terms left out and cut off.  A reciprocal within one ulp, a quotient too; conversions and quarters exact.
def test_integer_and_short_arithmetic(lib):
    e, recip, quot, bad_narrow, bad_widen, bad_quarter = call(lib.check_arithmetic, 400000, 8, n_out=6)
    assert e <= 2.0 / 3.0
    assert recip <= 1.0 and quot <= 1.0
    assert bad_narrow == bad_widen == bad_quarter == 0
