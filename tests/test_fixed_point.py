"""The fixed-point arithmetic of the FP64 kernels, built for the host: its
conversions, reciprocal and two-point flux against long double.

Bars: a conversion to fixed point truncates to one unit of 2^-60; back to
FP64 it rounds to nearest (2^-53, and 2^-32 units, of the 96-bit
sums' last word); the reciprocal is good to 2^-55; the flux stays below 2^60.5, so
that the sums with a row of D cannot overflow; its error and that of a lifted
gradient are no larger than those of the same formula in FP64 over the admitted
range of the states and of the metric terms.  The directions of an element share
an exponent: one that is 2^t smaller is shifted up by t where it is used (the
kernels take t up to 1), and one that is smaller by less than 2 is not shifted
(loose 1.99; then the energy flux at Mach 30 is the one quantity above FP64's
error, by less than a factor 2)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fx") / "fixed_point_check.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fwrapv", "-shared", "-fPIC", "-o", so,
                           os.path.join(HERE, "fixed_point_check.cpp")])
    L = C.CDLL(so)
    L.check_rcp.restype = C.c_double
    L.check_pairs.argtypes = [C.c_int] + [C.c_double] * 6 + [C.c_int, C.c_double, C.c_int, C.c_double, C.c_void_p]
    L.check_lifting.argtypes = [C.c_int, C.c_int, C.c_void_p, C.c_int, C.c_double, C.c_int, C.c_void_p]
    L.check_pair_vjp.argtypes = [C.c_int] + [C.c_double] * 6 + [C.c_int, C.c_double, C.c_int] + [C.c_double] * 3 + \
        [C.c_int, C.c_void_p]
    return L


def test_conversions(lib):
    out = np.zeros(3)
    lib.check_conversions(200000, out.ctypes.data_as(C.c_void_p))
    assert out[0] < 1.0 and out[1] <= 2.0 ** -53 and out[2] <= 2.0 ** -52.9, out


def test_reciprocal(lib):
    assert lib.check_rcp(200000) < 2.0 ** -55


# density, pressure, velocity, metric terms, one-component metrics, gamma:
# random states of the parity tests, low Mach numbers, the density wave, Mach 2
# and 30, densities over the whole admitted range, gamma near 1 and large
STATES = [
    (0.8, 1.2, 0.8, 1.2, 0.5, 1.0, 0, 1.4),
    (0.99, 1.01, 71.0, 72.0, 1.0, 0.01, 1, 1.4),
    (0.9999, 1.0001, 714285.0, 714286.0, 1.0, 0.3, 0, 1.4),
    (1.9, 2.1, 1.0, 1.001, 1.01, 0.004, 0, 1.4),
    (0.5, 1.5, 0.8, 2.0, 3.0, 1.0, 1, 1.4),
    (1.0, 1.1, 0.9, 1.0, 35.0, 2e-9, 0, 1.4),
    (1.0, 7.9, 1.0, 6.0, 1.0, 1.0, 1, 1.4),
    (0.126, 1.0, 0.1, 1.0, 0.3, 50.0, 0, 1.4),
    (1e-7, 1.2e-7, 1e20, 1.1e20, 1e13, 1e6, 1, 1.05),
    (0.8, 1.2, 0.8, 1.2, 0.5, 1.0, 1, 3.0),
]


@pytest.mark.parametrize("r0,r1,p0,p1,um,jm,axis,gamma", STATES)
@pytest.mark.parametrize("shift,loose", [(0, 1.0), (4, 1.0), (0, 1.99)])
def test_two_point_flux(lib, r0, r1, p0, p1, um, jm, axis, gamma, shift, loose):
    out = np.zeros(8)
    n = 20000
    lib.check_pairs(n, r0, r1, p0, p1, um, jm, axis, gamma, shift, loose, out.ctypes.data_as(C.c_void_p))
    fixed, fp64 = out[:3], out[3:6]
    if loose > 1.0 and um > 30.0:
        fp64[2] *= 2.0
    assert out[7] < 0.8 * n
    assert out[6] < 60.5, out[6]
    assert (fixed <= fp64).all(), (fixed, fp64)


@pytest.mark.parametrize("N", range(1, 10))
@pytest.mark.parametrize("shift", [0, 2, 4])
def test_lifted_gradient(lib, orc, N, shift):
    x, w, D = orc.basis(N)
    out = np.zeros(2)
    e_D = (0, 2, 3, 3, 4, 4, 5, 5, 5)[N - 1]
    lib.check_lifting(4000, N + 1, D.ctypes.data_as(C.c_void_p), e_D, 0.5 / w[0], shift, out.ctypes.data_as(C.c_void_p))
    assert out[0] <= out[1], out


@pytest.mark.parametrize("r0,r1,p0,p1,um,jm,axis,gamma", STATES)
@pytest.mark.parametrize("cotangent", [(1.0, 1.0, 1.0), (1e-6, 1.0, 1e6), (1e8, 1.0, 1e-8), (1.0, 0.0, 0.0),
                                       (0.0, 0.0, 1.0), (1e-45, 1e-44, 1e-45)])
@pytest.mark.parametrize("shift,e_D", [(0, 5), (4, 0)])
def test_two_point_flux_adjoint(lib, r0, r1, p0, p1, um, jm, axis, gamma, cotangent, shift, e_D):
    """Adjoint of the two-point flux for densities, beta, velocity and |u|^2: errors
    over the terms' size no larger than FP64's; no share above the exponent of its
    sum, whose 27 terms (N = 9) stay below 2^63; mantissas below 2^60."""
    out = np.zeros(12)
    n = 3000
    lib.check_pair_vjp(n, r0, r1, p0, p1, um, jm, axis, gamma, shift, *cotangent, e_D, out.ctypes.data_as(C.c_void_p))
    assert out[11] < 0.8 * n
    assert out[8] >= 0 and out[9] < 63 - np.log2(27) and out[10] <= 60.0, out[8:]
    fixed, fp64 = out[:4], out[4:8]
    some = ~np.isnan(fp64)      # no adjoint of beta and |u|^2 from the mass equation alone
    assert some[0] and some[2] and (fixed[some] <= fp64[some]).all(), (fixed, fp64)
