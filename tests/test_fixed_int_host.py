"""The integer arithmetic of the fixed-point FP64 kernels, built for the host
from the kernels' own header, against exact integers and rationals."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from .helpers import lobatto_derivative

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_1511_01561_gb300")


def _cuda_include():
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("fixed_int") / "fixed_int.so")
    cmd = ["g++", "-std=c++17", "-O1", "-fwrapv", "-ffp-contract=off", "-shared", "-fPIC", "-Wno-unknown-pragmas", "-I", HERE,
           "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(os.path.dirname(PKG), "include"), "-I", _cuda_include(),
           os.path.join(HERE, "fixed_int_host.cpp"), os.path.join(PKG, "csrc", "mesh.cpp"), "-o", lib, "-lpthread"]
    subprocess.run(cmd, check=True)
    fx = ctypes.CDLL(lib)
    fx.div_of.restype = ctypes.c_double
    fx.div_of.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_float]
    return fx


def _ints(n):
    return (ctypes.c_int * n)()


# values within 2^-31 below a power of two, where the diagonal momentum flux
# comes closest to its bound, and others around them
@pytest.mark.parametrize("pipe", [0, 1])
@pytest.mark.parametrize("N", range(1, 9))
def test_lines_of_extreme_fluxes(fx, N, pipe):
    """A uniform field's derivative is zero up to one unit a product, and the
    derivative of a field that changes sign along the line is D F: the sums of
    two mirrored nodes never leave 32 bits."""
    D = lobatto_derivative(N)
    e = int(np.frexp(float(max(sum(abs(v) for v in row) for row in D)))[1])
    rng = np.random.default_rng(N)
    near = lambda k: 2.0 ** k * (1.0 - 2.0 ** -rng.integers(31, 48))  # noqa: E731
    for trial in range(60):
        u = near(1)
        p = {0: near(2), 1: near(1), 2: near(3), 3: 0.0}.get(trial % 5, rng.uniform(0.0, 8.0))
        z = (ctypes.c_double * 8)(u, u, u, u, u, u, 300.0, p)
        f, g = _ints(24), _ints(3)
        assert fx.fluxes_of(z, pipe, f, g)
        for slot in range(12):
            lo, hi = f[2 * slot], f[2 * slot + 1]
            F = [lo + (hi << 29)] * (N + 1)
            if trial % 2:  # the antisymmetric combination
                F = [-v if m > N // 2 else v for m, v in enumerate(F)]
            h = [(v + (1 << 28)) >> 29 for v in F]
            arr = (ctypes.c_int * (2 * N + 2))(*[w for v, t in zip(F, h) for w in (v - (t << 29), t)])
            out = (ctypes.c_longlong * (N + 1))()
            fx.line_of(N, arr, e, out)
            for i in range(N + 1):
                want = sum(D[i][m] * F[m] for m in range(N + 1)) * Fraction(2) ** (2 - e)
                # a table entry and a dropped product of low parts, half a unit each, per node; the final rounding
                assert abs(out[i] - want) <= 2 * (N + 1) + 1, (trial, slot, i)


# a reciprocal seed anywhere within its documented error, densities on both
# sides of a power of two, where the exact reciprocal is an end of [1/2, 1)
@pytest.mark.parametrize("error", [-1.0, -0.5, 0.0, 0.5, 1.0])
@pytest.mark.parametrize("k", [-2, -1, 0, 3])
def test_division_next_to_powers_of_two(fx, k, error):
    rng = np.random.default_rng(k + 5)
    away = np.concatenate([np.ldexp(rng.uniform(0.5, 1.0, 200), -rng.integers(20, 53, 200)), [0.0, 2.0 ** -52, 2.0 ** -24]])
    for d in np.concatenate([away, -0.5 * away]):
        rho, x = float((1.0 + d) * 2.0 ** k), float(rng.uniform(1.0, 2.0))
        q = fx.div_of(x, rho, error)
        ulp = Fraction(float(np.spacing(q)))
        # half an ulp of rounding, and less than 1.5 of the 2^-57 carried, twice (reciprocal, product)
        assert abs(Fraction(q) - Fraction(x) / Fraction(rho)) <= Fraction(11, 16) * ulp, (d, q, x / rho)


# groups of zeros: exponents inside the range of the groups of other values, as
# the factor that a sum is multiplied by relies on
@pytest.mark.parametrize("pipe", [0, 1])
@pytest.mark.parametrize("U,u,th,p", [(0, 0, 300.0, 0), (0, 0, 300.0, 1e4), (0, 0, 0, 0), (2.0, 2.0, 0, 0), (3.0, 0, 1.0, 0)])
def test_groups_of_zeros(fx, pipe, U, u, th, p):
    f, e = _ints(24), _ints(3)
    assert fx.fluxes_of((ctypes.c_double * 8)(U, U, U, u, u, u, th, p), pipe, f, e)
    assert all(400 <= v <= 1600 for v in e), list(e)
    want = [U] * 3 + [U * u + p] * 3 + [U * u] * 3 + [U * th] * 3
    slots = [0, 5, 9, 1, 6, 10, 2, 3, 7, 4, 8, 11]
    for w, s, k in zip(want, slots, [0] * 3 + [1] * 6 + [2] * 3):
        assert (f[2 * s] + (f[2 * s + 1] << 29)) * Fraction(2) ** (e[k] - 1080) == Fraction(w)
