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
    fx.value_of.restype, fx.value_of.argtypes = ctypes.c_longlong, [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    fx.div_of.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_float]
    return fx


def _ints(n):
    return (ctypes.c_int * n)()


def _fluxes(fx, z, scale, shared):
    """The staged fields as integers, and the exponents of U, the momentum equations and theta U."""
    f, e = _ints(30), _ints(5)
    assert fx.fluxes_of((ctypes.c_double * 8)(*z), (ctypes.c_int * 3)(*scale), shared, f, e)
    return [f[2 * k] + (f[2 * k + 1] << 29) for k in range(12 if shared else 15)], list(e)


# values within 2^-31 below a power of two, where the diagonal momentum flux
# comes closest to its bound, and others around them
@pytest.mark.parametrize("shared", [0, 1])
@pytest.mark.parametrize("N", range(1, 9))
def test_lines_of_extreme_fluxes(fx, N, shared):
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
        for slot, v in enumerate(_fluxes(fx, [u] * 6 + [300.0, p], (0, 0, 0), shared)[0]):
            F = [v] * (N + 1)
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


SHARED = [0, 5, 9, 1, 6, 10, 2, 3, 7, 4, 8, 11]  # slots of U_x..z, T_xx..zz, T_xy, xz, yz, H_x..z


# fluxes of components and scales of very different size, in units of their
# equation: U_c and u_v cut by less than a unit each, the product rounded without its
# low parts by less than one, p' cut by less than one
@pytest.mark.parametrize("seed", range(40))
def test_fluxes_of_scaled_directions(fx, seed):
    rng = np.random.default_rng(seed)
    s = [int(v) for v in rng.integers(0, 40, 3)]
    s[rng.integers(3)] = 0
    U, rho = rng.uniform(-1.0, 1.0, 3) * 2.0 ** rng.integers(-30, 30, 3), rng.uniform(0.1, 2.0)
    z = [*U, *(U / rho), rng.uniform(200.0, 400.0), rng.uniform(-1.0, 1.0) * 2.0 ** float(rng.integers(-30, 30))]
    u = [Fraction(v) for v in z[3:6]]
    U, th, p = [Fraction(v) for v in z[:3]], Fraction(z[6]), Fraction(z[7])
    unit = lambda E: Fraction(2) ** (E - 1080)  # noqa: E731
    f, e = _fluxes(fx, z, s, 0)
    for c in range(3):
        down = Fraction(1, 2 ** s[c])
        want = [U[c]] + [U[c] * u[v] + (p if v == c else 0) for v in range(3)] + [U[c] * th]
        for v in range(5):
            assert abs(f[5 * c + v] * unit(e[v]) - want[v] * down) < 4 * unit(e[v]), (c, v)
            assert abs(f[5 * c + v]) < 3 << 57
    f, e2 = _fluxes(fx, z, s, 1)
    assert e2 == e
    for c in range(3):
        down = Fraction(1, 2 ** s[c])
        for k, E, want in ((c, e[0], U[c]), (3 + c, e[1 + c], U[c] * u[c] + p), (9 + c, e[4], U[c] * th)):
            assert abs(f[SHARED[k]] * unit(E) - want * down) < 4 * unit(E)
    for k, (a, b) in enumerate(((0, 1), (0, 2), (1, 2))):
        # U_a u_b in the smaller of the two units, and shifted to the unit of the other equation
        pair = fx.pair_of((ctypes.c_int * 3)(*e[1:4]), (ctypes.c_int * 3)(*s), a, b)
        T = f[SHARED[6 + k]]
        assert abs(T) < 1 << 58
        for eq, along, second in ((a, b, 0), (b, a, 1)):
            x, one = fx.value_of(T, pair, second), unit(e[1 + eq])
            # (u is rounded: the one product or the other stands for both)
            assert min(abs(x * one - t / 2 ** s[along]) for t in (U[a] * u[b], U[b] * u[a])) < 4 * one, (a, b, eq)


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
@pytest.mark.parametrize("shared", [0, 1])
@pytest.mark.parametrize("U,u,th,p", [(0, 0, 300.0, 0), (0, 0, 300.0, 1e4), (0, 0, 0, 0), (2.0, 2.0, 0, 0), (3.0, 0, 1.0, 0)])
def test_groups_of_zeros(fx, shared, U, u, th, p):
    f, e = _fluxes(fx, [U] * 3 + [u] * 3 + [th, p], (0, 0, 0), shared)
    assert all(400 <= v <= 1600 for v in e), e
    for c in range(3):
        for v in range(5):
            k = 5 * c + v if not shared else SHARED[c if v == 0 else 9 + c if v == 4 else 3 + c if v == c + 1 else 5 + c + v - 1]
            want = U if v == 0 else U * th if v == 4 else U * u + (p if v == c + 1 else 0)
            assert f[k] * Fraction(2) ** (e[v] - 1080) == Fraction(want)
