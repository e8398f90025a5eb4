"""The impedances of the face penalties, FP32, on the CPU (tests/host_penalty.cpp).

With the normal along x and unit factors the penalty of a unit velocity is Z itself and that of a unit
traction 1/Z, so that they can be read off: Z = sqrt(c / r), c = lambda/J + 2 mu/J or mu/J, r = 1/(rho J).
u = 2^-24.  Z_s: the quotient's u, halved by the root, and the root's u: 1.5 u; Z_p: the sum's u besides:
2 u; the reciprocals one u more.  1.001 for the terms of second order."""
import ctypes

import numpy as np
import pytest

from host_build import build

U = 2.0 ** -24


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    L = ctypes.CDLL(build("host_penalty.cpp", tmp_path_factory.mktemp("pen") / "libpen.so", shared=True))
    P = ctypes.c_void_p
    L.host_penalty.argtypes = [ctypes.c_int, ctypes.c_float, P, P, P, ctypes.c_int, P]
    return L


def _coefficients(n=20000, seed=3):
    g = np.random.default_rng(seed)
    J = 10.0 ** g.uniform(3, 14, n)
    rho, lam, mu = g.uniform(1000, 3500, n), g.uniform(-1e9, 5e10, n), g.uniform(1e9, 5e10, n)
    return np.ascontiguousarray(np.stack([1 / (rho * J), lam / J, mu / J], 1).astype(np.float32))


def _exact(mat):
    r, lam, mu = (mat[:, c].astype(np.float64) for c in range(3))
    return np.sqrt((lam + 2 * mu) / r), np.sqrt(mu / r)


def _penalty(lib, side, gamma, v, s, mat):
    out = np.empty((len(mat), 9), np.float32)
    v, s = np.array(v, np.float32), np.array(s, np.float32)
    lib.host_penalty(side, gamma, v.ctypes.data, s.ctypes.data, mat.ctypes.data, len(mat), out.ctypes.data)
    return np.abs(out.astype(np.float64))


@pytest.mark.parametrize("side", [0, 1])
def test_impedances_of_the_characteristic_penalty(lib, side):
    mat = _coefficients()
    Zp, Zs = _exact(mat)
    for got, want, bound in (
            (_penalty(lib, side, -1.0, [1, 0, 0], [0] * 6, mat)[:, 0], Zp, 2.0),
            (_penalty(lib, side, -1.0, [0, 1, 0], [0] * 6, mat)[:, 1], Zs, 1.5),
            (_penalty(lib, side, 1.0, [0] * 3, [1, 0, 0, 0, 0, 0], mat)[:, 3], 1 / Zp, 3.0),
            (_penalty(lib, side, 1.0, [0] * 3, [0, 0, 0, 1, 0, 0], mat)[:, 6], 1 / Zs, 2.5)):
        assert (np.abs(got / want - 1)).max() <= 1.001 * bound * U
