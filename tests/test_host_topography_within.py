"""The kernel's per-node topography check (products and integer comparisons) decides as the
deviation's quotients do, on the CPU: over the oracle's metrics of topography and other maps at
bounds on both sides of their deviations, and for zeros, infinities, NaN and negative ratios."""
import ctypes

import numpy as np
import pytest

from oracle.metrics import metrics
from workloads.geometry import make_map, node_coordinates

from host_build import build


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    L = ctypes.CDLL(build("host_topo_within.cpp", tmp_path_factory.mktemp("within") / "libwithin.so", shared=True))
    L.host_topography_within.argtypes = [ctypes.c_void_p] + [ctypes.c_int] * 3 + [ctypes.c_double] * 2 + [
        ctypes.c_void_p] * 2
    return L


def _check(lib, jm, c, tol):
    far, differ = ctypes.c_longlong(), ctypes.c_longlong()
    ns, nr, nq = jm.shape[1:]
    lib.host_topography_within(jm.ctypes.data, nq, nr, ns, c, tol, ctypes.byref(far), ctypes.byref(differ))
    return far.value, differ.value


@pytest.mark.parametrize("name,extent,nodes", [("gaussian_hill", (30000.0, 20000.0, 15000.0), (21, 19, 17)),
                                               ("curvy", (1000.0, 1100.0, 900.0), (21, 19, 17))])
@pytest.mark.parametrize("tol", [1e-17, 1e-14, 1e-11, 1e-3, 1.0])
def test_decides_as_the_deviation_does(lib, name, extent, nodes, tol):
    X = node_coordinates(make_map(name, extent), nodes)
    J, a = metrics(*X, 6)
    jm = np.ascontiguousarray(np.stack([J] + [a[xi][eta] for xi in range(3) for eta in range(3)]))
    c = jm[5].flat[0] / jm[1].flat[0]
    far, differ = _check(lib, jm, c, tol)
    assert differ == 0
    assert (far == 0) == (name != "curvy" and tol >= 1e-11) or tol in (1e-14, 1.0)


@pytest.mark.parametrize("field", range(1, 7))
@pytest.mark.parametrize("value", [0.0, -0.0, np.inf, -np.inf, np.nan, 1e-320, -3.0, 1e308])
def test_special_values(lib, field, value):
    jm = np.zeros((10, 1, 1, 2))
    jm[1], jm[5] = 2.0, 3.0
    jm[field, 0, 0, 1] = value
    assert _check(lib, jm, 1.5, 1e-11)[1] == 0
