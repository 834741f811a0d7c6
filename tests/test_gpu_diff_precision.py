"""How exact the FP32 differential at p = 6 is over the sizes it is used at: its error
against the FP64 pair sums of the same mesh, a mean over many noisy meshes, is held to
that of a kernel that kept every part of the sums in FP32 accumulators of its own,
measured on the same meshes (for each size: dE, then E). The bounds are 3% above for
dE, twice what two halves of the meshes differ by, and 20% above for E, whose errors
of both signs average less evenly."""
import numpy as np
import pytest

from synth import torus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,b,n,dE,E", [(20, 10, 64, 4.697e-7, 1.81e-8), (32, 8, 64, 4.350e-7, 2.19e-8),
                                        (41, 11, 64, 3.167e-7, 2.16e-8), (50, 13, 64, 2.404e-7, 1.73e-8),
                                        (64, 17, 48, 2.775e-7, 2.32e-8), (90, 23, 40, 3.201e-7, 3.98e-8),
                                        (110, 31, 32, 3.747e-7, 4.01e-8), (140, 36, 16, 3.620e-7, 2.89e-8)])
def test_error_of_the_differential(lib, a, b, n, dE, E):
    err = []
    for seed in range(n):
        V, F = torus(a, b, 1.0, 0.3)
        V = (V + 0.005 * np.random.default_rng(100 + seed).standard_normal(V.shape)).astype(np.float32).astype(float)
        with lib.Mesh(V, F) as m:
            g0, E0 = lib.tp_differential(m, lib.params(precision=lib.TP_PREC_FP64))
            g, E1 = lib.tp_differential(m, lib.params())
        err.append((np.linalg.norm(g - g0) / np.linalg.norm(g0), abs(E1 / E0 - 1)))
    m = np.mean(err, axis=0)
    assert m[0] <= 1.03 * dE and m[1] <= 1.2 * E, m
