"""The FP32 energy and differential at p = 6 around the switch to four targets a
thread, which the energy takes from 25 tiles of 128 faces on (148 to 152 SMs): last
rows of target tiles that hold one, two, three and four tiles, whole and ragged, and
the switch of the differential's FP32 sums at 8,192 faces, against the oracle at the
FP32 path's parity tolerance, 1e-5."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import small_mesh

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.mark.parametrize("a,b", [(64, 24), (64, 25), (51, 32), (64, 26), (69, 25), (53, 33), (64, 28), (59, 31),
                                 (128, 32), (91, 46)])
def test_sizes(lib, a, b):
    # tiles: 24, 25, 26 (ragged), 26, 27 (ragged), 28 (ragged), 28, 29 (ragged); 64 and 66 (ragged)
    V, F = small_mesh(f"torus{a}x{b}", seed=a)
    with lib.Mesh(V, F) as m:
        p = lib.params()
        E, (g, E2) = lib.tp_energy(m, p), lib.tp_differential(m, p)
    E0, g0 = O.energy(V, F), O.differential(V, F)
    assert abs(E / E0 - 1) <= TOL and abs(E2 / E0 - 1) <= TOL
    assert np.linalg.norm(g - g0) <= TOL * np.linalg.norm(g0)
