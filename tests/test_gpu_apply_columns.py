"""The FP32 all-pairs applies in passes of three, six and nine columns (equal runs of
256 x 128 units, partial sums in the slots of the blocks that share a row of targets) at
the sizes where the split changes - part of a tile, edges of tiles (128) and of target
rows (256), an odd number of tiles - and at the column counts that pad a pass,
against the oracle. FP32 pair terms carry a few 2^-24 each and the sums are compensated:
the parity tolerance of the FP32 path, 1e-5, holds."""
import numpy as np
import pytest

from oracle import tp_oracle as O
from synth import small_mesh

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.mark.parametrize("mesh", ["torus4x4", "torus16x4", "torus13x5", "torus43x3", "torus37x7", "torus48x32"])
@pytest.mark.parametrize("op", ["A", "B", "B0", "L"])
def test_sizes_and_columns(lib, mesh, op):
    V, F = small_mesh(mesh, seed=3)
    X = np.random.default_rng(5).standard_normal((len(V), 9))
    Y = O.apply_operator(V, F, X, op)
    with lib.Mesh(V, F) as m:
        for k in (1, 2, 3, 4, 6, 7, 9):
            y = lib.fractional_apply(m, op, np.ascontiguousarray(X[:, :k]), lib.params())
            assert np.linalg.norm(y - Y[:, :k]) <= TOL * np.linalg.norm(Y[:, :k]), k
