"""cotan_factor_info against the memory that the context counts for it: the stored factor and
update matrices are most of what the analysis allocates; beside them lie tables and solve
vectors, under 1,000 bytes a vertex (nine columns of two FP32 vectors, the supernodes' index
lists and update vectors)."""
import pytest

from synth import icosphere, torus

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,a,b", [("torus", 13, 7), ("torus", 200, 50), ("ico", 6, 0), ("ico", 7, 0)])
def test_stored_floats(lib, kind, a, b):
    V, F = icosphere(a) if kind == "ico" else torus(a, b, 1.0, 0.3)
    with lib.Context(0) as ctx:
        with lib.Mesh(V, F, ctx=ctx) as m:
            before = ctx.memory()[0]
            info = lib.cotan_factor_info(m)
            held = ctx.memory()[0] - before
    stored = 4 * (info["factor_floats"] + info["update_floats"])
    assert info["available"] == 1
    assert stored <= held <= stored + 1000 * len(V) + 65536, (stored, held)
