"""The first iterate of every FP32 correction, tau_0 r / m_i, is the FP64 product
rounded once.

A mass solve of two steps keeps the correction's support small: of a right-hand
side that is non-zero at one node, the result at a neighbour is one rounded
multiple of the first iterate at that node, and with two corrections the result
three nodes away along the diagonal is one rounded multiple of the second
correction's first iterate two nodes away.  Both follow in float32 arithmetic
without any knowledge of the library's node order, on an unjittered grid whose
interior rows have entries 1/12 and lumped mass 1."""
import math

import numpy as np
import pytest

from paper_1708_04678_gb300 import felbm as F
from paper_1708_04678_gb300 import inputs as I

pytestmark = pytest.mark.gpu

f32 = np.float32


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04678_gb300 import build
    build.build()


# exponents of the values, side of a cell: values whose product is formed in two
# floats, as they are (-92 to 28) and scaled (-116 to -92); smaller ones (denormal
# floats or zero), larger ones, and meshes with tau_0 / m of 2^20 and, out of the
# range, 2^-20
@pytest.mark.parametrize("low,high,side", [(-40, 40, 1.0), (-112, -94, 1.0), (-160, -112, 1.0), (-260, -150, 1.0),
                                           (40, 100, 1.0), (-40, 40, 2.0 ** -10), (-200, -100, 2.0 ** -10),
                                           (-40, 40, 1024.0)])
@pytest.mark.parametrize("blocked", [True, False])
@pytest.mark.parametrize("rows", [18, 5])
@pytest.mark.parametrize("rounds", [1, 2])
def test_first_iterate_is_the_fp64_product_rounded_once(rounds, rows, blocked, low, high, side):
    nx, ny = 24, 16
    w = I.small_sessile(nx=nx, ny=ny, R=5.0, jitter=0.0)
    m = w["mesh"]
    mesh = dict(m, xy=m["xy"] * side, period=tuple(side * p for p in m["period"]))
    st = F.State(F.Mesh.from_dict(mesh), F.params_derive(w["phys"], solver_iters=2, solver_rounds=rounds), w["C0"])
    st.sweep_tiled(blocked)
    node = {(round(x), round(y)): k for k, (x, y) in enumerate(m["xy"])}
    tau = [1.0 / (0.625 + 0.375 * math.cos((2 * j + 1) * math.pi / 4)) for j in (0, 1)]
    lumped = side * side                                      # powers of two: every product with them is exact
    mass, v = lumped * (0.5 / 12 + 0.5 / 12), f32(lumped * (0.5 / 12 + 0.5 / 12))
    rng = np.random.default_rng(5)
    for rep in range(4):
        centres = [(4, 5), (10, 8), (16, 6), (22, 9)]
        val = rng.standard_normal((rows, len(centres))) * 2.0 ** rng.uniform(low, high, (rows, len(centres)))

        def step(x0):            # one step at a neighbour whose own iterate and right-hand side are zero
            return f32(f32(tau[1]) / f32(lumped)) * (-(v * x0))

        e0 = (val * (tau[0] / lumped)).astype(f32)
        for c, (x, y) in enumerate(centres):
            B = np.zeros((rows, len(m["xy"])))
            B[:, node[x, y]] = val[:, c]
            X = st.mass_solve(B)
            if rounds == 1:
                at, want = node[x + 1, y + 1], step(e0[:, c])
            else:
                rho = -(mass * step(e0[:, c]).astype(np.float64))
                at, want = node[(x + 3) % nx, y + 3], step((rho * (tau[0] / lumped)).astype(f32))
            np.testing.assert_array_equal(X[:, at], want.astype(np.float64))
            assert (want != 0).all() or low < -112
