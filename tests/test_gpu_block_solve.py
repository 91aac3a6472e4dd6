"""The blocked FP32 solve (several sweeps of a node block per launch) against
one launch per sweep: the same arithmetic per row in the same order, so the
states agree bit for bit."""
import numpy as np
import pytest

from paper_1708_04678_gb300 import felbm as F
from paper_1708_04678_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04678_gb300 import build
    build.build()


def _refined(nx, ny, both):
    """2-triangle grid with the upper (or every) triangle split at its centroid:
    rows of up to 10 (13) entries."""
    w = I.small_sessile(nx=nx, ny=ny, R=ny / 3.0, jitter=0.05)
    m = w["mesh"]
    xy, tri = m["xy"], m["tri"]
    pick = np.arange(len(tri)) if both else np.arange(1, len(tri), 2)
    p = xy[tri[pick]].copy()
    p[:, 1:, 0] -= nx * np.round((p[:, 1:, 0] - p[:, :1, 0]) / nx)
    c = len(xy) + np.arange(len(pick))
    t = tri[pick]
    new = np.concatenate([np.stack([t[:, k], t[:, (k + 1) % 3], c], 1) for k in range(3)])
    keep = np.setdiff1d(np.arange(len(tri)), pick)
    mesh = dict(m, xy=np.concatenate([xy, p.mean(1)]), tri=np.concatenate([tri[keep], new]).astype(np.int32))
    phys = dict(w["phys"], dt=0.02)
    C0 = I.droplet_C0(mesh["xy"], (nx / 2.0, 0.0), ny / 3.0, 4.0, mesh["period"])
    return {"mesh": mesh, "phys": phys, "C0": C0}


CASES = {
    "one block": lambda: I.small_sessile(nx=16, ny=8, R=4.0),                # 144 nodes
    "two blocks": lambda: I.small_sessile(nx=24, ny=21, R=6.0),              # 528 nodes: 264 each
    "full blocks": lambda: I.small_free_droplet(n=32, R=8.0),                # 2,048 nodes: 512 each, rows of 9
    "ragged": lambda: I.rough_wall_droplet(width=192, height=64, rows=49, R=20.0),
    "all planes per block": lambda: I.rough_wall_droplet(width=448, height=400, rows=397, R=90.0),
    "rows of 10": lambda: _refined(40, 24, False),
    "rows of 13": lambda: _refined(30, 20, True),                            # not blocked: both gathered
}


@pytest.mark.parametrize("case,precision,iters", [
    ("one block", F.FP32_DEV, 0), ("one block", F.FP64, 2), ("two blocks", F.FP32_DEV, 3), ("two blocks", F.FP64, 0),
    ("full blocks", F.FP32_DEV, 2), ("full blocks", F.FP64, 19), ("ragged", F.FP32_DEV, 30), ("ragged", F.FP64, 0),
    ("all planes per block", F.FP32_DEV, 0), ("all planes per block", F.FP64, 0), ("rows of 10", F.FP32_DEV, 0),
    ("rows of 10", F.FP64, 0), ("rows of 13", F.FP32_DEV, 0)])
def test_blocked_solve_gives_the_gathered_bits(case, precision, iters):
    w = CASES[case]()
    mesh = F.Mesh.from_dict(w["mesh"])
    params = F.params_derive(w["phys"], precision=precision, solver_iters=iters)
    a, b = (F.State(mesh, params, w["C0"]) for _ in range(2))
    a.sweep_tiled(False)
    if case == "rows of 13":
        assert mesh.info()["max_degree"] == 13
        with pytest.raises(F.FelbmError):
            b.sweep_tiled(True)
    a.step(4)
    b.step(4)
    for x, y in zip(a.get_state(), b.get_state()):
        np.testing.assert_array_equal(x, y)
    B = np.random.default_rng(3).standard_normal((5, len(w["C0"])))
    np.testing.assert_array_equal(a.mass_solve(B), b.mass_solve(B))
    for st in (a, b):
        st.solver_check(True, 1e3)
        st.step(2)
    da, db = a.diagnostics(), b.diagnostics()
    assert da["solver_residual"] == db["solver_residual"] > 0
    for x, y in zip(a.get_state(), b.get_state()):
        np.testing.assert_array_equal(x, y)
    assert np.isfinite(x).all() and np.abs(x).max() > 0


@pytest.mark.parametrize("case", ["all planes per block", "free 208", "rows of 13, large"])
def test_fused_forces_match_the_fp64_step(case):
    """Large FP32 states form the residuals and gather them in one kernel (rows of
    7, 9 and 13 entries): the step agrees with the FP64 state's to the FP32 level
    that the separate kernels are held to."""
    w = {"all planes per block": CASES["all planes per block"],
         "free 208": lambda: I.small_free_droplet(n=208, R=50.0),
         "rows of 13, large": lambda: _refined(220, 180, True)}[case]()
    mesh = F.Mesh.from_dict(w["mesh"])
    st = F.State(mesh, F.params_derive(w["phys"], precision=F.FP32_DEV), w["C0"])
    st.timing_enable(True)
    st.step(3)
    assert st.timing_get()["rhs_ms"] < 0.3 * st.timing_get()["element_ms"]     # the gather ran in the element kernel
    ref = F.State(mesh, F.params_derive(w["phys"]), w["C0"])
    ref.step(3)
    (g, h), (gr, hr) = st.get_state(), ref.get_state()
    assert np.abs(h - hr).max() < 1e-6 * np.abs(hr).max()
    assert np.abs(g - gr).max() < 1e-4 * np.abs(gr).max()


@pytest.mark.parametrize("precision", [F.FP64, F.FP32_DEV])
@pytest.mark.parametrize("case", ["two blocks", "all planes per block"])
def test_mass_solve_of_some_rows(case, precision):
    """The blocked solve takes only the planes that hold the requested rows: at
    every boundary of the planes the rows are those of the gathered solve of all."""
    w = CASES[case]()
    mesh, params = F.Mesh.from_dict(w["mesh"]), F.params_derive(w["phys"], precision=precision)
    a, b = (F.State(mesh, params, w["C0"]) for _ in range(2))
    a.sweep_tiled(False)
    B = np.random.default_rng(4).standard_normal((18, len(w["C0"])))
    X = a.mass_solve(B)
    for k in (18, 1, 2, 5, 6, 9, 10, 11, 14, 15):
        np.testing.assert_array_equal(b.mass_solve(B[:k]), X[:k])
