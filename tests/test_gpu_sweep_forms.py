"""Every split of a node's right-hand sides over threads in the gathered solve
steps (1, 2, 3 or 6 threads a node) gives the same bits, with the blocked form
switched off on both sides, for every width of the matrix rows, in both storages,
with the first iterate formed inside the first step (FP32) and before it; and the
blocked form gives those bits too."""
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
    c, t = len(xy) + np.arange(len(pick)), tri[pick]
    new = np.concatenate([np.stack([t[:, k], t[:, (k + 1) % 3], c], 1) for k in range(3)])
    keep = np.setdiff1d(np.arange(len(tri)), pick)
    mesh = dict(m, xy=np.concatenate([xy, p.mean(1)]), tri=np.concatenate([tri[keep], new]).astype(np.int32))
    return {"mesh": mesh, "phys": dict(w["phys"], dt=0.02),
            "C0": I.droplet_C0(mesh["xy"], (nx / 2.0, 0.0), ny / 3.0, 4.0, mesh["period"])}


ROWS = {7: lambda: I.small_sessile(nx=43, ny=21, R=9.0, theta=60.0), 9: lambda: I.small_free_droplet(n=41, R=9.0, seed=5),
        10: lambda: _refined(40, 24, False), 13: lambda: _refined(30, 20, True)}


def _run(w, parts, blocked, **kw):
    st = F.State(F.Mesh.from_dict(w["mesh"]), F.params_derive(w["phys"], **kw), w["C0"])
    st.sweep_parts(parts)
    st.sweep_tiled(blocked)
    st.timing_enable(True)
    st.step(6)
    launches = st.timing_get()["solve_launches"]
    st.timing_enable(False)
    st.step(6)                       # without events between the kernels: dependent launches
    return launches, st.get_state()


@pytest.mark.parametrize("precision,iters", [(F.FP32_DEV, 0), (F.FP32_DEV, 2), (F.FP64, 0)])
@pytest.mark.parametrize("rows", ROWS)
def test_gathered_splits_and_the_blocked_form_give_the_same_bits(rows, precision, iters):
    w = ROWS[rows]()
    assert F.Mesh.from_dict(w["mesh"]).info()["max_degree"] == rows
    kw = dict(precision=precision, solver_iters=iters)
    gathered, ref = _run(w, 2, False, **kw)
    assert gathered == ((iters or 10) - 1 if precision == F.FP32_DEV else 3 * 13 + 2)
    for parts in (1, 3, 6):
        n, got = _run(w, parts, False, **kw)
        assert n == gathered
        for x, y in zip(got, ref):
            np.testing.assert_array_equal(x, y)
    if rows <= 12:
        n, got = _run(w, 2, True, **kw)
        assert n != gathered
        for x, y in zip(got, ref):
            np.testing.assert_array_equal(x, y)
    assert np.isfinite(ref[0]).all() and np.abs(ref[1]).max() > 0
