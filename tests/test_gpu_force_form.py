"""Which kernels form the residuals and gather them in an FP32 step (one kernel
per node block, or one per triangle and one per node), seen by the launches
before the solve, and that both give the same bits.

A batch of equal members fills the device and takes the one kernel; a member run
alone does not and takes the two.  Both number a member's nodes and triangles
alike, so the member's state is the same bit for bit, walls and field update
included."""
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


def _rows13(nx, ny, seed):
    """2-triangle grid, every triangle split at its centroid: rows of up to 13 entries."""
    w = I.small_sessile(nx=nx, ny=ny, seed=seed, R=ny / 3.0, jitter=0.05)
    m = w["mesh"]
    xy, tri = m["xy"], m["tri"]
    p = xy[tri].copy()
    p[:, 1:, 0] -= nx * np.round((p[:, 1:, 0] - p[:, :1, 0]) / nx)
    c = len(xy) + np.arange(len(tri))
    new = np.concatenate([np.stack([tri[:, k], tri[:, (k + 1) % 3], c], 1) for k in range(3)])
    mesh = dict(m, xy=np.concatenate([xy, p.mean(1)]), tri=new.astype(np.int32))
    return {"mesh": mesh, "phys": dict(w["phys"], dt=0.02),
            "C0": I.droplet_C0(mesh["xy"], (nx / 2.0, 0.0), ny / 3.0, 4.0, mesh["period"])}


def _batch(ws):
    ids = 1 + max(int(w["mesh"]["wall_id"].max(initial=-1)) for w in ws)
    return {"meshes": [w["mesh"] for w in ws], "C0": np.concatenate([w["C0"] for w in ws]),
            "phys": dict(ws[0]["phys"], theta_deg=tuple(ws[0]["phys"]["theta_deg"])[:ids])}


def _state(w, **kw):
    mesh = F.Mesh.batch(w["meshes"]) if "meshes" in w else F.Mesh.from_dict(w["mesh"])
    st = F.State(mesh, F.params_derive(w["phys"], precision=F.FP32_DEV, **kw), w["C0"])
    st.timing_enable(True)
    return st


def _kernels(st):
    """Launches of a step before the solve: 3 with residuals and gather in one kernel, else 4."""
    t = st.timing_get()
    return t["launches"] - t["solve_launches"]


def _uneven():
    return _batch([I.small_sessile(nx=nx, ny=nx // 2, seed=100 + k, R=nx / 5.0)
                   for k, nx in enumerate(np.linspace(44, 88, 64).astype(int))])


@pytest.mark.parametrize("case,kernels", [("less than a wave", 4), ("one full wave", 3), ("one full wave, walls", 3),
                                          ("partial waves, walls", 4), ("partial waves", 4), ("full waves", 3)])
def test_kernels_of_the_forces(case, kernels):
    w = {"less than a wave": lambda: I.small_sessile(nx=256, ny=128, R=40.0),                # 128 blocks
         "one full wave": lambda: I.small_free_droplet(n=208, R=50.0),                       # 256 blocks
         "one full wave, walls": lambda: I.small_sessile(nx=8000, ny=15, R=6.0),             # 256 blocks
         "partial waves, walls": _uneven,                                                    # 392 blocks
         "partial waves": lambda: _batch([I.small_free_droplet(n=64, R=12.0, seed=50 + k) for k in range(20)]),
         "full waves": lambda: I.rough_wall_droplet(width=448, height=400, rows=397, R=90.0)}[case]()   # 512 blocks
    st = _state(w)
    st.step(2)
    assert _kernels(st) == kernels
    assert st.diagnostics()["status"] == 0


@pytest.mark.parametrize("iters", [0, 2])
@pytest.mark.parametrize("rows,count,member", [
    (7, 16, lambda k: I.small_sessile(nx=97, ny=48, seed=40 + k, R=18.0)),
    (9, 16, lambda k: I.small_free_droplet(n=56, R=11.0, seed=50 + k)),
    (13, 32, lambda k: _rows13(40, 26, 60 + k))])
def test_one_kernel_gives_the_bits_of_two(rows, count, member, iters):
    ws = [member(k) for k in range(count)]
    both = _state(_batch(ws), solver_iters=iters)
    both.step(4)
    assert _kernels(both) == 3
    g, h = both.get_state()
    at = 0
    for k, w in enumerate(ws):
        n = len(w["C0"])
        if k in (0, 1, count - 1):
            one = _state(dict(w, phys=_batch(ws)["phys"]), solver_iters=iters)
            one.step(4)
            assert _kernels(one) == 4
            g1, h1 = one.get_state()
            np.testing.assert_array_equal(g[:, at:at + n], g1)
            np.testing.assert_array_equal(h[:, at:at + n], h1)
        at += n
    assert np.isfinite(g).all() and np.abs(h).max() > 0
