"""The per-member batch schedule (one thread block advances a member) on every
kind of matrix row: ELL rows of 7, 9 and 13 entries and CSR rows of 25, members
of fewer nodes than the block has threads and of several times as many.

The schedule runs the all-launch schedule's arithmetic on the same tables except
for the chemical potential, whose FP64 sum is ordered differently before it is
rounded to FP32; the bound is the one of the schedule test on rows of 7."""
import numpy as np
import pytest

from paper_1708_04678_gb300 import felbm as F
from paper_1708_04678_gb300 import inputs as I
from parity_util import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04678_gb300 import build
    build.build()


def _refined(nx, ny, seed, times):
    """2-triangle grid, every triangle split at its centroid `times` times: rows of
    up to 7, 13, 25 entries."""
    w = I.small_sessile(nx=nx, ny=ny, seed=seed, R=ny / 2.5, jitter=0.05)
    m = w["mesh"]
    xy, tri = m["xy"], m["tri"]
    for _ in range(times):
        p = xy[tri].copy()
        p[:, 1:, 0] -= nx * np.round((p[:, 1:, 0] - p[:, :1, 0]) / nx)
        c = len(xy) + np.arange(len(tri))
        tri = np.concatenate([np.stack([tri[:, k], tri[:, (k + 1) % 3], c], 1) for k in range(3)]).astype(np.int32)
        xy = np.concatenate([xy, p.mean(1)])
    mesh = dict(m, xy=xy, tri=tri)
    phys = dict(w["phys"], dt=(0.1, 0.02, 0.004)[times])
    return mesh, I.droplet_C0(xy, (nx / 2.0, 0.0), ny / 2.5, 4.0, mesh["period"]), phys


@pytest.mark.parametrize("rows", [7, 9, 13, 25])
def test_per_member_schedule_follows_the_launches(rows):
    if rows == 9:
        ws = [I.small_free_droplet(n=n, R=n / 4.0, seed=n) for n in (14, 21, 30)]
        members = [(w["mesh"], w["C0"], w["phys"]) for w in ws]
    else:
        times = {7: 0, 13: 1, 25: 2}[rows]
        members = [_refined(nx, ny, 30 + nx, times) for nx, ny in {7: ((24, 12), (50, 31)), 13: ((16, 12), (30, 20)),
                                                                   25: ((12, 10), (20, 14))}[rows]]
    mesh = F.Mesh.batch([m[0] for m in members])
    assert mesh.info()["max_degree"] == rows
    C0 = np.concatenate([m[1] for m in members])
    phys = dict(members[0][2])
    ids = 1 + max(int(m[0]["wall_id"].max(initial=-1)) for m in members)
    phys["theta_deg"] = (80.0,) * ids
    params = F.params_derive(phys, precision=F.FP32_DEV)
    a, b = (F.State(mesh, params, C0) for _ in range(2))
    b.batch_schedule(10 ** 6)
    a.step(20)
    b.step(20)
    for x, y in zip(b.get_state(), a.get_state()):
        assert np.isfinite(x).all() and rel_err(x, y) < 1e-6
