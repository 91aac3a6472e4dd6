"""A batch whose small members have a thread block of their own: the launches of a
step cover the other members, so their number and their forms follow those
members alone, and those members keep the bits of a run of their own."""
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


def _state(ws, **kw):
    ids = len(ws[0]["phys"]["theta_deg"])
    mesh = F.Mesh.batch([w["mesh"] for w in ws])
    phys = dict(ws[0]["phys"], theta_deg=tuple(ws[0]["phys"]["theta_deg"])[:ids])
    st = F.State(mesh, F.params_derive(phys, precision=F.FP32_DEV, **kw), np.concatenate([w["C0"] for w in ws]))
    st.timing_enable(True)
    return st


# large member, launches of a step before the solve and in it
LARGE = {
    "a plane per thread block, forces in two kernels": ((256, 128), 4, 3),      # 128 blocks
    "one full wave, forces in one kernel": ((400, 200), 3, 2),                  # 256 blocks
}


@pytest.mark.parametrize("case", LARGE)
def test_launches_follow_the_members_without_a_block_of_their_own(case):
    (nx, ny), before, solve = LARGE[case]
    small = [I.small_sessile(nx=60, ny=32, seed=70 + k, R=12.0) for k in range(30)]     # 8 blocks each
    big = I.small_sessile(nx=nx, ny=ny, seed=69, R=nx / 6.0)
    st = _state([big] + small)
    st.batch_schedule(5000)
    one = _state([big])
    for s in (st, one):
        s.step(4)
    t, t1 = st.timing_get(), one.timing_get()
    assert (t1["launches"], t1["solve_launches"]) == (before + solve, solve)
    assert (t["launches"], t["solve_launches"]) == (1 + before + solve, solve)
    n = len(big["C0"])
    (g, h), (g1, h1) = st.get_state(), one.get_state()
    np.testing.assert_array_equal(g[:, :n], g1)
    np.testing.assert_array_equal(h[:, :n], h1)
    assert np.isfinite(g).all()
    st.batch_schedule(10 ** 6)
    st.step(1)
    t = st.timing_get()
    assert (t["launches"], t["solve_launches"]) == (1, 0)
