"""Which form the FP32 solve takes by default (one launch per step, or several
steps of a node block per launch), seen by its launches, and the bits of the
default against both forms."""
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


def _batch():
    """64 droplets of 1,012 to 3,960 nodes: 392 blocks, more than one wave of them
    and not two, in L2."""
    return I.batch([I.small_sessile(nx=nx, ny=nx // 2, seed=100 + k, R=nx / 5.0)
                    for k, nx in enumerate(np.linspace(44, 88, 64).astype(int))])


def _periodic_batch():
    """20 periodic droplets of 16 blocks of 512 nodes: 320 blocks in two waves, the
    second nearly empty."""
    ws = [I.small_free_droplet(n=64, R=12.0, seed=50 + k) for k in range(20)]
    return {"meshes": [w["mesh"] for w in ws], "C0": np.concatenate([w["C0"] for w in ws]), "phys": ws[0]["phys"]}


# workload, node order, solver_iters, launches of the solve phase of one step
CASES = {
    "a plane per thread block": (lambda: I.small_sessile(nx=64, ny=32, R=12.0), None, 0, 3),       # 2 + field update
    "one wave": (lambda: I.small_sessile(nx=400, ny=200, R=60.0), None, 0, 2),
    "full blocks": (lambda: I.small_sessile(nx=723, ny=361, R=90.0), None, 0, 3),
    "beyond L2": (lambda: I.small_sessile(nx=1024, ny=512, R=100.0), None, 0, 2),
    "partial waves": (_batch, None, 0, 9),
    "partial waves of full blocks": (_periodic_batch, None, 0, 9),
    "small blocks": (lambda: I.small_free_droplet(n=258, R=50.0), None, 0, 9),
    "one step": (lambda: I.small_sessile(nx=64, ny=32, R=12.0), None, 2, 1),
    "one layer": (lambda: I.small_sessile(nx=120, ny=300, R=40.0), "rcm", 0, 9),
}


@pytest.mark.parametrize("case", CASES)
def test_default_form_of_the_solve(case, monkeypatch):
    make, order, iters, launches = CASES[case]
    if order:
        monkeypatch.setenv("FELBM_ORDER", order)
    w = make()
    mesh = F.Mesh.batch(w["meshes"]) if "meshes" in w else F.Mesh.from_dict(w["mesh"])
    params = F.params_derive(w["phys"], precision=F.FP32_DEV, solver_iters=iters)
    ref = None
    for form in (None, True, False):
        st = F.State(mesh, params, w["C0"])
        if form is not None:
            st.sweep_tiled(form)
        st.timing_enable(True)
        st.step(3)
        n = st.timing_get()["solve_launches"]
        if form is None:
            assert n == launches
        elif form is False:
            assert n == (iters or 10) - 1
        got = st.get_state()
        ref = ref or got
        for x, y in zip(got, ref):
            np.testing.assert_array_equal(x, y)
        st.close()
    assert np.isfinite(ref[0]).all() and np.abs(ref[1]).max() > 0
