"""Edge matching of the mesh set-up: meshes with shuffled node numbers are
taken, faulty edges and walls refused."""
import numpy as np
import pytest

from paper_1708_04678_gb300 import felbm as F
from paper_1708_04678_gb300 import inputs as I


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1708_04678_gb300 import build
    build.build()


def _mesh(seed):
    """A walled, x-periodic grid with its nodes renumbered at random."""
    m = I.small_sessile(nx=12, ny=7, R=3.0)["mesh"]
    p = np.random.default_rng(seed).permutation(len(m["xy"])).astype(np.int32)
    xy = np.empty_like(m["xy"])
    xy[p] = m["xy"]
    return dict(m, xy=xy, tri=p[m["tri"]], wall_edges=p[m["wall_edges"]])


def _tripled(m):
    return dict(m, tri=np.concatenate([m["tri"], m["tri"][5:6]]))


def _hole(m):
    return dict(m, tri=np.delete(m["tri"], 40, 0))


def _duplicate(m):
    return dict(m, wall_edges=np.concatenate([m["wall_edges"], m["wall_edges"][3:4, ::-1]]),
                wall_id=np.concatenate([m["wall_id"], m["wall_id"][3:4]]))


def _missing(m):
    return dict(m, wall_edges=m["wall_edges"][1:], wall_id=m["wall_id"][1:])


def _inside(m):
    walls = {frozenset(e) for e in m["wall_edges"].tolist()}
    e = next(t[:2] for t in m["tri"].tolist() if frozenset(t[:2]) not in walls)
    return dict(m, wall_edges=np.concatenate([m["wall_edges"], np.array([e], np.int32)]),
                wall_id=np.concatenate([m["wall_id"], m["wall_id"][:1]]))


@pytest.mark.parametrize("seed", [0, 1])
@pytest.mark.parametrize("change,message", [
    (_tripled, "more than two triangles"), (_hole, "not a wall edge"), (_duplicate, "duplicate wall edge"),
    (_missing, "not a wall edge"), (_inside, "not a boundary edge")])
def test_faulty_edges_are_refused(seed, change, message):
    m = _mesh(seed)
    F.Mesh.from_dict(m).close()
    with pytest.raises(F.FelbmError, match=message):
        F.Mesh.from_dict({k: np.ascontiguousarray(v) if isinstance(v, np.ndarray) else v for k, v in change(m).items()})
