"""Workloads of the framework, as a user's program runs them.

Every case goes through the public Python API (``felbm``, ``felbm3d``,
``adjoint``): time steps of a droplet mesh from a snapshot to the state read
back, a batch of droplets, a loss differentiated through the steps, a mass
solve, and single monitored steps fed from host buffers.  Meshes and droplets
are those of ``inputs.py`` and ``inputs3d.py``; the seed jitters the mesh.

FP64 states return their float64 distributions; FP32-deviation states, whose
content is single precision, return them as float32.
"""
import math

import numpy as np
import torch

from paper_1708_04678_gb300 import adjoint
from paper_1708_04678_gb300 import felbm as F
from paper_1708_04678_gb300 import felbm3d as F3
from paper_1708_04678_gb300 import inputs as I
from paper_1708_04678_gb300 import inputs3d as I3


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # the smallest useful run: one droplet on a flat wall, reference precision (launches and latency)
        {"name": "sessile_64x32_fp64", "kind": "steps", "mesh": "sessile", "nx": 64, "ny": 32,
         "precision": "fp64", "nodal": False, "steps": 50},
        # one monitored step per call, state in and out through host buffers, odd sizes
        {"name": "monitor_97x45_fp64", "kind": "monitor", "mesh": "sessile", "nx": 97, "ny": 45,
         "precision": "fp64", "nodal": False, "steps": 1},
        # capillary intrusion between plates: interior walls, nodal Laplacian of mu, many cheap steps
        {"name": "capillary_16_fp32_nodal", "kind": "steps", "mesh": "capillary", "nx": 16, "ny": 20,
         "precision": "fp32", "nodal": True, "steps": 50},
        # static free droplet, 4-triangle cells (rows of up to 9 entries): FP64 at small size
        {"name": "free_96_fp64", "kind": "steps", "mesh": "free", "nx": 96, "ny": 96,
         "precision": "fp64", "nodal": False, "steps": 20},
        # the spurious-current benchmark: 131,072 nodes, whose working set sits in the L2 cache
        {"name": "free_256_fp32", "kind": "steps", "mesh": "free", "nx": 256, "ny": 256,
         "precision": "fp32", "nodal": False, "steps": 50},
        # a quarter of the rough-wall droplet in reference precision (520,704 nodes)
        {"name": "rough_512_fp64", "kind": "steps", "mesh": "rough", "nx": 512, "ny": 1016,
         "precision": "fp64", "nodal": False, "steps": 10},
        # the headline: the whole rough-wall droplet, 2,082,816 nodes, FP32 deviations
        {"name": "rough_2048_fp32", "kind": "steps", "mesh": "rough", "nx": 2048, "ny": 1016,
         "precision": "fp32", "nodal": False, "steps": 40},
        # a contact-angle sweep: 16 uneven droplets advanced by the same launches
        {"name": "sweep_16_fp32", "kind": "sweep", "members": 16, "w_min": 64, "w_max": 512, "draw": 2,
         "precision": "fp32", "steps": 20},
        # gradient of a wetted-length loss through 20 steps, checkpointed every 10
        {"name": "adjoint_128x64", "kind": "adjoint", "nx": 128, "ny": 64, "steps": 20, "every": 10},
        # L2 projection of five nodal fields held on the device
        {"name": "project_200_k5", "kind": "project", "nx": 200, "ny": 200, "rows": 5},
        # the paper's own 3D setting: static droplet on 1.57 M tetrahedra
        {"name": "static3d_64_fp32", "kind": "steps3d", "nx": 64, "ny": 64, "nz": 64, "walls": False,
         "precision": "fp32", "steps": 10},
        # a small 3D droplet on a substrate in reference precision, uneven sides
        {"name": "sessile3d_25x21x13_fp64", "kind": "steps3d", "nx": 25, "ny": 21, "nz": 13, "walls": True,
         "precision": "fp64", "steps": 10},
    ]


def draw(rng):
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    precision = rng.choice(("fp32", "fp64"))
    kind = rng.choice(("sessile", "sessile", "free", "free", "rough", "capillary", "monitor", "sweep", "adjoint",
                       "project", "steps3d", "steps3d"))
    if kind == "sessile":
        nx = span(40, 500)
        return {"kind": "steps", "mesh": "sessile", "nx": nx, "ny": max(24, nx // 2 + rng.randint(-5, 5)),
                "precision": precision, "nodal": rng.random() < 0.3, "steps": rng.randint(5, 40)}
    if kind == "free":
        nx = span(24, 300 if precision == "fp32" else 180)
        return {"kind": "steps", "mesh": "free", "nx": nx, "ny": nx, "precision": precision,
                "nodal": rng.random() < 0.3, "steps": rng.randint(5, 40)}
    if kind == "rough":
        return {"kind": "steps", "mesh": "rough", "nx": 64 * rng.randint(1, 10), "ny": span(200, 1016),
                "precision": precision, "nodal": False, "steps": rng.randint(3, 15)}
    if kind == "capillary":
        return {"kind": "steps", "mesh": "capillary", "nx": rng.randint(6, 30), "ny": rng.randint(8, 20),
                "precision": precision, "nodal": True, "steps": rng.randint(10, 50)}
    if kind == "monitor":
        nx = span(40, 400)
        return {"kind": "monitor", "mesh": "sessile", "nx": nx, "ny": max(24, nx // 2 + rng.randint(-5, 5)),
                "precision": "fp64", "nodal": False, "steps": 1}
    if kind == "sweep":
        return {"kind": "sweep", "members": rng.randint(3, 24), "w_min": 64, "w_max": rng.randint(96, 400),
                "draw": rng.randint(0, 9999), "precision": precision, "steps": rng.randint(4, 15)}
    if kind == "adjoint":
        nx = span(40, 200)
        return {"kind": "adjoint", "nx": nx, "ny": max(24, nx // 2), "steps": rng.randint(6, 20),
                "every": rng.randint(3, 10)}
    if kind == "project":
        nx = span(30, 220)
        return {"kind": "project", "nx": nx, "ny": nx, "rows": rng.randint(1, 18)}
    nx, walls = span(10, 40 if precision == "fp32" else 26), rng.random() < 0.5
    return {"kind": "steps3d", "nx": nx, "ny": max(8, nx + rng.randint(-3, 6)), "nz": max(8, nx // (2 if walls else 1)),
            "walls": walls, "precision": precision, "steps": rng.randint(3, 10)}


# ----------------------------------------------------------------- inputs --
def _pinned(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, pin_memory=torch.cuda.is_available())


def _workload(case, seed):
    """Mesh, initial composition and physics of a 2D case."""
    if case["kind"] in ("adjoint", "monitor") or case.get("mesh") == "sessile":
        nx, ny = case["nx"], case["ny"]
        mesh = I.grid_mesh(nx, ny, 0.2, seed)
        centre, R = (nx / 2.0, 0.0), 0.1875 * nx
        phys = dict(dt=I.DT_GRID, tau_l=0.8, tau_v=0.8, rho_l=1.0, rho_v=0.1, sigma=0.01, xi=4.0, mobility=0.02,
                    theta_deg=(90.0 if case["kind"] == "adjoint" else 70.0, 90.0))
        C0 = I.droplet_C0(mesh["xy"], centre, R, phys["xi"], mesh["period"])
        return {"mesh": mesh, "C0": C0, "phys": phys, "R": R}
    if case["kind"] == "project" or case.get("mesh") == "free":
        return I.free_droplet_256(seed=seed, n=case["nx"], R=0.1875 * case["nx"])
    if case["mesh"] == "rough":
        height = 1024.0 * case["ny"] / 1016.0
        return I.rough_wall_droplet(seed=seed, width=case["nx"], height=height, rows=case["ny"] + 1,
                                    R=0.293 * min(height, case["nx"]))
    w = I.capillary_channel(H=case["nx"], length_factor=case["ny"], dt=0.05, xi=4.0, mobility=1.0, jitter=0.1,
                            seed=seed)
    return dict(w, R=w["H"])


def _initial(w):
    """Initial p and u: the droplet's Laplace pressure and a slow stirring (1e-3, as late in a run)."""
    xy, C0 = w["mesh"]["xy"], w["C0"]
    span = xy.max(axis=0) + 1e-9
    a, b = 2.0 * np.pi * xy[:, 0] / span[0], np.pi * xy[:, 1] / span[1]
    return w["phys"]["sigma"] / w["R"] * C0, 1e-3 * np.stack([np.sin(a) * np.sin(2 * b), np.cos(a) * np.sin(b) ** 2])


def _members(case, seed):
    rng = np.random.default_rng(case["draw"])
    widths = 2 * rng.integers(case["w_min"] // 2, case["w_max"] // 2 + 1, size=case["members"])
    thetas = rng.uniform(30.0, 150.0, size=case["members"])
    out = []
    for k, (W, theta) in enumerate(zip(widths, thetas)):
        W = int(W)
        w = _workload({"kind": "steps", "mesh": "sessile", "nx": W, "ny": W // 2}, [seed, k])
        w["phys"]["theta_deg"] = (float(theta), 90.0)
        out.append(dict(w, name="member", steps=case["steps"]))
    return out


def _workload3(case, seed):
    mesh = I3.kuhn_box(case["nx"], case["ny"], case["nz"], 0.15, seed, walls=case["walls"])
    low = min(case["nx"], case["ny"], case["nz"] * (2 if case["walls"] else 1))
    centre = (case["nx"] / 2.0, case["ny"] / 2.0, 0.0 if case["walls"] else case["nz"] / 2.0)
    phys = dict(dt=I3.DT_KUHN, tau_l=0.8, tau_v=0.8, rho_l=1.0, rho_v=0.5, sigma=0.01, xi=4.0, mobility=0.02,
                theta_deg=(60.0, 90.0) if case["walls"] else ())
    C0 = I3.droplet_C0_3d(mesh["xyz"], centre, 0.25 * low, phys["xi"], mesh["period"])
    return {"mesh": mesh, "C0": C0, "phys": phys, "R": 0.25 * low}


def _equilibrium(E, W, phys, C, p, u, g, h):
    """Distributions at equilibrium with C, p, u, written to g, h (all on one device)."""
    rho = phys["rho_v"] + C * (phys["rho_l"] - phys["rho_v"])
    uu = 1.5 * sum(x * x for x in u)
    for q in range(len(W)):
        eu = sum(float(E[q][k]) * u[k] for k in range(len(u)))
        T = 3.0 * eu + 4.5 * eu * eu - uu
        g[q] = float(W[q]) * (p + rho * T / 3.0)
        h[q] = float(W[q]) * (1.0 + T) * C


def _state_arrays(case, w):
    """Initial (g, h), float64, of a case that starts from distributions."""
    E, W = (E2, W2) if "xy" in w["mesh"] else (E3, W3)
    C = torch.from_numpy(np.ascontiguousarray(w["C0"]))
    if "xy" in w["mesh"]:
        p, u = (torch.from_numpy(np.ascontiguousarray(a)) for a in _initial(w))
    else:
        xyz = torch.from_numpy(w["mesh"]["xyz"])
        p = w["phys"]["sigma"] / w["R"] * C
        a, b = 2 * math.pi * xyz[:, 0] / case["nx"], 2 * math.pi * xyz[:, 1] / case["ny"]
        c = math.pi * xyz[:, 2] / case["nz"]
        u = 1e-3 * torch.stack([torch.sin(a) * torch.sin(c), torch.cos(b) * torch.sin(c), torch.sin(a + b) * torch.sin(c) ** 2])
    g, h = _pinned(len(W), len(C)), _pinned(len(W), len(C))
    _equilibrium(E, W, w["phys"], C, p, u, g, h)
    return g, h


E2 = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)], dtype=np.float64)
W2 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
E3 = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
               (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
               (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)], dtype=np.float64)
W3 = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _params(case, phys):
    return F.params_derive(phys, precision=F.FP32_DEV if case.get("precision") == "fp32" else F.FP64,
                           lapmu_mode=F.LAPMU_NODAL if case.get("nodal") else F.LAPMU_FACE)


def _with_buffers(s, case, q, n):
    """Host buffers the state is read back into: pinned float64, and single precision for FP32 states."""
    s["g"], s["h"] = _pinned(q, n), _pinned(q, n)
    if case["precision"] == "fp32":
        s["out"] = torch.empty(q, n, dtype=torch.float32), torch.empty(q, n, dtype=torch.float32)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "steps3d":
        w = _workload3(case, seed)
        st = F3.State3D(F3.Mesh3D.from_dict(w["mesh"]), _params(case, w["phys"]), w["C0"])
        g0, h0 = _state_arrays(case, w)
        return _with_buffers({"case": case, "st": st, "g0": g0, "h0": h0}, case, 19, st.N)
    if kind == "sweep":
        b = I.batch(_members(case, seed))
        st = F.State(F.Mesh.batch(b["meshes"]), _params(case, b["phys"]), b["C0"])
        s = {"case": case, "st": st}
    else:
        w = _workload(case, seed)
        mesh = F.Mesh.from_dict(w["mesh"])
        if kind == "project":
            st = F.State(mesh, _params(case, w["phys"]), w["C0"])
            gen = torch.Generator(device="cuda").manual_seed(int(seed))
            B = torch.randn(case["rows"], st.N, dtype=torch.float64, device="cuda", generator=gen)
            return {"case": case, "st": st, "B": B, "X": torch.empty_like(B)}
        if kind == "adjoint":
            params = _params(case, w["phys"])
            st = F.State(mesh, params, w["C0"])
            phi = torch.tensor([params.phi_c[k] for k in range(params.n_wall_ids)], dtype=torch.float64)
            return {"case": case, "st": st, "C0": torch.from_numpy(w["C0"]), "phi": phi,
                    "edges": adjoint.wall_edge_table(w["mesh"], 0), "target": 0.3 * case["nx"]}
        if kind == "monitor":
            st = F.State(mesh, _params(case, w["phys"]), w["C0"])
            g0, h0 = _state_arrays(case, w)
            s = {"case": case, "st": st, "g0": g0, "h0": h0, "slots": _pinned(F.DIAG_SLOTS)}
            return _with_buffers(s, case, 9, st.N)
        p0, u0 = _initial(w)
        st = F.State(mesh, _params(case, w["phys"]), w["C0"], p0=p0, u0=u0)
        s = {"case": case, "st": st}
    # a snapshot in device memory, from which every run of the program restarts
    s["ck"] = torch.empty(st.checkpoint_bytes(), dtype=torch.uint8, device="cuda")
    st.checkpoint_save(s["ck"])
    return _with_buffers(s, case, 9, st.N)


# -------------------------------------------------------------------- run --
def run(s):
    case, st = s["case"], s["st"]
    kind = case["kind"]
    if kind == "project":
        st.mass_solve_static(s["B"], s["X"])
        return s["X"]
    if kind == "adjoint":
        C0, phi = s["C0"].clone().requires_grad_(), s["phi"].clone().requires_grad_()
        g, h = adjoint.run(st, C0, phi, case["steps"], every=case["every"])
        loss = (adjoint.wetted_length(h, s["edges"]) - s["target"]) ** 2
        loss.backward()
        return {"g": g.detach(), "h": h.detach(), "dC0": C0.grad, "dphi": phi.grad}
    if kind == "monitor":
        st.set_state(s["g0"], s["h0"])
        st.step(case["steps"])
        st.diagnostics_enqueue(s["slots"])
        st.get_state(s["g"], s["h"])
        d = st.diag_finish(s["slots"])
        return {"g": s["g"], "h": s["h"],
                "diag": [float(d[k]) for k in ("mass", "kinetic_energy", "max_u", "wetted_length", "height", "theta_deg")]}
    if kind == "steps3d":
        st.set_state(s["g0"], s["h0"])
    else:
        st.checkpoint_load(s["ck"])
    st.step(case["steps"])
    st.get_state(s["g"], s["h"])
    if case["precision"] == "fp32":
        s["out"][0].copy_(s["g"])
        s["out"][1].copy_(s["h"])
        return {"g": s["out"][0], "h": s["out"][1]}
    return {"g": s["g"], "h": s["h"]}


# ------------------------------------------------------------------- work --
def _counts(case):
    """(nodes, elements) of a case's mesh."""
    nx, ny = case.get("nx"), case.get("ny")
    if case["kind"] == "steps3d":
        return nx * ny * (case["nz"] + (1 if case["walls"] else 0)), 6 * nx * ny * case["nz"]
    if case["kind"] == "sweep":
        rng = np.random.default_rng(case["draw"])
        widths = 2 * rng.integers(case["w_min"] // 2, case["w_max"] // 2 + 1, size=case["members"])
        return int(sum(w * (w // 2 + 1) for w in widths)), int(sum(w * w for w in widths))
    if case["kind"] == "project" or case.get("mesh") == "free":
        return 2 * nx * ny, 4 * nx * ny
    if case.get("mesh") == "capillary":
        fluid = nx * nx * ny + 2 * 4 * nx * 3 * nx
        return fluid, 2 * fluid
    return nx * (ny + 1), 2 * nx * ny


def work(case):
    """Each step reads and writes the state once and reads the mesh once (vertices, coordinates); what is read
    back crosses to the host.  Flops: residuals and forces per element, the gather and the solve per node."""
    n, t = _counts(case)
    d = 3 if case["kind"] == "steps3d" else 2
    q = 38 if d == 3 else 18
    row = 15 if d == 3 else 7
    mesh = 4 * (d + 1) * t + 8 * d * n
    if case["kind"] == "project":
        return {"bytes": 16.0 * case["rows"] * n + mesh, "flops": 32.0 * case["rows"] * n * (2 * row + 4)}
    fp32 = case.get("precision") == "fp32"
    state = n * (4 * q + 8 + 4 * (d + 1) if fp32 else 8 * q)
    sweeps = (16 if d == 3 else 10) if fp32 else (48 if d == 3 else 42)
    step_flops = t * (24.0 * q) + n * (2.0 * q * t / n * (d + 1) + sweeps * q * (2 * row + 4))
    steps = case["steps"] * (4 if case["kind"] == "adjoint" else 1)
    return {"bytes": float(steps * (2 * state + mesh) + 8 * q * n), "flops": float(steps * step_flops)}


# ------------------------------------------------- the same in 64-bit torch --
class _Reference:
    """The FE-LBM step (Sec. II of arXiv:1708.04678) in d dimensions with dense torch operations in float64,
    differentiable; rows of psi are nodes, columns the populations of g then h."""

    def __init__(self, xy, elem, facets, facet_id, period, phys, nodal, device):
        self.dev, self.phys, self.nodal = device, phys, nodal
        x = torch.as_tensor(xy, dtype=torch.float64, device=device)
        self.el = el = torch.as_tensor(np.asarray(elem), dtype=torch.int64, device=device)
        self.N, self.d = x.shape[0], x.shape[1]
        d = self.d
        self.E = torch.as_tensor(E2 if d == 2 else E3, device=device)
        self.W = torch.as_tensor(W2 if d == 2 else W3, device=device)
        self.opp = [int(((self.E + self.E[q]) == 0).all(1).nonzero()[0, 0]) for q in range(len(self.W))]

        def image(v):
            for k in range(d):
                if period[k] > 0:
                    v[..., k] -= period[k] * torch.round(v[..., k] / period[k])
            return v

        J = image(x[el[:, 1:]] - x[el[:, :1]])                        # rows: edge vectors
        self.vol = torch.linalg.det(J) / math.factorial(d)
        b = torch.linalg.inv(J).transpose(1, 2)                       # gradients of the shape functions 1..d
        self.b = torch.cat([-b.sum(1, keepdim=True), b], 1)           # (T, d+1, d)
        self.patch = self.gather([self.vol] * (d + 1))
        self.lumped = self.patch / (d + 1)
        rows, cols, mass, stiff = [], [], [], []
        for i in range(d + 1):
            for j in range(d + 1):
                rows.append(el[:, i])
                cols.append(el[:, j])
                mass.append(self.vol * ((2.0 if i == j else 1.0) / ((d + 1) * (d + 2))))
                stiff.append(self.vol * (self.b[:, i] * self.b[:, j]).sum(1))
        at = torch.stack([torch.cat(rows), torch.cat(cols)])
        self.M, self.K = (torch.sparse_coo_tensor(at, torch.cat(v), (self.N, self.N)).coalesce().to_sparse_csr()
                          for v in (mass, stiff))
        # the element across the facet opposite vertex k (-1: wall)
        T = el.shape[0]
        key = []
        for k in range(d + 1):
            f = el[:, [j for j in range(d + 1) if j != k]].sort(1).values
            v = f[:, 0]
            for j in range(1, d):
                v = v * self.N + f[:, j]
            key.append(v)
        key, order = torch.cat(key).sort()
        same = (key[1:] == key[:-1]).nonzero()[:, 0]
        nbr = torch.full(((d + 1) * T,), -1, dtype=torch.int64, device=device)
        nbr[order[same]] = order[same + 1] % T
        nbr[order[same + 1]] = order[same] % T
        self.nbr = nbr.reshape(d + 1, T)
        # wall facets: measure, unit normal out of the fluid
        self.wall = torch.as_tensor(np.asarray(facets), dtype=torch.int64, device=device).reshape(-1, d)
        self.wall_id = torch.as_tensor(np.asarray(facet_id), dtype=torch.int64, device=device)
        if len(self.wall):
            open_ = (self.nbr < 0).nonzero()                          # (facet slot, element)
            slot, tt = open_[:, 0], open_[:, 1]
            others = torch.stack([torch.tensor([j for j in range(d + 1) if j != k], device=device) for k in range(d + 1)])
            f = torch.gather(el[tt], 1, others[slot]).sort(1).values
            code, want = f[:, 0], self.wall.sort(1).values
            wcode = want[:, 0]
            for j in range(1, d):
                code, wcode = code * self.N + f[:, j], wcode * self.N + want[:, j]
            code, order = code.sort()
            pick = order[torch.searchsorted(code, wcode)]
            nu = -d * self.vol[tt[pick], None] * self.b[tt[pick], slot[pick]]
            self.wall_len = nu.norm(dim=1)
            self.wall_n = nu / self.wall_len[:, None]

    def gather(self, parts):
        out = torch.zeros((self.N,) + parts[0].shape[1:], dtype=torch.float64, device=self.dev)
        for k, v in enumerate(parts):
            out = out.index_add(0, self.el[:, k], v)
        return out

    def spmm(self, A, X):
        return torch.sparse.mm(A, X)

    def solve(self, B, steps=44):
        """Chebyshev recurrence on the spectrum [1/(d+2), 1] of the lumped-preconditioned mass matrix."""
        theta, delta = 0.5 * (1 + 1 / (self.d + 2)), 0.5 * (1 - 1 / (self.d + 2))
        Z = 1.0 / self.lumped[:, None]
        rho, p = delta / theta, Z * B / theta
        X = p
        for _ in range(steps):
            rho_n = 1.0 / (2.0 * theta / delta - rho)
            p = rho_n * rho * p + (2.0 * rho_n / delta) * Z * (B - self.spmm(self.M, X))
            X = X + p
            rho = rho_n
        return X

    def gamma(self, u):
        eu = u @ self.E.T
        return self.W * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(1, keepdim=True))

    def lap(self, f):
        return -self.spmm(self.K, f[:, None])[:, 0] / self.lumped

    def step(self, g, h, phi):
        c, d, el, b, Q = self.phys, self.d, self.el, self.b, len(self.W)
        sig, xi = c["sigma"], c["xi"]
        kappa, beta = 1.5 * sig * xi, 12.0 * sig / xi
        C, p = h.sum(1), g.sum(1)
        drho = c["rho_l"] - c["rho_v"]
        rho = c["rho_v"] + C * drho
        u = 3.0 * (g @ self.E) / rho[:, None]
        flux = torch.zeros_like(C)
        if len(self.wall):
            Cw = C[self.wall]
            s1, s2 = Cw.sum(1), (Cw * Cw).sum(1)
            q = -phi[self.wall_id] * self.wall_len * (s1 / d - (s2 + s1 * s1) / (d * (d + 1)))
            for k in range(d):
                flux = flux.index_add(0, self.wall[:, k], q / d)
        mu = 2 * beta * C * (C - 1) * (2 * C - 1) - kappa * self.lap(C) - flux / self.lumped
        grad = lambda f: sum(f[el[:, k], None] * b[:, k] for k in range(1, d + 1)) + f[el[:, 0], None] * b[:, 0]
        mean = lambda f: f[el].mean(1)
        if self.nodal:
            lapmu = mean(self.lap(mu))
        else:
            G = grad(mu)
            lapmu = torch.zeros_like(self.vol)
            for k in range(d + 1):
                inner = (self.nbr[k] >= 0).to(torch.float64)
                lapmu = lapmu - 0.5 * d * inner * ((G + G[self.nbr[k].clamp(min=0)]) * b[:, k]).sum(1)
        Cb, ub, mub = mean(C), mean(u), mean(mu)
        rhob = c["rho_v"] + Cb * drho
        gC, gp = grad(C), grad(p)
        Gb = self.gamma(ub)
        eC = gC @ self.E.T - (ub * gC).sum(1, keepdim=True)
        vh = gC - (3 * Cb / rhob)[:, None] * (gp - mub[:, None] * gC)
        ev = vh @ self.E.T - (ub * vh).sum(1, keepdim=True)
        R = torch.cat([drho / 3 * (Gb - self.W) * eC + mub[:, None] * Gb * eC,
                       (ev + c["mobility"] * lapmu[:, None]) * Gb], 1)
        om = 1 / (1 / (C / c["tau_l"] + (1 - C) / c["tau_v"]) + 0.5)
        Gn = self.gamma(u)
        geq = self.W * p[:, None] + rho[:, None] / 3 * (Gn - self.W)
        psi = torch.cat([g - om[:, None] * (g - geq), h - om[:, None] * (h - Gn * C[:, None])], 1)
        for k in range(d + 1):
            R = R - psi[el[:, k]] * (b[:, k] @ self.E.T).repeat(1, 2)
        R = R * self.vol[:, None]
        dt = c["dt"]
        rhs = self.gather([R * (dt / (d + 1) + 0.5 * dt * dt * (b[:, k] @ self.E.T)).repeat(1, 2) for k in range(d + 1)])
        if len(self.wall):
            en = (self.wall_n @ self.E.T).clamp(max=0.0).repeat(1, 2)
            diff = psi[:, self.opp + [Q + o for o in self.opp]] - psi
            dw = [diff[self.wall[:, k]] for k in range(d)]
            tot = sum(dw)
            for k in range(d):
                rhs = rhs.index_add(0, self.wall[:, k],
                                    -dt * en * (self.wall_len / (d * (d + 1)))[:, None] * (tot + dw[k]))
        psi = psi + self.solve(rhs)
        return psi[:, :Q], psi[:, Q:]


def _phi(phys):
    return torch.tensor([-6.0 * phys["sigma"] * math.cos(math.radians(t)) for t in phys["theta_deg"]] or [0.0],
                        dtype=torch.float64)


def _reference(w, nodal, device):
    m = w["mesh"]
    if "xy" in m:
        return _Reference(m["xy"], m["tri"], m["wall_edges"], m["wall_id"], m["period"], w["phys"], nodal, device)
    return _Reference(m["xyz"], m["tet"], m["wall_faces"], m["wall_id"], m["period"], w["phys"], nodal, device)


def _advance(w, case, g, h, device):
    """(g, h) after the case's steps, [directions][nodes], float64 on the host."""
    ref, phi = _reference(w, bool(case.get("nodal")), device), _phi(w["phys"]).to(device)
    g, h = g.to(device).T.contiguous(), h.to(device).T.contiguous()
    for _ in range(case["steps"]):
        g, h = ref.step(g, h, phi)
    return g.T.contiguous().cpu(), h.T.contiguous().cpu()


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "sweep":
        parts = []
        for w in _members(case, seed):
            C = torch.from_numpy(w["C0"])
            g, h = torch.zeros(9, len(C), dtype=torch.float64), torch.from_numpy(W2)[:, None] * C
            parts.append(_advance(w, case, g, h, device))
        return {"g": torch.cat([p[0] for p in parts], 1), "h": torch.cat([p[1] for p in parts], 1)}
    w = _workload3(case, seed) if kind == "steps3d" else _workload(case, seed)
    if kind == "project":
        ref = _reference(w, False, device)
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        B = torch.randn(case["rows"], ref.N, dtype=torch.float64, device="cuda", generator=gen)
        return ref.solve(B.T.contiguous()).T.contiguous()
    if kind == "adjoint":
        ref, phi = _reference(w, False, device), _phi(w["phys"]).to(device).requires_grad_()
        C0 = torch.from_numpy(w["C0"]).to(device).requires_grad_()
        g, h = torch.zeros(ref.N, 9, dtype=torch.float64, device=device), C0[:, None] * ref.W
        for _ in range(case["steps"]):
            g, h = ref.step(g, h, phi)
        C = h.sum(1)[ref.wall[ref.wall_id == 0]]
        hi, lo = C.max(1).values, C.min(1).values
        part = torch.where((hi >= 0.5) & (lo < 0.5), (hi - 0.5) / (hi - lo).clamp(min=1e-30), torch.zeros_like(hi))
        length = (ref.wall_len[ref.wall_id == 0] * torch.where(lo >= 0.5, torch.ones_like(hi), part)).sum()
        ((length - 0.3 * case["nx"]) ** 2).backward()
        return {"g": g.detach().T.contiguous().cpu(), "h": h.detach().T.contiguous().cpu(),
                "dC0": C0.grad.cpu(), "dphi": phi.grad.cpu()}
    g, h = _advance(w, case, *_state_arrays(case, w), device)
    return {"g": g, "h": h, "diag": None} if kind == "monitor" else {"g": g, "h": h}
