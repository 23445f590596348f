"""The work a user of the solver has it do, as cases that can be timed and checked.

A case is one call pattern on one mesh: load a state from device memory, run
p-multigrid V-cycles or explicit high-order steps, read the state and the
residual history back; or a batch of requests through the server.  Meshes,
settings and states are those of the repository's benchmark and tests: the
lid-driven cavity, the hybrid cylinder O-mesh, the shock reflection box, the
sphere shell and the 3-D box.  Every state carries a smooth perturbation drawn
from the seed, so another seed is another input.

`exact` evaluates the same scheme in 64 bits with plain numpy and torch: its
own faces, colours, least-squares operators, fluxes and relaxation.
"""
import math

import numpy as np
import torch

from paper_2109_09965_gb300 import cgks, meshgen

GAMMA = 1.4
P_INF = 1.0 / GAMMA
# flow settings: Mach number and Reynolds number (0: inviscid) of each flow
FLOWS = {
    "cavity": (0.15, 1000.0), "cylinder": (0.38, 0.0), "shock": (2.9, 0.0), "sphere": (0.2, 118.0),
    "box3": (0.15, 100.0),
}


def listed():
    return [
        # the smallest solve anyone runs (smoke and unit-test size): one V-cycle, all latency
        dict(name="cavity128_fp64", flow="cavity", a=8, b=0, c=0, mode="cycles", n=1, precision="fp64", scheme="S1O2",
             limited=False, lf=False),
        # configuration 1: the 2048-cell lid-driven cavity, V-cycles in FP64 and mixed precision
        dict(name="cavity2k_fp64", flow="cavity", a=32, b=0, c=0, mode="cycles", n=8, precision="fp64", scheme="S1O2",
             limited=False, lf=False),
        dict(name="cavity2k_mixed", flow="cavity", a=32, b=0, c=0, mode="cycles", n=8, precision="mixed",
             scheme="S1O2", limited=False, lf=False),
        # the headline workload: the 57,344-cell cylinder, V-cycles in both precisions
        dict(name="cylinder57k_fp64", flow="cylinder", a=256, b=32, c=96, mode="cycles", n=2, precision="fp64",
             scheme="S1O2", limited=False, lf=False),
        dict(name="cylinder57k_mixed", flow="cylinder", a=256, b=32, c=96, mode="cycles", n=4, precision="mixed",
             scheme="S1O2", limited=False, lf=False),
        # a ragged transonic cylinder as a served request has it: full flux, compact WENO, Lax-Friedrichs low level
        dict(name="cylinder6k_limited", flow="cylinder", a=97, b=11, c=27, mode="cycles", n=3, precision="fp64",
             scheme="S1O2", limited=True, lf=True),
        # the shock reflection problem: full flux, characteristic WENO, explicit two-stage steps (the paper's S2O4)
        dict(name="shock_fp64", flow="shock", a=120, b=30, c=0, mode="explicit", n=8, precision="fp64", scheme="S2O4",
             limited=True, lf=False),
        # 3-D laminar sphere shell in FP64 at 128,000 cells: V-cycle with the viscous low level
        dict(name="sphere128k_fp64", flow="sphere", a=3, b=40, c=20, mode="cycles", n=1, precision="fp64",
             scheme="S1O2", limited=False, lf=False),
        # configuration 3: the 512,000-cell sphere, mixed precision V-cycle
        dict(name="sphere512k_mixed", flow="sphere", a=4, b=40, c=20, mode="cycles", n=1, precision="mixed",
             scheme="S1O2", limited=False, lf=False),
        # compressible sphere with the full flux and compact WENO, explicit S2O4 steps in mixed precision
        dict(name="sphere128k_limited", flow="sphere", a=3, b=40, c=20, mode="explicit", n=1, precision="mixed",
             scheme="S2O4", limited=True, lf=False),
        # a ragged hexahedral box in FP64, explicit S2O4 steps
        dict(name="box9k_explicit", flow="box3", a=23, b=21, c=19, mode="explicit", n=2, precision="fp64",
             scheme="S2O4", limited=False, lf=False),
        # the server: requests of both flux classes through one continuous batch, submission to retirement
        dict(name="serve6_mixed", flow="serve", a=6, b=2000, c=20000, mode="serve", n=24, precision="mixed",
             scheme="S1O2", limited=False, lf=False),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    flow = rng.choice(["cavity", "cavity", "cylinder", "cylinder", "shock", "sphere", "sphere", "box3", "serve"])
    c = dict(flow=flow, b=0, c=0, mode=rng.choice(["cycles", "cycles", "explicit"]), n=rng.randint(1, 4),
             precision=rng.choice(["fp64", "mixed"]), scheme=rng.choice(["S1O2", "S2O4"]), limited=False, lf=False)
    if flow == "cavity":
        c.update(a=log_int(8, 180), lf=rng.random() < 0.25)
    elif flow == "cylinder":
        a = log_int(24, 256)
        c.update(a=a, b=max(2, a // 8 + rng.randint(-1, 1)), c=max(4, 3 * a // 8 + rng.randint(-3, 3)),
                 limited=rng.random() < 0.4, lf=rng.random() < 0.25)
    elif flow == "shock":
        c.update(a=log_int(40, 240), b=log_int(10, 60), mode="explicit", limited=True)
    elif flow == "sphere":
        c.update(a=rng.choice([2, 2, 3]), b=rng.randint(20, 40), c=rng.randint(10, 20), n=1,
                 limited=rng.random() < 0.3)
        if c["limited"]:
            c.update(mode="explicit")
    elif flow == "box3":
        c.update(a=log_int(5, 32), b=log_int(5, 32), c=log_int(5, 32))
    else:
        c.update(a=rng.randint(2, 8), b=2000, c=log_int(4000, 20000), mode="serve", n=rng.randint(8, 24),
                 scheme="S1O2")
    return c


# ------------------------------------------------------------------ inputs
_MESHES = {}   # a user's mesh outlives the solves on it


def _mesh_of(flow, a, b, c, seed=1):
    key = (flow, a, b, c, seed)
    if key not in _MESHES:
        if len(_MESHES) > 40:
            _MESHES.clear()
        if flow == "cavity":
            m = meshgen.cavity(a, seed=seed)
        elif flow == "cylinder":
            m = meshgen.cylinder(a, b, c, growth=meshgen.cylinder_growth_isotropic(a, b) if a < 256 else 1.08)
        elif flow == "shock":
            m = meshgen.shock_reflection(a, b)
        elif flow == "sphere":
            m = meshgen.sphere(a, b, c, h0=1e-3, R_far=5.0)
        else:
            m = meshgen.box3(a, b, c, cells="hex", jitter=0.1, seed=3)
        _MESHES[key] = (m, cgks.Mesh(m))
    return _MESHES[key]


def _spec(case, ma=None, re=None):
    flow = case["flow"]
    ma0, re0 = FLOWS[flow]
    ma, re = ma0 if ma is None else ma, re0 if re is None else re
    free = dict(kind="farfield", rho=1.0, u=(ma, 0.0, 0.0) if flow == "sphere" else (ma, 0.0), p=P_INF)
    if flow == "cavity":
        bcs = [dict(kind="noslip"), dict(kind="noslip", uw=(ma, 0.0))]
    elif flow == "cylinder":
        bcs = [dict(kind="slip"), free]
    elif flow == "shock":
        def state(q):
            return dict(kind="dirichlet", rho=q[0], u=(q[1], q[2]), p=q[3])
        bcs = [dict(kind="slip"), dict(kind="outflow"), state(meshgen.SR_UP), state(meshgen.SR_LEFT)]
    elif flow == "sphere":
        bcs = [dict(kind="noslip"), free]
    else:
        bcs = [dict(kind="noslip")] * 5 + [dict(kind="noslip", uw=(ma, 0.0, 0.0))]
    spec = dict(gamma=GAMMA, mu=ma / re if re else 0.0, cfl_hi=0.4, cfl_lo=1000.0, n_implicit=6, n_sweeps=2,
                time_scheme=case["scheme"], precision=case["precision"], bcs=bcs,
                flux_lo="lf" if case["lf"] else "kfvs", lo_viscous=1 if flow == "sphere" else 0)
    if case["limited"]:
        spec.update(flux_hi="full", weno_eps=1e-2,
                    weno_vars="characteristic" if flow == "shock" else "conservative")
    return spec


def _state(mesh, flow, ma, seed):
    """Uniform stream (or rest, or the shock problem's left state) with a 1 %
    smooth perturbation of density, velocity and pressure."""
    rng = np.random.default_rng(seed)
    D = mesh.dim
    ptr = mesh.cell_ptr
    x = np.add.reduceat(mesh.nodes[mesh.cell_nodes], ptr[:-1], axis=0) / np.diff(ptr)[:, None]
    rho, p, u = 1.0, P_INF, np.zeros(D)
    if flow == "shock":
        rho, p, u[:2] = meshgen.SR_LEFT[0], meshgen.SR_LEFT[3], meshgen.SR_LEFT[1:3]
    elif flow in ("cylinder", "sphere"):
        u[0] = ma
    k = rng.uniform(0.5, 2.5, (D + 2, D)) * rng.choice([-1.0, 1.0], (D + 2, D))
    ph = rng.uniform(0.0, 2.0 * math.pi, D + 2)
    w = 0.01 * np.sin(x @ k.T + ph)                            # [n, D + 2]
    r = rho * (1.0 + w[:, 0])
    v = u[None, :] + max(ma, 0.1) * w[:, 1:1 + D]
    pr = p * (1.0 + w[:, D + 1])
    E = pr / (GAMMA - 1.0) + 0.5 * r * (v * v).sum(1)
    return np.concatenate([r[:, None], r[:, None] * v, E[:, None]], axis=1)


def _requests(case, seed):
    """Half cavities (smooth flux), half cylinders (the limited class), cell
    counts log-uniform in [b, c]: the benchmark's serving mix."""
    rng = np.random.default_rng(case["a"] * 100003 + case["c"])
    out = []
    for r in range(case["a"]):
        cells = math.exp(rng.uniform(math.log(case["b"]), math.log(case["c"])))
        if r % 2 == 0:
            sub = dict(case, flow="cavity", a=max(8, int(round(math.sqrt(cells / 2.0)))), b=0, c=0)
            ma, re = 0.15, math.exp(rng.uniform(math.log(100.0), math.log(3200.0)))
        else:
            nt = max(16, 8 * int(round(math.sqrt(cells * 8.0 / 7.0) / 8.0)))
            sub = dict(case, flow="cylinder", a=nt, b=nt // 8, c=3 * nt // 8, limited=True)
            ma, re = rng.uniform(0.2, 0.5), 0.0
        m, g = _mesh_of(sub["flow"], sub["a"], sub["b"], sub["c"], seed=1 + r if sub["flow"] == "cavity" else 1)
        out.append((m, g, _spec(sub, ma, re), _state(m, sub["flow"], ma, seed * 1000 + r)))
    return out


TUNE_UNITS = 16   # V-cycles or steps after which a solver's launch shapes are final


def prepare(case, seed):
    if case["mode"] == "serve":
        # a running server (shapes tuned on earlier requests) and the requests in hand
        srv = cgks.Server(6 << 30, precision=case["precision"], max_active=16, max_cycles=1000, lo_viscous=1)
        warm = _requests(dict(case, a=2, c=case["b"] + 1), 0)
        for _, g, spec, W in warm:
            srv.submit(g, spec, W, 1e-300, TUNE_UNITS)
        while srv.step():
            pass
        return dict(case=case, srv=srv, reqs=_requests(case, seed))
    m, g = _mesh_of(case["flow"], case["a"], case["b"], case["c"])
    s = cgks.Solver(g, _spec(case))
    W = torch.from_numpy(_state(m, case["flow"], FLOWS[case["flow"]][0], seed)).cuda()
    st = dict(case=case, s=s, W=W, Wo=torch.empty_like(W),
              Xo=torch.empty((m.n_cells, m.dim, m.dim + 2), dtype=torch.float64, device="cuda"))
    # the solver's first cycles pick its launch shapes; a program keeps the solver for thousands
    s.set_state_device(W.data_ptr())
    (s.pmg_cycle if case["mode"] == "cycles" else s.explicit_steps)(TUNE_UNITS, record=False)
    return st


def run(state):
    case = state["case"]
    if case["mode"] == "serve":
        srv = state["srv"]
        ids = [srv.submit(g, spec, W, 1e-300, case["n"]) for _, g, spec, W in state["reqs"]]
        while srv.step():
            pass
        done = [srv.poll(i)[1] for i in ids]
        return [_handed_over(case, torch.from_numpy(w)) for w in done]
    s = state["s"]
    s.set_state_device(state["W"].data_ptr())
    res = (s.pmg_cycle if case["mode"] == "cycles" else s.explicit_steps)(case["n"])
    s.get_state_device(state["Wo"].data_ptr(), state["Xo"].data_ptr())
    return dict(W=_handed_over(case, state["Wo"]), Wx=_handed_over(case, state["Xo"]),
                res=_handed_over(case, torch.from_numpy(res)))


def _handed_over(case, x):
    """A mixed-precision solve evaluates its fluxes in FP32, so its fields are
    single precision data and are handed on as such."""
    return x.float() if case["precision"] == "mixed" else x


def work(case):
    if case["mode"] == "serve":
        b = f = 0.0
        for m, g, spec, _ in _requests(case, 1):
            w = _work(dict(case, mode="cycles", limited="flux_hi" in spec), m, g)
            b, f = b + w["bytes"], f + w["flops"]
        return dict(bytes=b, flops=f)
    return _work(case, *_mesh_of(case["flow"], case["a"], case["b"], case["c"]))


def _work(case, m, g):
    """Bytes: state in and out, and the mesh tables once per pass.  Flops of
    the scheme's formulas per Gauss point, face, cell and relaxation."""
    D, nv = m.dim, m.dim + 2
    el = 8 if case["precision"] == "fp64" else 4
    N, F = g.n_cells, g.n_faces
    slots = 3.0 if D == 2 else 4.5
    nq, gp = (5, 2) if D == 2 else (9, 3.3)
    geo = N * (slots * ((D + 1) * nq + D + 3) + nq + 6) + F * (2 * gp * D + D * D + 3)
    byts = geo * el + N * nv * 8 * (2 + D)
    point = (450 if D == 2 else 900) * (4 if case["limited"] else 1)
    ev = F * gp * point + N * 2 * nv * nq * (slots * (D + 1) + D)
    cell = N * slots * nv * 2 * (2 + D)
    evals = 2 if case["scheme"] == "S2O4" else 1
    if case["mode"] == "explicit":
        return dict(bytes=byts, flops=case["n"] * evals * (ev + cell))
    lo = 6 * (F * 110 + N * (40 + slots * 2 * nv) + 8 * N * slots * (16 + 6 * D) / 2)
    return dict(bytes=byts, flops=case["n"] * ((evals + 1) * (ev + cell) + lo))


# ------------------------------------------------------ the scheme in 64 bits
def exact(case, seed):
    if case["mode"] == "serve":
        out = []
        for m, _, spec, W in _requests(case, seed):
            e = _Scheme(m, dict(spec, lo_viscous=1))
            e.set(W)
            e.cycles(case["n"])
            out.append(e.W.cpu().numpy())
        return out
    m, _ = _mesh_of(case["flow"], case["a"], case["b"], case["c"])
    e = _Scheme(m, _spec(case))
    e.set(_state(m, case["flow"], FLOWS[case["flow"]][0], seed))
    res = e.cycles(case["n"]) if case["mode"] == "cycles" else e.steps(case["n"])
    return dict(W=e.W.cpu().numpy(), Wx=e.Wx.cpu().numpy(), res=np.array(res))


# faces of each cell type by node position, counter-clockwise from outside
_FACES = {
    0: [(0, 1), (1, 2), (2, 0)], 1: [(0, 1), (1, 2), (2, 3), (3, 0)],
    2: [(0, 2, 1), (0, 1, 3), (1, 2, 3), (2, 0, 3)],
    3: [(0, 2, 1), (3, 4, 5), (0, 1, 4, 3), (1, 2, 5, 4), (2, 0, 3, 5)],
    4: [(0, 3, 2, 1), (0, 1, 4), (1, 2, 4), (2, 3, 4), (3, 0, 4)],
    5: [(0, 3, 2, 1), (4, 5, 6, 7), (0, 1, 5, 4), (1, 2, 6, 5), (2, 3, 7, 6), (3, 0, 4, 7)],
}
_SIZE = {0: 3, 1: 4, 2: 4, 3: 6, 4: 5, 5: 8}


class _Geometry:
    """Cells, faces, slots and colours of a raw mesh."""

    def __init__(self, mesh):
        D, n = mesh.dim, mesh.n_cells
        self.D, self.n = D, n
        S = 4 if D == 2 else 6
        self.vol, self.xc, self.c2 = np.zeros(n), np.zeros((n, D)), np.zeros((n, D, D))
        keys, cell, slot, nodes = [], [], [], []
        for t, faces in _FACES.items():
            ids = np.nonzero(mesh.cell_type == t)[0]
            if not ids.size or (D == 2) != (t < 2):
                continue
            nd = mesh.cell_nodes[mesh.cell_ptr[ids][:, None] + np.arange(_SIZE[t])]
            self._moments(ids, mesh.nodes[nd], faces)
            for k, f in enumerate(faces):
                q = np.full((ids.size, 4), -1, np.int64)
                q[:, :len(f)] = nd[:, list(f)]
                keys.append(np.sort(q, axis=1)); cell.append(ids); nodes.append(q)
                slot.append(np.full(ids.size, k))
        # a boundary face is the second user of its face, with cell -1 - tag
        nb = mesh.n_bfaces
        ln = np.diff(mesh.bface_ptr)
        q = np.full((nb, 4), -1, np.int64)
        for k in range(int(ln.max()) if nb else 0):
            has = ln > k
            q[has, k] = mesh.bface_nodes[mesh.bface_ptr[:-1][has] + k]
        keys.append(np.sort(q, axis=1)); cell.append(-1 - mesh.bface_tag.astype(np.int64)); nodes.append(q)
        slot.append(np.full(nb, -1))
        keys, cell, slot, nodes = (np.concatenate(v) for v in (keys, cell, slot, nodes))
        order = np.lexsort((-cell, keys[:, 0], keys[:, 1], keys[:, 2], keys[:, 3]))
        first, second = order[0::2], order[1::2]
        assert (keys[first] == keys[second]).all()
        self.c0, self.c1 = cell[first], cell[second]
        nf = self.c0.size
        self.cf, self.sg, self.nbr = np.full((n, S), -1), np.zeros((n, S)), np.full((n, S), -1)
        self.cf[self.c0, slot[first]] = np.arange(nf)
        self.sg[self.c0, slot[first]] = 1.0
        self.nbr[self.c0, slot[first]] = np.maximum(self.c1, -1)
        i = self.c1 >= 0
        self.cf[self.c1[i], slot[second][i]] = np.nonzero(i)[0]
        self.sg[self.c1[i], slot[second][i]] = -1.0
        self.nbr[self.c1[i], slot[second][i]] = self.c0[i]
        self._faces(mesh.nodes, nodes[first])
        self.h = self.vol ** (1.0 / D)
        area = np.zeros(n)
        np.add.at(area, self.c0, self.S)
        np.add.at(area, self.c1[i], self.S[i])
        self.hdt = D * self.vol / area
        self.delta = np.abs(((np.where(i[:, None], self.xc[np.maximum(self.c1, 0)], self.xf) - self.xc[self.c0])
                             * self.nrm).sum(1)) * np.where(i, 1.0, 2.0)
        self.colours = self._colour(i)

    def _moments(self, ids, X, faces):
        D = self.D
        o = X.mean(1)
        X = X - o[:, None]
        simplices = []
        for f in faces:
            P = X[:, list(f)]
            if D == 2 or len(f) == 3:
                simplices.append(P)
            else:
                mid = P.mean(1)
                simplices += [np.stack([P[:, e], P[:, (e + 1) % 4], mid], 1) for e in range(4)]
        V, S1, S2 = 0.0, 0.0, 0.0
        for P in simplices:                                   # with the origin as further vertex
            v = np.linalg.det(P) / math.factorial(D)
            s = P.sum(1)
            V = V + v
            S1 = S1 + v[:, None] * s / (D + 1)
            S2 = S2 + (v / ((D + 1) * (D + 2)))[:, None, None] * (
                s[:, :, None] * s[:, None, :] + np.einsum("mki,mkj->mij", P, P))
        c = S1 / V[:, None]
        self.vol[ids], self.xc[ids] = V, o + c
        self.c2[ids] = S2 / V[:, None, None] - c[:, :, None] * c[:, None, :]

    def _faces(self, X, nodes):
        D, nf = self.D, nodes.shape[0]
        G = 2 if D == 2 else 4
        self.nrm, self.S, self.xf = np.zeros((nf, D)), np.zeros(nf), np.zeros((nf, D))
        self.xg, self.w = np.zeros((nf, G, D)), np.zeros((nf, G))
        if D == 2:
            a, b = X[nodes[:, 0]], X[nodes[:, 1]]
            d = b - a
            self.S = np.hypot(d[:, 0], d[:, 1])
            self.nrm = np.stack([d[:, 1], -d[:, 0]], 1) / self.S[:, None]
            g = 0.5 / math.sqrt(3.0)
            self.xg = np.stack([a + (0.5 - g) * d, a + (0.5 + g) * d], 1)
            self.w[:] = 0.5
            self.xf = 0.5 * (a + b)
            return
        tri = np.nonzero(nodes[:, 3] < 0)[0]
        P = X[nodes[tri][:, :3]]
        A = np.zeros((nf, 3))
        A[tri] = 0.5 * np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
        self.xf[tri] = P.mean(1)
        self.xg[tri] = self.xf[tri][:, None]
        self.xg[tri, :3] = (3.0 * P + P.sum(1, keepdims=True)) / 6.0
        self.w[tri, :3] = 1.0 / 3.0
        qd = np.nonzero(nodes[:, 3] >= 0)[0]
        P = X[nodes[qd]]
        self.xf[qd] = P.mean(1)
        g = 1.0 / math.sqrt(3.0)
        sx, sy = np.array([-1, 1, 1, -1.0]), np.array([-1, -1, 1, 1.0])
        for k in range(4):
            s, t = sx[k] * g, sy[k] * g
            self.xg[qd, k] = np.einsum("a,mad->md", 0.25 * (1 + sx * s) * (1 + sy * t), P)
            c = np.cross(np.einsum("a,mad->md", 0.25 * sx * (1 + sy * t), P),
                         np.einsum("a,mad->md", 0.25 * sy * (1 + sx * s), P))
            A[qd] += c
            self.w[qd, k] = np.linalg.norm(c, axis=1)
        self.w[qd] /= self.w[qd].sum(1, keepdims=True)
        self.S = np.linalg.norm(A, axis=1)
        self.nrm = A / self.S[:, None]

    def _colour(self, inner):
        """Greedy colouring in the reverse Cuthill-McKee order (start: lowest
        index of least degree; neighbours by degree, then index)."""
        n = self.n
        adj = [[int(j) for j in row if j >= 0] for row in self.nbr]
        deg = np.array([len(a) for a in adj])
        rank = (deg * n + np.arange(n)).tolist()
        seen, cm = bytearray(n), []
        for start in np.argsort(deg, kind="stable").tolist():
            if seen[start]:
                continue
            seen[start] = 1
            head = len(cm)
            cm.append(start)
            while head < len(cm):
                nb = [w for w in adj[cm[head]] if not seen[w]]
                head += 1
                if nb:
                    nb.sort(key=rank.__getitem__)
                    for w in nb:
                        seen[w] = 1
                    cm += nb
        colour = [-1] * n
        for v in reversed(cm):
            used = {colour[w] for w in adj[v]}
            c = 0
            while c in used:
                c += 1
            colour[v] = c
        colour = np.array(colour)
        return [np.nonzero(colour == c)[0] for c in range(colour.max() + 1)]


_GEOMETRY = {}


class _Scheme:
    """High-order step, low-order relaxation and V-cycle; states are [n, D + 2], gradients [n, D, D + 2]."""

    def __init__(self, mesh, spec):
        if id(mesh) not in _GEOMETRY:
            _GEOMETRY.clear()
            _GEOMETRY[id(mesh)] = (mesh, _Geometry(mesh))
        G = self.G = _GEOMETRY[id(mesh)][1]
        self.spec, self.D = spec, G.D
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        f, i = self._f, self._i
        D = G.D
        self.vol, self.h, self.hdt, self.xc = f(G.vol), f(G.h), f(G.hdt), f(G.xc)
        self.M = f(G.c2 / (G.h ** 2)[:, None, None])
        self.c0, self.c1, self.nb, self.cf, self.sg = i(G.c0), i(G.c1), i(G.nbr), i(G.cf), f(G.sg)
        self.nrm, self.S, self.xg, self.w = f(G.nrm), f(G.S), f(G.xg), f(G.w)
        self.has = self.cf >= 0
        self.cfz = self.cf.clamp(min=0)
        self.inner = self.c1 >= 0
        self.colours = [i(c) for c in G.colours]
        self.gamma = g = spec["gamma"]
        self.K = 2.0 / (g - 1.0) - D
        self.mu = spec["mu"]
        self.ajump, self.idl = 0.5 / f(G.delta), 1.0 / f(G.delta)
        # orthonormal frame of every face, first row the normal
        e = torch.zeros(self.S.numel(), D, D, dtype=torch.float64, device=self.dev)
        e[:, 0] = self.nrm
        if D == 2:
            e[:, 1, 0], e[:, 1, 1] = -self.nrm[:, 1], self.nrm[:, 0]
        else:
            a = torch.zeros_like(self.nrm)
            a.scatter_(1, self.nrm.abs().argmin(1, keepdim=True), 1.0)
            t = torch.linalg.cross(a, self.nrm)
            e[:, 1] = t / t.norm(dim=1, keepdim=True)
            e[:, 2] = torch.linalg.cross(self.nrm, e[:, 1])
        self.e = e
        tag = np.where(G.c1 < 0, -1 - G.c1, 0)
        kind = np.array([b["kind"] for b in spec["bcs"]])[tag]
        self.kind = {k: i(np.nonzero((kind == k) & (G.c1 < 0))[0])
                     for k in ("slip", "noslip", "farfield", "dirichlet", "outflow")}

        def table(key, default, width):
            rows = [np.resize(np.append(np.asarray(b.get(key, default), float), np.zeros(3)), width) for b in spec["bcs"]]
            return f(np.array(rows)[tag])
        self.bu, self.buw = table("u", (0.0,), D), table("uw", (0.0,), D)
        self.brho = f(np.array([b.get("rho", 1.0) for b in spec["bcs"]])[tag])
        self.bp = f(np.array([b.get("p", 1.0 / g) for b in spec["bcs"]])[tag])
        self.wallface = torch.zeros(self.S.numel(), dtype=torch.bool, device=self.dev)
        for k in ("slip", "noslip"):
            self.wallface[self.kind[k]] = True
        self.pairs = [(a, b) for a in range(D) for b in range(a, D)]
        self._operator()

    def _f(self, x):
        return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=self.dev)

    def _i(self, x):
        return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.int64, device=self.dev)

    # -------- primitives
    def prim(self, W):
        D = self.D
        u = W[..., 1:1 + D] / W[..., :1]
        p = (self.gamma - 1.0) * (W[..., D + 1] - 0.5 * W[..., 0] * (u * u).sum(-1))
        return W[..., 0], u, p

    def cons(self, r, u, p):
        E = p / (self.gamma - 1.0) + 0.5 * r * (u * u).sum(-1)
        return torch.cat([r[..., None], r[..., None] * u, E[..., None]], -1)

    # -------- least-squares quadratic
    def _operator(self):
        D, n = self.D, self.vol.numel()
        Sn = self.nb.shape[1]
        nq = D + len(self.pairs)
        rows = Sn * (D + 1) + D
        A = torch.zeros(n, rows, nq, dtype=torch.float64, device=self.dev)
        T = torch.zeros(n, D, D, dtype=torch.float64, device=self.dev)
        h = self.h[:, None]
        mean = lambda C: torch.stack([C[:, a, b] for a, b in self.pairs], 1)  # noqa: E731
        count = torch.zeros(n, dtype=torch.int64, device=self.dev)
        eye = torch.eye(D, dtype=torch.float64, device=self.dev)
        self.slot = []
        for s in range(Sn):
            j, fz = self.nb[:, s], self.cfz[:, s]
            wall = self.has[:, s] & (j < 0) & self.wallface[fz]
            use = (j >= 0) | wall
            self.slot.append((use, wall))
            jz = j.clamp(min=0)
            nr = self.nrm[fz]
            d = self.xc[jz] - self.xc
            off = ((self.xc - self.xg[fz, 0]) * nr).sum(1, keepdim=True)
            d = torch.where(wall[:, None], -2.0 * off * nr, d) / h
            C = self.M[jz] * (self.h[jz] / self.h)[:, None, None] ** 2
            R = eye - 2.0 * nr[:, :, None] * nr[:, None, :]
            C = torch.where(wall[:, None, None], R @ self.M @ R, C)
            m = use.double()[:, None]
            r0 = s * (D + 1)
            A[:, r0, :D] = d * m
            A[:, r0, D:] = (mean(C + d[:, :, None] * d[:, None, :]) - mean(self.M)) * m
            for k in range(D):
                A[:, r0 + 1 + k, k] = m[:, 0]
                for q, (a, b) in enumerate(self.pairs):
                    A[:, r0 + 1 + k, D + q] = ((a == k) * d[:, b] + (b == k) * d[:, a]) * m[:, 0]
            T += m[:, :, None] * d[:, :, None] * d[:, None, :]
            count += use
        for k in range(D):
            A[:, Sn * (D + 1) + k, k] = 1.0
        if D == 2:
            quad = count >= 2
        else:
            tr = T.diagonal(dim1=1, dim2=2).sum(1)
            quad = (count >= 3) & (torch.linalg.det(T) >= 1e-3 * tr ** 3 / 27.0) & (tr > 0)
        # modified Gram-Schmidt, then back substitution
        Q = [A[:, :, q].clone() for q in range(nq)]
        R = [[None] * nq for _ in range(nq)]
        for q in range(nq):
            for k in range(q):
                R[k][q] = (Q[k] * Q[q]).sum(1, keepdim=True)
                Q[q] = Q[q] - R[k][q] * Q[k]
            R[q][q] = Q[q].norm(dim=1, keepdim=True)
            quad = quad & (R[q][q][:, 0] > 1e-13)
            Q[q] = Q[q] / R[q][q]
        X = [None] * nq
        for q in reversed(range(nq)):
            X[q] = (Q[q] - sum((R[q][k] * X[k] for k in range(q + 1, nq)), torch.zeros_like(Q[q]))) / R[q][q]
        op = torch.stack(X, 1)                                # [n, nq, rows]
        lin = torch.zeros_like(op)
        for k in range(D):
            lin[:, k, Sn * (D + 1) + k] = 1.0
        op = torch.where(quad[:, None, None], op, lin)
        grad = torch.ones(rows, dtype=torch.float64, device=self.dev)
        grad[:Sn * (D + 1):D + 1] = 0.0
        self.op = op * torch.where(grad > 0, self.h[:, None, None], torch.ones_like(self.h)[:, None, None])
        self.quad = quad

    def mirror(self, fz, W, Wx):
        """Mean and gradient of the mirror cell across wall faces fz."""
        D = self.D
        nr = self.nrm[fz]
        R = torch.eye(D, dtype=torch.float64, device=self.dev) - 2.0 * nr[:, :, None] * nr[:, None, :]
        slip = torch.zeros(self.S.numel(), dtype=torch.bool, device=self.dev)
        slip[self.kind["slip"]] = True
        slip = slip[fz]

        def reflect(x):
            return torch.cat([x[..., :1], torch.einsum("nab,n...b->n...a", R, x[..., 1:1 + D]), x[..., D + 1:]], -1)
        Ws = reflect(W)
        gs = torch.einsum("nde,nev->ndv", R, reflect(Wx))
        r, u, p = self.prim(W)
        dr = Wx[..., 0]
        du = (Wx[..., 1:1 + D] - u[:, None] * dr[..., None]) / r[:, None, None]
        dp = (self.gamma - 1.0) * (Wx[..., D + 1] - 0.5 * (u * u).sum(-1)[:, None] * dr
                                   - r[:, None] * (u[:, None] * du).sum(-1))
        ug = 2.0 * self.buw[fz] - u
        dr, dp = torch.einsum("nde,ne->nd", R, dr), torch.einsum("nde,ne->nd", R, dp)
        du = -torch.einsum("nde,nea->nda", R, du)
        Wn = self.cons(r, ug, p)
        gn = torch.cat([dr[..., None], ug[:, None] * dr[..., None] + r[:, None, None] * du,
                        (dp / (self.gamma - 1.0) + 0.5 * (ug * ug).sum(-1)[:, None] * dr
                         + r[:, None] * (ug[:, None] * du).sum(-1))[..., None]], -1)
        return torch.where(slip[:, None], Ws, Wn), torch.where(slip[:, None, None], gs, gn)

    def weno(self, c, M, lin, on, apply):
        """Nonlinear weights: c [n, nq, v], candidates lin [k][n, D, v] (on: which exist)."""
        D, eps, g0 = self.D, self.spec["weno_eps"], self.spec.get("weno_g0", 0.95)
        H = torch.zeros(c.shape[0], D, D, c.shape[2], dtype=torch.float64, device=self.dev)
        b0 = (c[:, :D] ** 2).sum(1)
        for q, (a, b) in enumerate(self.pairs):
            x = c[:, D + q]
            if a == b:
                H[:, a, a] = 2.0 * x
                b0 = b0 + 4.0 * x * x
            else:
                H[:, a, b] = H[:, b, a] = x
                b0 = b0 + x * x
        b0 = b0 + torch.einsum("ndav,nae,ndev->nv", H, M, H)
        nk = sum(o.double() for o in on)[:, None]
        gk = (1.0 - g0) / nk
        w0 = g0 / (b0 + eps) ** 2
        wk = [o[:, None] * gk / ((x * x).sum(1) + eps) ** 2 for x, o in zip(lin, on)]
        ws = w0 + sum(wk)
        l1 = sum((o[:, None] * gk)[:, None] * x for x, o in zip(lin, on))
        sel = sum((w / ws)[:, None] * x for x, w in zip(lin, wk))
        f0 = (w0 / ws / g0)[:, None]
        out = torch.cat([f0 * (c[:, :D] - l1) + sel, f0 * c[:, D:]], 1)
        return torch.where(apply[:, None, None], out, c)

    def recon(self, W, Wx):
        D = self.D
        B, lin, on = [], [self.h[:, None, None] * Wx], [torch.ones_like(self.h, dtype=torch.bool)]
        for s, (use, wall) in enumerate(self.slot):
            jz = self.nb[:, s].clamp(min=0)
            Wj, gj = W[jz], Wx[jz]
            k = wall.nonzero()[:, 0]
            if k.numel():
                Wj[k], gj[k] = self.mirror(self.cfz[k, s], W[k], Wx[k])
            B += [((Wj - W) * use[:, None])[:, None], gj * use[:, None, None]]
            lin.append(self.h[:, None, None] * gj)
            on.append(self.nb[:, s] >= 0)
        c = torch.einsum("nqr,nrv->nqv", self.op, torch.cat(B + [Wx], 1))
        if self.spec.get("weno_eps", 0.0) > 0.0 and self.spec["weno_vars"] == "conservative":
            c = self.weno(c, self.M, lin, on, self.quad)
        return c

    def char_side(self, c, i, Wx, wref):
        """Polynomial of cells i limited in the characteristic variables of faces (all faces in order), 2-D."""
        nx, ny = self.nrm[:, 0], self.nrm[:, 1]
        r, u, p = self.prim(wref)
        a = torch.sqrt(self.gamma * p / r)
        H = (wref[:, 3] + p) / r
        q2 = (u * u).sum(1)
        un = u[:, 0] * nx + u[:, 1] * ny
        ut = -u[:, 0] * ny + u[:, 1] * nx
        one, zero = torch.ones_like(a), torch.zeros_like(a)
        R = torch.stack([torch.stack(x, 1) for x in (
            (one, one, zero, one), (u[:, 0] - a * nx, u[:, 0], -ny, u[:, 0] + a * nx),
            (u[:, 1] - a * ny, u[:, 1], nx, u[:, 1] + a * ny), (H - a * un, 0.5 * q2, ut, H + a * un))], 1)
        L = torch.linalg.inv(R)
        project = lambda x: torch.einsum("nab,nkb->nka", L, x)  # noqa: E731
        h = self.h[i][:, None, None]
        lin, on = [h * project(Wx[i])], [torch.ones_like(a, dtype=torch.bool)]
        for s in range(self.nb.shape[1]):
            j = self.nb[i, s]
            lin.append(h * project(Wx[j.clamp(min=0)]))
            on.append(j >= 0)
        out = self.weno(project(c[i]), self.M[i], lin, on, torch.ones_like(on[0]))
        out = torch.einsum("nab,nkb->nka", R, out)
        return torch.where(self.quad[i][:, None, None], out, c[i])

    def side(self, c, i, W, x):
        """Value and gradient at x of the polynomials c of cells i."""
        D = self.D
        xi = (x - self.xc[i]) / self.h[i][:, None]
        M = self.M[i]
        val, g = W[i].clone(), [c[:, k].clone() for k in range(D)]
        for k in range(D):
            val = val + c[:, k] * xi[:, k, None]
        for q, (a, b) in enumerate(self.pairs):
            val = val + c[:, D + q] * (xi[:, a] * xi[:, b] - M[:, a, b])[:, None]
            g[a] = g[a] + c[:, D + q] * xi[:, b, None]
            g[b] = g[b] + c[:, D + q] * xi[:, a, None]
        return val, torch.stack(g, 1) / self.h[i][:, None, None]

    def to_local(self, x):
        D = self.D
        return torch.cat([x[..., :1], torch.einsum("nab,n...b->n...a", self.e, x[..., 1:1 + D]), x[..., D + 1:]], -1)

    def to_global(self, x):
        D = self.D
        return torch.cat([x[..., :1], torch.einsum("nab,n...a->n...b", self.e, x[..., 1:1 + D]), x[..., D + 1:]], -1)

    def farfield(self, k, Wi):
        """Riemann-invariant state at far-field faces k from the inside state (local frame)."""
        g = self.gamma
        ri, ui, pi = self.prim(Wi)
        ue = torch.einsum("nab,nb->na", self.e[k], self.bu[k])
        re, pe = self.brho[k], self.bp[k]
        ci, ce = torch.sqrt(g * pi / ri), torch.sqrt(g * pe / re)
        Rp, Rm = ui[:, 0] + 2 * ci / (g - 1), ue[:, 0] - 2 * ce / (g - 1)
        un, cb = 0.5 * (Rp + Rm), 0.25 * (g - 1) * (Rp - Rm)
        out = un >= 0
        s = torch.where(out, pi / ri ** g, pe / re ** g)
        ub = torch.where(out[:, None], ui, ue).clone()
        ub[:, 0] = un
        rb = (cb * cb / (g * s)) ** (1.0 / (g - 1))
        pb = rb * cb * cb / g
        for cond, (r, u, p) in ((ui[:, 0] <= -ci, (re, ue, pe)), (ui[:, 0] >= ci, (ri, ui, pi))):
            rb, pb, ub = torch.where(cond, r, rb), torch.where(cond, p, pb), torch.where(cond[:, None], u, ub)
        return self.cons(rb, ub, pb)

    def ghosts(self, W, wl, dl, wr, dr):
        """Outside states (local frame) of the boundary faces; dl, dr [nf, D, v] or None for cell means."""
        D = self.D
        k = self.kind["outflow"]
        wr[k] = wl[k]
        if dr is not None:
            dr[k] = dl[k]
        for name in ("farfield", "dirichlet"):
            k = self.kind[name]
            if k.numel():
                if name == "farfield":
                    mean = W[self.c0[k]]
                    wi = torch.cat([mean[:, :1], torch.einsum("nab,nb->na", self.e[k], mean[:, 1:1 + D]),
                                    mean[:, D + 1:]], 1)
                    wr[k] = self.farfield(k, wi)
                else:
                    wr[k] = self.cons(self.brho[k], torch.einsum("nab,nb->na", self.e[k], self.bu[k]), self.bp[k])
                if dr is not None:
                    dr[k] = 0.0
        flip = torch.ones(D, dtype=torch.float64, device=self.dev)
        flip[0] = -1.0
        k = self.kind["slip"]
        if k.numel():
            sign = torch.ones(D + 2, dtype=torch.float64, device=self.dev)
            sign[1] = -1.0
            wr[k] = wl[k] * sign
            if dr is not None:
                dr[k] = dl[k] * sign * flip[:, None]
        k = self.kind["noslip"]
        if k.numel():
            r, u, p = self.prim(wl[k])
            ug = 2.0 * torch.einsum("nab,nb->na", self.e[k], self.buw[k]) - u
            wr[k] = self.cons(r, ug, p)
            if dr is not None:
                d = dl[k]
                rho = d[..., 0]
                du = (d[..., 1:1 + D] - u[:, None] * rho[..., None]) / r[:, None, None]
                dp = (self.gamma - 1) * (d[..., D + 1] - 0.5 * (u * u).sum(-1)[:, None] * rho
                                         - r[:, None] * (u[:, None] * du).sum(-1))
                rho, dp, du = flip * rho, flip * dp, -flip[:, None] * du
                dr[k] = torch.cat([rho[..., None], ug[:, None] * rho[..., None] + r[:, None, None] * du,
                                   (dp / (self.gamma - 1) + 0.5 * (ug * ug).sum(-1)[:, None] * rho
                                    + r[:, None] * (ug[:, None] * du).sum(-1))[..., None]], -1)
        return wr, dr

    # -------- kinetic moments; a Maxwellian is (rho, U [n, D], th = 1 / (2 lambda))
    def maxw(self, W):
        r, u, p = self.prim(W)
        return r, u, p / r

    def table(self, u, th, half=0):
        """Moments of each velocity component (the normal one over a half range for half = +-1) and of xi."""
        m = []
        for k in range(self.D):
            U = u[:, k]
            if k == 0 and half:
                z = U / torch.sqrt(2.0 * th)
                a = [0.5 * torch.special.erfc(-half * z)]
                a.append(U * a[0] + half * 0.5 * torch.exp(-z * z) * torch.sqrt(2.0 * th / math.pi))
            else:
                a = [torch.ones_like(U), U]
            for q in range(2, 7):
                a.append(U * a[q - 1] + (q - 1) * th * a[q - 2])
            m.append(a)
        return m, [torch.ones_like(th), self.K * th, self.K * (self.K + 2) * th * th]

    def mom(self, t, powers, d, s):
        """<u^powers xi^(2d) (s0 + s.u + s_E (u^2 + xi^2) / 2)>, s [n, v] or None for 1."""
        m, x = t

        def base(p, dd):
            out = x[dd]
            for k in range(self.D):
                out = out * m[k][p[k]]
            return out
        if s is None:
            return base(powers, d)
        up = lambda k, q: tuple(v + (q if a == k else 0) for a, v in enumerate(powers))  # noqa: E731
        out = s[:, 0] * base(powers, d) + 0.5 * s[:, self.D + 1] * base(powers, d + 1)
        for k in range(self.D):
            out = out + s[:, 1 + k] * base(up(k, 1), d) + 0.5 * s[:, self.D + 1] * base(up(k, 2), d)
        return out

    def psi(self, t, powers, s):
        up = lambda k, q: tuple(v + (q if a == k else 0) for a, v in enumerate(powers))  # noqa: E731
        E = self.mom(t, powers, 1, s)
        for k in range(self.D):
            E = E + self.mom(t, up(k, 2), 0, s)
        return torch.stack([self.mom(t, powers, 0, s)] + [self.mom(t, up(k, 1), 0, s) for k in range(self.D)]
                           + [0.5 * E], 1)

    def slopes(self, g, d):
        """Spatial slopes from local derivatives d [n, D, v], and the temporal one."""
        r, U, th = g
        q = (U * U).sum(1) + (self.K + self.D) * th

        def solve(b):
            RE = 2.0 * b[:, -1] - q * b[:, 0]
            Rk = b[:, 1:-1] - U * b[:, :1]
            sE = (RE - 2.0 * (U * Rk).sum(1)) / ((self.K + self.D) * th * th)
            sk = Rk / th[:, None] - U * sE[:, None]
            s0 = b[:, 0] - (U * sk).sum(1) - 0.5 * sE * q
            return torch.cat([s0[:, None], sk, sE[:, None]], 1)
        a = [solve(d[:, k] / r[:, None]) for k in range(self.D)]
        t = self.table(U, th)
        unit = [tuple(int(k == m) for k in range(self.D)) for m in range(self.D)]
        return a, solve(-sum(self.psi(t, unit[k], a[k]) for k in range(self.D)))

    def piece(self, r, t, a, A):
        """rho-weighted (<u psi>, <u a.u psi>, <u A psi>) and (<psi>, <a.u psi>, <A psi>)."""
        zero = (0,) * self.D
        n1 = tuple(int(k == 0) for k in range(self.D))
        add = lambda p, k: tuple(v + int(m == k) for m, v in enumerate(p))  # noqa: E731
        out = []
        for p in (n1, zero):
            out.append([r[:, None] * x for x in (
                self.psi(t, p, None), sum(self.psi(t, add(p, k), a[k]) for k in range(self.D)), self.psi(t, p, A))])
        return out

    def flux(self, wl, wr, dl, dr, dt):
        """F0, F1, Wc, Wt at one Gauss point of every face, local frame."""
        gl, gr = self.maxw(wl), self.maxw(wr)
        tl, tr = self.table(gl[1], gl[2], 1), self.table(gr[1], gr[2], -1)
        zero = (0,) * self.D
        Wc = gl[0][:, None] * self.psi(tl, zero, None) + gr[0][:, None] * self.psi(tr, zero, None)
        gc = self.maxw(Wc)
        d = 0.5 * (dl + dr)
        d[:, 0] += self.ajump[:, None] * (wr - wl)
        a, A = self.slopes(gc, d)
        Q0, P0 = self.piece(gc[0], self.table(gc[1], gc[2]), a, A)
        tau = (self.mu / (gc[0] * gc[2]))[:, None]
        if self.spec.get("flux_hi", "smooth") == "smooth":
            return Q0[0] - tau * (Q0[1] + Q0[2]), Q0[2], Wc, P0[2]
        QL, PL = self.piece(gl[0], tl, *self.slopes(gl, dl))
        QR, PR = self.piece(gr[0], tr, *self.slopes(gr, dr))
        pl, pr = gl[0] * gl[2], gr[0] * gr[2]
        tn = tau + (0.01 * dt + dt * (pl - pr).abs() / (pl + pr))[:, None]
        res = []
        for X0, XL, XR, integral in ((Q0, QL, QR, True), (P0, PL, PR, False)):
            s = [x + y for x, y in zip(XL, XR)]
            at = []
            for t in (dt, 0.5 * dt):
                e, om = torch.exp(-t / tn), -torch.expm1(-t / tn)
                if integral:
                    ie = tn * om
                    ite = tn * tn * om - tn * t * e
                    c = (t - ie, ite + tau * ie - tau * t, 0.5 * t * t - tau * t + tau * ie, ie, ite)
                else:
                    c = (1 - e, (t + tau) * e - tau, t - tau + tau * e, e, t * e)
                at.append(c[0] * X0[0] + c[1] * X0[1] + c[2] * X0[2]
                          + c[3] * (s[0] - tau * s[1] - tau * s[2]) - c[4] * s[1])
            full, half = at
            res += ([(4 * half - full) / dt, 4 * (full - 2 * half) / dt ** 2] if integral
                    else [2 * half - full, 2 * (full - half) / dt])
        return res

    def evaluate(self, W, Wx, dt):
        c = self.recon(W, Wx)
        i0, i1 = self.c0, torch.where(self.inner, self.c1, self.c0)
        if self.spec.get("weno_eps", 0.0) > 0.0 and self.spec["weno_vars"] == "characteristic":
            wref = 0.5 * (W[i0] + W[i1])
            cl, cr = self.char_side(c, i0, Wx, wref), self.char_side(c, i1, Wx, wref)
        else:
            cl, cr = c[i0], c[i1]
        out = None
        for k in range(self.w.shape[1]):
            pts = []
            for i, cc in ((i0, cl), (i1, cr)):
                v, g = self.side(cc, i, W, self.xg[:, k])
                pts += [self.to_local(v), self.to_local(torch.einsum("nad,ndv->nav", self.e, g))]
            wl, dl, wr, dr = pts
            wr, dr = self.ghosts(W, wl, dl, wr, dr)
            f = [self.w[:, k, None] * self.to_global(x) for x in self.flux(wl, wr, dl, dr, dt)]
            out = f if out is None else [x + y for x, y in zip(out, f)]
        return out

    def gather(self, F):
        """sum over a cell's faces of sgn S F."""
        out = torch.zeros(self.vol.numel(), *F.shape[1:], dtype=torch.float64, device=self.dev)
        for s in range(self.cf.shape[1]):
            wgt = self.sg[:, s] * self.S[self.cfz[:, s]]
            out += wgt.view(-1, *[1] * (F.dim() - 1)) * F[self.cfz[:, s]]
        return out

    def set(self, W):
        self.W = self._f(W)
        self.Wx = torch.zeros(W.shape[0], self.D, self.D + 2, dtype=torch.float64, device=self.dev)

    def time_step(self):
        r, u, p = self.prim(self.W)
        speed = u.norm(dim=1) + torch.sqrt(self.gamma * p / r) + 2.0 * (self.mu / r) / self.hdt
        return self.spec["cfl_hi"] * (self.hdt / speed).min()

    def high(self, dt):
        """One high-order step: (W, Wx) at the new time."""
        def grad(Wp):
            return self.gather(self.nrm[:, :, None] * Wp[:, None]) / self.vol[:, None, None]
        k = (dt / self.vol)[:, None]
        A = self.evaluate(self.W, self.Wx, dt)
        if self.spec["time_scheme"] == "S1O2":
            return self.W - k * self.gather(A[0] + 0.5 * dt * A[1]), grad(A[2] + dt * A[3])
        Ws = self.W - k * self.gather(0.5 * A[0] + 0.125 * dt * A[1])
        B = self.evaluate(Ws, grad(A[2] + 0.5 * dt * A[3]), dt)
        return self.W - k * self.gather(A[0] + dt / 6.0 * (A[1] + 2.0 * B[1])), grad(A[2] + dt * B[3])

    def steps(self, n):
        res = []
        for _ in range(n):
            old = self.W
            self.W, self.Wx = self.high(self.time_step())
            res.append(float((self.W[:, 0] - old[:, 0]).abs().sum() / old[:, 0].sum()))
        return res

    # -------- low-order level
    def euler(self, W, nr):
        D = self.D
        r, u, p = self.prim(W)
        un = (u * nr).sum(-1, keepdim=True)
        F = W * un
        F[..., 1:1 + D] += p[..., None] * nr
        F[..., D + 1:] += p[..., None] * un
        return F

    def low_flux(self, U):
        D, g = self.D, self.gamma
        wl = self.to_local(U[self.c0])
        wr = self.to_local(U[torch.where(self.inner, self.c1, self.c0)])
        wr, _ = self.ghosts(U, wl, None, wr, None)
        (rl, ul, pl), (rr, ur, pr) = self.prim(wl), self.prim(wr)
        v0 = self.vol[self.c0]
        v1 = torch.where(self.inner, self.vol[self.c1.clamp(min=0)], v0)
        lam = torch.maximum(ul[:, 0].abs() + torch.sqrt(g * pl / rl) + 2 * (self.mu / rl) * self.S / v0,
                            ur[:, 0].abs() + torch.sqrt(g * pr / rr) + 2 * (self.mu / rr) * self.S / v1)
        n1 = torch.zeros_like(ul)
        n1[:, 0] = 1.0
        if self.spec["flux_lo"] == "lf":
            F = 0.5 * (self.euler(wl, n1) + self.euler(wr, n1)) - 0.5 * lam[:, None] * (wr - wl)
        else:
            p1 = tuple(int(k == 0) for k in range(D))
            F = (rl[:, None] * self.psi(self.table(ul, pl / rl, 1), p1, None)
                 + rr[:, None] * self.psi(self.table(ur, pr / rr, -1), p1, None))
        if self.spec.get("lo_viscous") and self.mu > 0:
            md = (self.mu * self.idl)[:, None]
            du = ur - ul
            tau = md * (du + du[:, :1] / 3.0 * n1)
            qn = -md[:, 0] * g / (g - 1) * (pr / rr - pl / rl)
            F = F.clone()
            F[:, 1:1 + D] -= tau
            F[:, D + 1] -= (tau * 0.5 * (ul + ur)).sum(1) - qn
        return self.to_global(F), lam

    def relax(self, U, R, lam):
        sp = self.spec
        tot = self.gather((lam * 1.0)[:, None]) * 0.0
        for s in range(self.cf.shape[1]):
            tot[:, 0] += torch.where(self.has[:, s], lam[self.cfz[:, s]] * self.S[self.cfz[:, s]], 0.0)
        D = tot / sp["cfl_lo"] + 0.5 * tot
        dU = torch.zeros_like(U)
        order = list(range(len(self.colours)))
        for c in (order + order[::-1]) * sp["n_sweeps"]:
            i = self.colours[c]
            acc = R[i].clone()
            for s in range(self.cf.shape[1]):
                j, f = self.nb[i, s], self.cfz[i, s]
                on = (j >= 0).double()[:, None]
                jz = j.clamp(min=0)
                nr = self.nrm[f] * self.sg[i, s, None]
                d = dU[jz]
                t = self.euler(U[jz] + d, nr) - self.euler(U[jz], nr) - lam[f][:, None] * d
                acc -= on * 0.5 * self.S[f][:, None] * t
            dU[i] = acc / D[i]
        return dU

    def cycles(self, n):
        res = []
        for _ in range(n):
            old, dt = self.W, self.time_step()
            Wn, self.Wx = self.high(dt)
            A = self.evaluate(Wn, self.Wx, dt)
            Rp0 = -self.gather(A[0] + 0.5 * dt * A[1])
            U, src = Wn, None
            for _ in range(self.spec["n_implicit"]):
                F, lam = self.low_flux(U)
                R = -self.gather(F)
                src = Rp0 - R if src is None else src
                U = U + self.relax(U, R + src, lam)
            self.W = U
            res.append(float((U[:, 0] - old[:, 0]).abs().sum() / old[:, 0].sum()))
        return res
