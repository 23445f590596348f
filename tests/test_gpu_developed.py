"""Parity on developed flow at full size (FP64 against the CPU oracle).

The 57,344-cell cylinder of the benchmark, started from the free stream
plus a seeded smooth perturbation (so every cell carries gradients from the
first cycle), run for 20 V-cycles in the launch configuration the benchmark
times; and a 3-D sphere shell of 30,720 cells (icosphere level 3, 12 prism
and 4 split-tet layers) for 5 V-cycles.  Residual histories within 1e-9,
the fields within 1e-12 relative L2 (W) per the FP64 bar."""
import math

import numpy as np
import pytest

from paper_2109_09965_gb300 import meshgen as MG
from tests import exact

pytestmark = pytest.mark.gpu
GAM = 1.4
TOL = 1e-12


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def node_centroids(mesh):
    ptr = mesh.cell_ptr
    return np.add.reduceat(mesh.nodes[mesh.cell_nodes], ptr[:-1], axis=0) / np.diff(ptr)[:, None]


def perturbed(mesh, vel, amp, seed):
    """Free stream plus a smooth seeded perturbation at the cell centres,
    its analytic gradient as the cell gradients."""
    rng = np.random.default_rng(seed)
    dim = mesh.nodes.shape[1]
    k = rng.uniform(0.8, 2.0, dim)
    ph = rng.uniform(0.0, 1.0, dim)
    x = node_centroids(mesh)

    def f(x):
        s = amp * np.prod([np.sin(k[d] * x[:, d] + ph[d]) for d in range(dim)], axis=0)
        rho, p = 1.0 + s, (1.0 + 0.7 * s) / GAM
        u = [vel[d] + (0.5, -0.3, 0.2)[d] * s for d in range(dim)]
        ke = 0.5 * rho * sum(ud * ud for ud in u)
        return np.stack([rho] + [rho * ud for ud in u] + [p / (GAM - 1) + ke], -1)
    h = 1e-6
    Wx = np.stack([(f(x + h * e) - f(x - h * e)) / (2 * h) for e in np.eye(dim)], axis=1)
    return f(x), Wx


@pytest.fixture(scope="module")
def libs(oracle_lib):
    from oracle import oracle3
    from paper_2109_09965_gb300 import cgks
    oracle3.build()
    cgks.lib()
    return cgks, oracle_lib, oracle3


def test_cylinder_57344_developed_flow_20_cycles(libs):
    cgks, O, _ = libs
    mesh = MG.cylinder(256, 32, 96)
    assert mesh.n_cells == 57344
    ma = 0.38
    spec = dict(gamma=GAM, mu=0.0, cfl_hi=0.4, cfl_lo=1000.0, n_implicit=6, n_sweeps=2, time_scheme="S1O2",
                bcs=[dict(kind="slip"), dict(kind="farfield", rho=1.0, u=(ma, 0.0), p=1 / GAM)])
    W, Wx = perturbed(mesh, (ma, 0.0), 0.04, seed=57)
    g = cgks.Solver(cgks.Mesh(mesh), spec)
    o = O.OracleSolver(O.OracleMesh(mesh), spec)
    g.set_state(W, Wx)
    o.set_state(W, Wx)
    hg, ho = g.pmg_cycle(20), o.pmg_cycles(20)
    Wg, Xg = g.get_state()
    Wo, Xo = o.get_state()
    eW, eX = rel(Wg, Wo), rel(Xg, Xo)
    print(f"57k developed: rel W {eW:.2e}  Wx {eX:.2e}  Res {np.abs(hg / ho - 1).max():.2e}")
    np.testing.assert_allclose(hg, ho, rtol=1e-9)
    assert eW < TOL, eW
    assert eX < TOL, eX
    assert rel(W, Wo) > 1e-4          # the field did change


def test_sphere_shell_30720_developed_flow_5_cycles(libs):
    cgks, _, O3 = libs
    mesh = MG.sphere(3, 12, 4, h0=5e-3, growth=1.35, R_far=5.0)
    assert mesh.n_cells == 30720
    vel = (0.2, 0.0, 0.0)
    spec = dict(gamma=GAM, mu=0.2 / 118, bcs=[dict(kind="noslip"), dict(kind="farfield", rho=1.0, u=vel, p=1 / GAM)])
    W, Wx = perturbed(mesh, vel, 0.03, seed=30)
    g = cgks.Solver(cgks.Mesh(mesh), spec)
    o = O3.OracleSolver3(O3.OracleMesh3(mesh), spec)
    g.set_state(W, Wx)
    o.set_state(W, Wx)
    hg, ho = g.pmg_cycle(5), o.pmg_cycles(5)
    Wg, Xg = g.get_state()
    Wo, Xo = o.get_state()
    eW, eX = rel(Wg, Wo), rel(Xg, Xo)
    print(f"sphere 30720 developed: rel W {eW:.2e}  Wx {eX:.2e}  Res {np.abs(hg / ho - 1).max():.2e}")
    np.testing.assert_allclose(hg, ho, rtol=1e-9)
    assert eW < TOL, eW
    assert eX < TOL, eX


_LARGE = {}


def large_colours(name, O3):
    """Mesh, spec, perturbed state and the oracle's state after one V-cycle."""
    if name not in _LARGE:
        vel = (0.2, 0.0, 0.0)
        far = dict(kind="farfield", rho=1.0, u=vel, p=1 / GAM)
        if name == "sphere":
            mesh = MG.sphere(3, 20, 15, h0=5e-3, R_far=5.0)
            spec = dict(gamma=GAM, mu=0.2 / 118, bcs=[dict(kind="noslip"), far])
        else:
            mesh = MG.box3(28, 28, 28, jitter=0.1, seed=4, cells="prism", tags=(0, 0, 0, 0, 1, 1))
            spec = dict(gamma=GAM, mu=0.002, bcs=[far, dict(kind="slip")])
        W, Wx = perturbed(mesh, vel, 0.03, seed=30)
        o = O3.OracleSolver3(O3.OracleMesh3(mesh), spec)
        o.set_state(W, Wx)
        o.pmg_cycles(1)
        _LARGE[name] = (mesh, spec, (W, Wx), o.get_state())
    return _LARGE[name]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name, colours", [("sphere", 4), ("prisms", 2)])
def test_sweeps_with_one_thread_per_cell_match_the_oracle(libs, name, colours, precision):
    """A V-cycle whose colours hold more cells than the eight-lane form serves
    (4,864 in FP64, 14,000 in mixed): full passes up and down, and on the sphere
    (32,995 / 32,203 / 14,190 / 3,812 cells) descending passes over a part of a
    colour whose other cells advance on the way up, and one colour swept with
    eight lanes between them."""
    cgks, _, O3 = libs
    mesh, spec, state, (Wo, Xo) = large_colours(name, O3)
    gm = cgks.Mesh(mesh)
    cells = np.bincount(gm.ordering()[1])
    assert cells.size == colours and (cells[:3] >= 14000).all()
    g = cgks.Solver(gm, dict(spec, precision=precision))
    g.set_state(*state)
    g.pmg_cycle(1)
    Wg, Xg = g.get_state()
    g.close()
    assert rel(Wg, Wo) < (TOL if precision == "fp64" else 1e-5)
    assert rel(Xg, Xo) < (TOL if precision == "fp64" else 1e-4)
    assert rel(state[0], Wo) > 1e-4          # the field did change
