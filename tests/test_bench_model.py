"""The benchmark's work model of the point relaxation against a walk through
its launches, cell by cell (host only)."""
import numpy as np
import pytest

import bench
from paper_2109_09965_gb300 import cgks
from paper_2109_09965_gb300 import meshgen as MG

SPEC = dict(n_sweeps=2, n_implicit=6, time_scheme="S1O2")


def walk(nbrs, colour, three, fp64):
    """Bytes and FP64 operations of the relaxation launches of one implicit step."""
    w, C = 8 if fp64 else 4, int(colour.max()) + 1
    nv = 5 if three else 4
    rec = (10 if fp64 else 8) if three else (8 if fp64 else 4)      # increment record
    seen = (5 if fp64 else 8) if three else (4 if fp64 else 8)      # part of a base record a neighbour reads
    base, normal = (16, 3) if three else (12, 2)
    per_nb, per_cell, adv = ((bench.SWEEP3_FLOPS_PER_NEIGHBOUR, bench.SWEEP3_FLOPS_PER_CELL,
                              bench.SWEEP3_FLOPS_ADVANCE) if three else
                             (bench.SWEEP_FLOPS_PER_NEIGHBOUR, bench.SWEEP_FLOPS_PER_CELL,
                              bench.SWEEP_FLOPS_ADVANCE))
    launches = []
    for _ in range(SPEC["n_sweeps"]):
        launches += [(c, False) for c in range(1, C)] + [(c, True) for c in range(C - 2, -1, -1)]
    byts = flops = count = 0
    last = {}
    for k, (c, down) in enumerate(launches):
        cells = [i for i in range(len(nbrs)) if colour[i] == c]
        if three and down and c > 0:   # the others' inputs have not changed
            cells = [i for i in cells if any(colour[j] > c for j in nbrs[i])]
        if not cells:
            continue
        count += 1
        for i in cells:
            last[i] = k
            byts += (nv + 1) * w + (4 * w if fp64 else 0) + rec * w
            byts += len(nbrs[i]) * (4 + (normal + 1 + (not fp64)) * w)
            flops += per_cell + per_nb * len(nbrs[i])
        byts += len({j for i in cells for j in nbrs[i]}) * (seen + rec) * w
    assert len(last) == len(nbrs)
    byts += len(last) * (2 * nv * 8 + base * w)                     # U in and out, next base record
    return byts, flops + adv * len(last), count


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim", [2, 3])
def test_relaxation_work_counts_what_the_launches_touch(dim, precision):
    mesh = MG.cavity(5) if dim == 2 else MG.sphere(1, 3, 2, h0=0.05, R_far=5.0)
    gm = cgks.Mesh(mesh)
    if dim == 2:
        nbrs = bench.topology(mesh, gm)[1]
    else:
        nbrs = [[] for _ in range(mesh.n_cells)]
        _, a, b, _, _ = bench.topology3(mesh, gm)
        for i, j in zip(a, b):
            nbrs[i].append(j)
            nbrs[j].append(i)
    _, colour = gm.ordering()
    model = (bench.work_model if dim == 2 else bench.work_model3)(mesh, gm, SPEC, precision)
    byts, flops, count = walk(nbrs, np.asarray(colour), dim == 3, precision == "fp64")
    ni, n = SPEC["n_implicit"], mesh.n_cells
    assert model["sweep_launches"] == ni * count
    assert model["bytes"]["k_sweep"] == ni * byts
    assert model["sweep_flops"] == ni * flops
    # the first base records: W_p0 in, U and the records out
    assert model["bytes"]["k_lo_cell"] == n * (2 * 8 * (dim + 2) + (12 if dim == 2 else 16) * (8 if precision == "fp64" else 4))
