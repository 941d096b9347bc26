"""Shared factors at their edges.

Few columns on the largest grids: two knots a circle and n = 7,168 nodes take the tiled solve for the
boundary columns, and so must the source columns.  The oracle is the disk's own solution: with f = 1 and
g = 0 the source part of a row is (R^2 - rho^2) / 2 for c = 0 (a polynomial, which every grid resolves), and
the boundary part sums to -1 (a constant is harmonic); bar 1e-9 (FP32 factors refined to 1e-12, n = 7,168)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _lattice(m, n_knots, n_r, n_theta, op):
    cfg = workloads.tiny(paths=32, h=1e-3)
    s = 1.0 / m
    cfg["domain"] = {"kind": "square", "p": [0.0, 0.0, 1.0, 1.0]}
    cfg["cover"] = {"kind": "square_lattice", "nx": m, "ny": m, "x_origin": 0.5 * s, "y_origin": 0.5 * s,
                    "spacing": s, "radius": 0.8 * s}
    cfg |= {"n_knots": n_knots, "n_r": n_r, "n_theta": n_theta, "op": op}
    return cfg


def _floating_b(cfg, precision):
    import paper_2311_08946_gb300 as pdd

    cov = pdd.Cover(cfg)
    a = {k: v.cpu().numpy() for k, v in cov.arrays().items()}
    s = pdd.System(cov, cfg, precision)
    assert s.stats()["unconverged_disks"] == 0
    sub = a["row_sub"]
    rows = np.flatnonzero((sub >= 0) & (a["floating"][np.maximum(sub, 0)] != 0))
    return cov, s, a, rows


def test_two_knots_on_a_large_grid():
    cfg = _lattice(8, 2, 64, 112, {"b": "zero", "c": "zero", "f": "one", "g": "zero"})
    cov, s, a, rows = _floating_b(cfg, "mixed")
    assert s.stats()["floating_disks"] == 36 and rows.size
    c = {k: v.cpu().numpy() for k, v in s.csr().items()}
    sub = a["row_sub"][rows]
    rho2 = (a["kx"][rows] - a["cx"][sub]) ** 2 + (a["ky"][rows] - a["cy"][sub]) ** 2
    want = (a["r"][sub] ** 2 - rho2) / 2
    assert np.abs(c["b"][rows] - want).max() <= 1e-9 * want.max()
    sums = np.add.reduceat(c["val"], a["rowptr"][:-1])[rows]
    assert np.abs(sums).max() <= 1e-9                     # 1 on the diagonal, -1 in all
