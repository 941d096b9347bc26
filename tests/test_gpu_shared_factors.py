"""Disks of an operator without drift and killing, factored once per grid shape, against the same disks
factored one by one (killing by one Gaussian of weight zero takes that form): every kind of source,
radii that differ, two grid shapes (of 48 disks, whose source columns are solved 17 at a time, and of a
few, which with a source are factored one by one), grids below the pivot-free factorisation's block, each
factorisation.

Both forms solve the same equations: FP64 to the rounding of an LU with condition below 1e5, mixed with
refinement to 1e-12 of the largest entry.  Bar: 1e-10 of each floating row, and of max(1, |b|)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _config(f, n_r, n_theta, n_knots):
    cfg = workloads.tiny(paths=32)
    nx, ny, s = 10, 9, 0.25
    rng = np.random.default_rng(3)
    n = nx * ny
    cfg["domain"] = {"kind": "square", "p": [0.0, 0.0, nx * s, ny * s]}
    cx, cy = np.meshgrid((np.arange(nx) + 0.5) * s, (np.arange(ny) + 0.5) * s)
    other = np.arange(n) % 7 == 3                       # a second shape, of few disks
    pick = lambda a, b: np.where(other, b, a).astype(np.int32)
    cfg["cover"] = {"kind": "explicit", "cx": cx.ravel(), "cy": cy.ravel(), "r": s * rng.uniform(0.76, 0.84, n),
                    "n_knots": pick(n_knots, n_knots + 2), "n_r": pick(n_r, n_r + 1),
                    "n_theta": pick(n_theta, n_theta + 2)}
    cfg["n_knots"] = cfg["n_r"] = cfg["n_theta"] = 0
    cfg["op"] = {"b": "zero", "c": "zero", "f": f, "g": "exp_sin"}
    if f == "rbf":
        cfg["op"]["frbf"] = workloads.rbf_field(5, seed=6, sigma=0.25, domain=cfg["domain"])
    return cfg


@pytest.mark.parametrize("precision,f,n_r,n_theta,n_knots,kw", [
    ("mixed", "zero", 12, 20, 12, {}), ("mixed", "one", 12, 20, 12, {}), ("mixed", "manufactured", 9, 22, 10, {}),
    ("mixed", "eq46", 12, 20, 24, {}), ("mixed", "rbf", 4, 8, 8, {}), ("mixed", "rbf", 12, 20, 12, {"factor": "blocked"}),
    ("mixed", "rbf", 12, 20, 12, {"lu_leaf_width": 16}), ("fp64", "zero", 12, 20, 12, {}),
    ("fp64", "rbf", 12, 20, 12, {}), ("fp64", "manufactured", 4, 8, 8, {})])
def test_shared_equals_one_by_one(precision, f, n_r, n_theta, n_knots, kw):
    import paper_2311_08946_gb300 as pdd

    cfg = _config(f, n_r, n_theta, n_knots)
    cov = pdd.Cover(cfg)
    a = {k: v.cpu().numpy() for k, v in cov.arrays().items()}
    got = pdd.System(cov, cfg, precision, **kw)
    cfg["op"] = dict(cfg["op"], c="rbf", rbf={"x": np.array([0.5]), "y": np.array([0.5]), "w": np.array([0.0]),
                                              "sigma": 0.2})
    ref = pdd.System(cov, cfg, precision, **kw)
    assert got.stats()["unconverged_disks"] == ref.stats()["unconverged_disks"] == 0
    for k in ("floating_disks", "floating_rows"):
        assert got.stats()[k] == ref.stats()[k]
    assert got.stats()["floating_disks"] > 40
    g, r = ({k: v.cpu().numpy() for k, v in s.csr().items()} for s in (got, ref))
    for i in range(cov.N):
        if a["row_sub"][i] < 0 or not a["floating"][a["row_sub"][i]]:
            continue
        s = slice(a["rowptr"][i], a["rowptr"][i + 1])
        assert np.linalg.norm(g["val"][s] - r["val"][s]) <= 1e-10 * np.linalg.norm(r["val"][s]), i
        assert abs(g["b"][i] - r["b"][i]) <= 1e-10 * max(1.0, abs(r["b"][i])), i
